// FP32 coefficient tiles (PB_VARIANT_C32): the collision sweep of Eq. 2 over the upper block
// triangle of the branch-merged pair matrix, stored as 64 x 64 tiles of FP32 (P_in, P_out),
// 8 bytes per state pair: half the bytes of the float-float tiles.  Included by device.cu after
// kernels.cuh (it uses the tile, mbarrier and bulk-copy helpers there).
//
// Why a per-entry net term.  The pair (s, p) adds
//     n(s,p) = P_in f_p (1 - f_s) - P_out f_s (1 - f_p)
// to I_s / c and -n(s,p) to I_p / c (the reverse channel swaps P_in and P_out).  Near a steady
// state the two products are much larger than their difference, so sums of them (the A and C
// sums of the float-float sweep) rounded to FP32 carry errors of 2^-24 of the gross scattering,
// which the closing difference turns into 1e-6 of df/dt and more along a 1000-step trajectory.
// Here every entry forms n(s,p) itself, with the larger product made exact by an FMA error term:
//     n = P_in f_p - P_out f_s - d f_s f_p,   d = P_in - P_out,
//     u = fl(P_in f_p),  e = P_in f_p - u (exact, one FMA),  v = fl(P_out f_s - u) (one FMA),
//     n = fl(-d fl(f_s f_p) + (e - v)),
// so the rounding left in n is relative to n.  The occupations are float-float (f = f_h + f_l);
// n is taken at f_h and the entry adds its first-order change in f_l,
//     t(s,p) = n + f_l,p (P_in - f_s d) - f_l,s (P_out + f_p d)
// (dn/df_p = P_in - f_s d, dn/df_s = -(P_out + f_p d); the second-order term f_l,s f_l,p d is
// below 2^-48 of the products).  t(p,s) = -t(s,p) for every f, so the row of s adds t and the
// row of p subtracts the same FP32 value: each state needs one sum, I_s = c sum_p t(s,p).
//
// The states keep their natural order here (the float-float tiles are in energy order and skip the
// blocks out of reach): the FP32 sums of a block depend on which states share it, and in energy order
// the RK4 state moved by up to 1.5e-9, as much as the sums' own rounding (36^3, 4 steps: 193 -> 124 us
// with the blocks out of reach skipped).
//
namespace pb {
namespace dev {

constexpr int kC32Threads = 256;
constexpr int kC32RatioUlps = 2;
constexpr unsigned kC32TileBytes = kTile * kTile * sizeof(float2);
constexpr unsigned kC32StageBytes = kC32TileBytes + 2 * kTile * sizeof(float2);
constexpr size_t kC32ColFloats = (size_t)(kC32Threads / 32) * kTile;  // [8 warps][64 columns]
// dynamic shared memory of a launch shape with NST stages (and the double-buffered column table)
template <int NST>
constexpr size_t c32_smem() {
  return (size_t)NST * kC32StageBytes + 320 + 2 * kC32ColFloats * sizeof(float);
}

// (a, b) ~ (P_in, P_out) in FP32 with the ratio kept (see above); zero stays zero.
__device__ __forceinline__ float2 c32_round_pair(double pin, double pout) {
  const float a0 = __double2float_rn(pin);
  if (!(a0 > 0.f) || !(pout > 0.0)) return make_float2(a0, __double2float_rn(pout));
  const double r = pout / pin;
  float ba = a0, bb = __double2float_rn((double)a0 * r);
  double be = fabs((double)bb / (double)ba - r);
  for (int k = -kC32RatioUlps; k <= kC32RatioUlps; ++k) {
    if (k == 0) continue;
    const float a = __int_as_float(__float_as_int(a0) + k);
    if (!(a > 0.f) || isinf(a)) continue;
    const float b = __double2float_rn((double)a * r);
    if (!(b > 0.f) || isinf(b)) continue;
    const double e = fabs((double)b / (double)a - r);
    if (e < be) {
      be = e;
      ba = a;
      bb = b;
    }
  }
  return make_float2(ba, bb);
}

// The symmetric tiles from the branch-merged pair rows (complete or not): one warp per row s, every
// stored pair (s, p) written to its tile entries; the tiles were zeroed before, pairs without channels
// stay zero.  pmap: each state's row in the padded energy order (of one system, or of a batch's systems
// one after the other); tbase[I] = (the index of tile (I, I), the last block column stored for block
// row I): tiles of a block row are numbered consecutively, and pairs beyond the last column have zero
// coefficients (energy_reach).
// Float-float (float4 per entry): a pair's P_in(s, p) is P_in of entry (s, p) and, by the reverse
// channels, P_out of entry (p, s), so each half of an entry is one row's stored P_in to 2^-49.  P_in + D
// of one row would lose the smaller direction to cancellation (P_out / P_in = exp(-hbar w / kT): the
// absorption rates were off by up to 5e-13 at 100 K, and the scattering rates of occupied states with them).
// C32: the pairs P_in, P_in + D of the upper triangle rounded to FP32 with their ratio kept.
template <bool C32, typename IDX>
__global__ void k_tiles_scatter(const long long *__restrict__ srp, int ns, const IDX *__restrict__ pidx,
                                const float2 *__restrict__ coefA, const float2 *__restrict__ coefB,
                                const int *__restrict__ pmap, const int2 *__restrict__ tbase, void *__restrict__ tc) {
  const int lane = threadIdx.x & 31;
  const int w0 = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)(((long long)gridDim.x * blockDim.x) >> 5);
  for (int r = w0; r < ns; r += nw) {
    const int pr = pmap[r], I = pr / kTile;
    const int2 tb = tbase[I];
    for (long long e = srp[r] + lane; e < srp[r + 1]; e += 32) {
      const float2 a = coefA[e];
      if (C32) {
        const float2 b = coefB[e];
        if (a.x == 0.f && a.y == 0.f && b.x == 0.f && b.y == 0.f) continue;
        const int pp = pmap[pidx[e]], J = pp / kTile;
        if (J < I || J > tb.y) continue;
        const long long k = (long long)(tb.x + (J - I)) * kTile * kTile + (pr % kTile) * kTile + pp % kTile;
        const double pin = ff_to_double(a.x, a.y), pout = pin + ff_to_double(b.x, b.y);
        ((float2 *)tc)[k] = c32_round_pair(pin, pout);
      } else {
        if (a.x == 0.f && a.y == 0.f) continue;
        const int pp = pmap[pidx[e]], J = pp / kTile;
        if (J >= I && J <= tb.y)
          ((float2 *)tc)[2 * ((long long)(tb.x + (J - I)) * kTile * kTile + (pr % kTile) * kTile + pp % kTile)] = a;
        if (J <= I) {
          const int2 tj = tbase[J];
          if (I <= tj.y)
            ((float2 *)tc)[2 * ((long long)(tj.x + (I - J)) * kTile * kTile + (pp % kTile) * kTile + pr % kTile) + 1] = a;
        }
      }
    }
  }
}

// t(s, p) above from the entry's rounded (P_in, P_out) = (a, b) and the float-float occupations
// fs of s and fp of p
__device__ __forceinline__ float c32_term(float a, float b, float2 fs, float2 fp) {
  const float d = __fsub_rn(a, b);
  const float u = __fmul_rn(a, fp.x);
  const float ex = __fmaf_rn(a, fp.x, -u);
  const float v = __fmaf_rn(b, fs.x, -u);
  const float w = __fmul_rn(fs.x, fp.x);
  float t = __fmaf_rn(-d, w, __fsub_rn(ex, v));
  t = __fmaf_rn(fp.y, __fmaf_rn(-fs.x, d, a), t);
  return __fmaf_rn(-fs.y, __fmaf_rn(fp.x, d, b), t);
}

// reduce-scatter of NV floats over the 2 * TOP lanes that differ in lane bits log2 TOP .. 0: at
// the end v[0] holds the total of value index idx(lane) = those bits of the lane, most
// significant first (the float-float version is ff_reduce_scatter)
template <int NV, int TOP>
__device__ __forceinline__ void f32_reduce_scatter(float (&v)[NV], int lane) {
  int n = NV;
#pragma unroll
  for (int mask = TOP; mask > 0; mask >>= 1) {
    if (n > 1) {
      const bool up = lane & mask;
      const int h = n >> 1;
#pragma unroll
      for (int k = 0; k < NV / 2; ++k) {
        if (k < h) {
          const float send = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
          v[k] = __fadd_rn(keep, __shfl_xor_sync(0xFFFFFFFFu, send, mask));
        }
      }
      n = h;
    } else {
      v[0] = __fadd_rn(v[0], __shfl_xor_sync(0xFFFFFFFFu, v[0], mask));
    }
  }
}

// the column sums of a finished off-diagonal tile: threads 0..63 add the 8 warps' values of
// one column each and write them to the tile's column slots
__device__ __forceinline__ void c32_columns_out(const float *__restrict__ colred, int cb, int cs, int tid,
                                                float *__restrict__ tp) {
  if (tid >= kTile) return;
  float acc = colred[tid];
#pragma unroll
  for (int w = 1; w < kC32Threads / 32; ++w) acc = __fadd_rn(acc, colred[w * kTile + tid]);
  tp[cb + tid * cs] = acc;
}

// One persistent 256-thread CTA (CPS per SM) streams its share of the tiles through NST
// shared-memory stages filled by bulk copies (thread 0 issues, completion counted in bytes on
// one mbarrier per stage, every wait bounded), as k_stream_sym_bulk does for the float-float
// tiles.  Thread (ti, tj) takes rows 4 ti .. 4 ti + 3 and columns tj + 16 j.  One FP32 partial
// per (state, block of partner states): MODE_COLL the sum of t above; MODE_RATE the sum of the
// 1/tau_s summands P_out + f_p d (row s) and P_in - f_s d (column p, the reverse channel), each
// with its f_l term.  The per-warp column table is double buffered and combined in the next
// iteration, so a tile costs one CTA barrier.
// rev: take the tile list from its end (tile nt - 1 - t in place of t), so that a sweep following
// one in list order starts on the tiles the L2 still holds.
template <int MODE, int NST, int CPS, bool PDL>
__global__ void __launch_bounds__(kC32Threads, CPS) k_stream_c32(const TileD *__restrict__ tiles, int nt,
                                                                  const float2 *__restrict__ tc,
                                                                  const float2 *fg,
                                                                  float *__restrict__ tp, int *__restrict__ err,
                                                                  int rev = 0) {
  // the stage of tile k - 1 is refilled (with tile k - 1 + NST) only after the wait for tile k, so
  // one stage would wait for a copy not yet issued
  static_assert(NST >= 2 && NST <= 8, "the ring needs 2..8 stages");
  constexpr int R = 4;
  extern __shared__ __align__(128) unsigned char ssm[];
  unsigned long long *bars = (unsigned long long *)(ssm + NST * kC32StageBytes);
  TileD *stile = (TileD *)(bars + 8);
  float *colred0 = (float *)(ssm + NST * kC32StageBytes + 320);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, tj = tid & 15, ti = tid >> 4;
  const int G = (int)gridDim.x;
  const int nloc = (int)blockIdx.x < nt ? (nt - 1 - (int)blockIdx.x) / G + 1 : 0;
  if (tid == 0) {
    for (int k = 0; k < NST; ++k) mbar_init(bars + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int issued = 0;
  auto tix = [&](int k) {  // the CTA's k-th tile
    const int t = (int)blockIdx.x + k * G;
    return rev ? nt - 1 - t : t;
  };
  auto issue_f = [&](int k, const TileD &D) {  // the f slices of the CTA's tile k
    const int s = k % NST;
    unsigned char *buf = ssm + (size_t)s * kC32StageBytes + kC32TileBytes;
    bulk_g2s(buf, fg + (size_t)D.I * kTile, kTile * sizeof(float2), bars + s);
    bulk_g2s(buf + kTile * sizeof(float2), fg + (size_t)D.J * kTile, kTile * sizeof(float2), bars + s);
  };
  auto issue = [&](int k, const TileD &D) {  // its coefficients
    const int s = k % NST;
    const int t = tix(k);
    stile[s] = D;
    unsigned char *buf = ssm + (size_t)s * kC32StageBytes;
    mbar_expect_tx(bars + s, kC32StageBytes);
    const unsigned char *src = (const unsigned char *)(tc + (size_t)t * kTile * kTile);
#pragma unroll
    for (int q = 0; q < 2; ++q) bulk_g2s(buf + q * (kC32TileBytes / 2), src + q * (kC32TileBytes / 2), kC32TileBytes / 2, bars + s);
  };
  if (tid == 0) {
    for (; issued < NST && issued < nloc; ++issued) {
      const TileD D = load_tile(tiles, tix(issued));
      issue(issued, D);
      if (!PDL) issue_f(issued, D);
    }
    if (PDL) {
      pdl_wait();  // f comes from the kernel before this one, which may still read the partials
      for (int k = 0; k < issued; ++k) issue_f(k, stile[k]);
    }
  }
  TileD next{};
  if (tid == 0 && issued < nloc) next = load_tile(tiles, tix(issued));
  int pcb = -1, pcs = 0;  // column slots of the previous tile (-1: diagonal, or none)
  bool ok = true;
  for (int k = 0; k <= nloc; ++k) {
    const bool have = k < nloc;
    if (!__syncthreads_and(tid == 0 && have ? mbar_wait(bars + k % NST, (unsigned)((k / NST) & 1)) : true)) {
      ok = false;
      break;
    }
    if (tid == 0 && k >= 1 && issued < nloc) {
      fence_proxy_async();  // the generic reads of tile k-1's stage before its refill
      issue(issued, next);
      issue_f(issued, next);
      ++issued;
      if (issued < nloc) next = load_tile(tiles, tix(issued));
    }
    if (k >= 1 && pcb >= 0) c32_columns_out(colred0 + ((k - 1) & 1) * kC32ColFloats, pcb, pcs, tid, tp);
    if (!have) break;
    if (PDL && k + 1 == nloc) pdl_trigger();
    const int s = k % NST;
    const TileD D = stile[s];
    const bool diag = D.I == D.J;
    pcb = diag ? -1 : D.cb;
    pcs = D.cs;
    const float2 *__restrict__ T = (const float2 *)(ssm + (size_t)s * kC32StageBytes);
    const float2 *__restrict__ fr = (const float2 *)(ssm + (size_t)s * kC32StageBytes + kC32TileBytes);
    const float2 *__restrict__ fc = fr + kTile;
    float2 fcol[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) fcol[j] = fc[tj + 16 * j];
    float rv[R], cv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) rv[i] = cv[i] = 0.f;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int row = ti * R + i;
      const float2 fs = fr[row];
      float2 e[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) e[j] = T[row * kTile + tj + 16 * j];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = e[j].x, b = e[j].y, fp = fcol[j].x, flp = fcol[j].y;
        if (MODE == MODE_COLL) {
          const float t = c32_term(a, b, fs, fcol[j]);
          rv[i] = __fadd_rn(rv[i], t);
          if (!diag) cv[j] = __fsub_rn(cv[j], t);
        } else {  // 1/tau summands: row s: P_out + f_p d; column p (reverse channel): P_in - f_s d
          const float d = __fsub_rn(a, b);
          rv[i] = __fadd_rn(rv[i], __fmaf_rn(flp, d, __fmaf_rn(fp, d, b)));
          if (!diag) cv[j] = __fadd_rn(cv[j], __fmaf_rn(-fs.y, d, __fmaf_rn(-fs.x, d, a)));
        }
      }
    }
    // rows: the 16 lanes of a half-warp share them; lanes 4i .. 4i + 3 end with the total of row i
    f32_reduce_scatter<R, 8>(rv, lane);
    if ((tj & 3) == 0) tp[D.rb + (ti * R + (tj >> 2)) * D.rs] = rv[0];
    if (!diag) {
      // columns: lanes tj and tj + 16 share them (one level), then the 8 warps (next iteration)
      float *colred = colred0 + (k & 1) * kC32ColFloats;
      const bool up = lane & 16;
#pragma unroll
      for (int jk = 0; jk < 2; ++jk) {
        const int jo = jk + 2;  // kept / sent column slot
        const float kept = up ? cv[jo] : cv[jk], sent = up ? cv[jk] : cv[jo];
        colred[wid * kTile + tj + 16 * ((up ? 2 : 0) + jk)] = __fadd_rn(kept, __shfl_xor_sync(0xFFFFFFFFu, sent, 16));
      }
    }
  }
  if (!ok) {
    *err = 2;
    if (tid == 0) {
      for (int k = 0; k < NST; ++k) {
        const int uses = issued / NST + (k < issued % NST ? 1 : 0);
        if (uses > 0) mbar_wait(bars + k, (unsigned)((uses - 1) & 1));
      }
    }
  }
}

// The same sweep in half-tiles (32 rows x 64 columns, 16 KB, contiguous in the tile): a tile's
// column sums stay in registers across its two halves and go through the per-warp table after the
// second, which is combined after the next unit's barrier (columns are written only every other
// unit, so one table suffices).  Three 17 KB stages and the 2 KB table take 53 KB, so four CTAs
// (32 warps) fit on an SM.  Thread (ti, tj) takes rows 2 ti, 2 ti + 1 of the unit and columns
// tj + 16 j.
constexpr unsigned kC32HalfBytes = kC32TileBytes / 2;
constexpr unsigned kC32HalfStageBytes = kC32HalfBytes + (kTile / 2 + kTile) * sizeof(float2);
template <int NST>
constexpr size_t c32_half_smem() {
  return (size_t)NST * kC32HalfStageBytes + 320 + kC32ColFloats * sizeof(float);
}

template <int MODE, int NST, int CPS, bool PDL>
__global__ void __launch_bounds__(kC32Threads, CPS) k_stream_c32_half(const TileD *__restrict__ tiles, int nt,
                                                                       const float2 *__restrict__ tc,
                                                                       const float2 *fg,
                                                                       float *__restrict__ tp, int *__restrict__ err,
                                                                       int rev = 0) {
  static_assert(NST >= 2 && NST <= 8, "the ring needs 2..8 stages");
  constexpr int R = 2, HR = kTile / 2;
  extern __shared__ __align__(128) unsigned char ssm[];
  unsigned long long *bars = (unsigned long long *)(ssm + NST * kC32HalfStageBytes);
  TileD *stile = (TileD *)(bars + 8);
  float *colred = (float *)(ssm + NST * kC32HalfStageBytes + 320);  // [8 warps][64 columns]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, tj = tid & 15, ti = tid >> 4;
  const int G = (int)gridDim.x;
  const int nloc = (int)blockIdx.x < nt ? (nt - 1 - (int)blockIdx.x) / G + 1 : 0;
  const int nunit = 2 * nloc;
  if (tid == 0) {
    for (int k = 0; k < NST; ++k) mbar_init(bars + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int issued = 0;
  auto tix = [&](int k) {  // the CTA's k-th tile
    const int t = (int)blockIdx.x + k * G;
    return rev ? nt - 1 - t : t;
  };
  TileD iss{}, ahead{};
  if (tid == 0 && nloc > 0) {
    iss = load_tile(tiles, tix(0));
    if (nloc > 1) ahead = load_tile(tiles, tix(1));
  }
  auto issue_f = [&](int v, const TileD &D) {  // the f slices of unit v
    const int h = v & 1, s = v % NST;
    unsigned char *buf = ssm + (size_t)s * kC32HalfStageBytes + kC32HalfBytes;
    bulk_g2s(buf, fg + (size_t)D.I * kTile + h * HR, HR * sizeof(float2), bars + s);
    bulk_g2s(buf + HR * sizeof(float2), fg + (size_t)D.J * kTile, kTile * sizeof(float2), bars + s);
  };
  auto issue = [&](int v) {  // (coefficients) unit v = 2 k + h: half h of the CTA's tile k
    const int k = v >> 1, h = v & 1, s = v % NST;
    if (h == 0 && k > 0) {
      iss = ahead;
      if (k + 1 < nloc) ahead = load_tile(tiles, tix(k + 1));
    }
    const int t = tix(k);
    stile[s] = iss;
    unsigned char *buf = ssm + (size_t)s * kC32HalfStageBytes;
    mbar_expect_tx(bars + s, kC32HalfStageBytes);
    const unsigned char *src = (const unsigned char *)(tc + (size_t)t * kTile * kTile) + (size_t)h * kC32HalfBytes;
    bulk_g2s(buf, src, kC32HalfBytes, bars + s);
  };
  if (tid == 0) {
    for (; issued < NST && issued < nunit; ++issued) {
      issue(issued);
      if (!PDL) issue_f(issued, iss);
    }
    if (PDL) {
      pdl_wait();  // f comes from the kernel before this one, which may still read the partials
      for (int v = 0; v < issued; ++v) issue_f(v, stile[v]);
    }
  }
  int pcb = -1, pcs = 0;  // column slots of the previous unit's tile (-1: diagonal, or none)
  bool ok = true;
  float cv[4];  // column sums of the current tile, carried across its halves
  for (int u = 0; u <= nunit; ++u) {
    const bool have = u < nunit;
    if (!__syncthreads_and(tid == 0 && have ? mbar_wait(bars + u % NST, (unsigned)((u / NST) & 1)) : true)) {
      ok = false;
      break;
    }
    if (tid == 0 && u >= 1 && issued < nunit) {
      fence_proxy_async();  // the generic reads of unit u-1's stage before its refill
      issue(issued);
      issue_f(issued, iss);
      ++issued;
    }
    if ((u & 1) == 0 && u >= 2 && pcb >= 0) c32_columns_out(colred, pcb, pcs, tid, tp);
    if (!have) break;
    if (PDL && u + 1 == nunit) pdl_trigger();
    const int s = u % NST, h = u & 1;
    const TileD D = stile[s];
    const bool diag = D.I == D.J;
    pcb = diag ? -1 : D.cb;
    pcs = D.cs;
    const float2 *__restrict__ T = (const float2 *)(ssm + (size_t)s * kC32HalfStageBytes);
    const float2 *__restrict__ fr = (const float2 *)(ssm + (size_t)s * kC32HalfStageBytes + kC32HalfBytes);
    const float2 *__restrict__ fc = fr + HR;
    float2 fcol[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) fcol[j] = fc[tj + 16 * j];
    if (h == 0)
#pragma unroll
      for (int j = 0; j < 4; ++j) cv[j] = 0.f;
    float rv[R];
#pragma unroll
    for (int i = 0; i < R; ++i) rv[i] = 0.f;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int row = ti * R + i;
      const float2 fs = fr[row];
      float2 e[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) e[j] = T[row * kTile + tj + 16 * j];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = e[j].x, b = e[j].y;
        if (MODE == MODE_COLL) {
          const float t = c32_term(a, b, fs, fcol[j]);
          rv[i] = __fadd_rn(rv[i], t);
          if (!diag) cv[j] = __fsub_rn(cv[j], t);
        } else {  // 1/tau summands: row s: P_out + f_p d; column p (reverse channel): P_in - f_s d
          const float d = __fsub_rn(a, b);
          rv[i] = __fadd_rn(rv[i], __fmaf_rn(fcol[j].y, d, __fmaf_rn(fcol[j].x, d, b)));
          if (!diag) cv[j] = __fadd_rn(cv[j], __fmaf_rn(-fs.y, d, __fmaf_rn(-fs.x, d, a)));
        }
      }
    }
    // rows: the 16 lanes of a half-warp share them; lanes 8i .. 8i + 7 end with the total of row i
    f32_reduce_scatter<R, 8>(rv, lane);
    if ((tj & 7) == 0) tp[D.rb + (h * HR + ti * R + (tj >> 3)) * D.rs] = rv[0];
    if (!diag && h == 1) {
      // columns of the whole tile: lanes tj and tj + 16 share them (one level), then the warps
      // (after the next unit's barrier)
      const bool up = lane & 16;
#pragma unroll
      for (int jk = 0; jk < 2; ++jk) {
        const int jo = jk + 2;
        const float kept = up ? cv[jo] : cv[jk], sent = up ? cv[jk] : cv[jo];
        colred[wid * kTile + tj + 16 * ((up ? 2 : 0) + jk)] = __fadd_rn(kept, __shfl_xor_sync(0xFFFFFFFFu, sent, 16));
      }
    }
  }
  if (!ok) {
    *err = 2;
    if (tid == 0) {
      for (int k = 0; k < NST; ++k) {
        const int uses = issued / NST + (k < issued % NST ? 1 : 0);
        if (uses > 0) mbar_wait(bars + k, (unsigned)((uses - 1) & 1));
      }
    }
  }
}

// The same FP32 pair coefficients as a row stream, for the batched rt-BTE (precision 2): entry
// e of the branch-merged rows holds C[e] = rounded (P_in, P_out) of (row state, partner colp[e]);
// one warp per item (a piece of one row), each lane two 4-entry groups per trip, partners'
// float-float f gathered through L1; part[item].x = sum of t(s, p) over the item.
template <typename IDX>
__global__ void __launch_bounds__(kBlock) k_stream_c32_rows(const Item *__restrict__ items, int nitems,
                                                            const float4 *__restrict__ C4,
                                                            const IDX *__restrict__ colp,
                                                            const float2 *__restrict__ fg,
                                                            Part4 *__restrict__ part) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int it = warp; it < nitems; it += nwarps) {
    const Item I = items[it];
    const long long g0 = I.start >> 2;
    const int ng = I.len >> 2;
    const float2 fs = fg[I.row];
    float acc = 0.f, acc2 = 0.f;
    int g = lane;
    for (; g + 32 < ng; g += 64) {
      const long long q0 = g0 + g, q1 = q0 + 32;
      const uint4 c0 = partners4(colp, q0), c1 = partners4(colp, q1);
      const float4 x0 = __ldcs(C4 + 2 * q0), y0 = __ldcs(C4 + 2 * q0 + 1);
      const float4 x1 = __ldcs(C4 + 2 * q1), y1 = __ldcs(C4 + 2 * q1 + 1);
      acc = __fadd_rn(acc, c32_term(x0.x, x0.y, fs, fg[c0.x]));
      acc2 = __fadd_rn(acc2, c32_term(x1.x, x1.y, fs, fg[c1.x]));
      acc = __fadd_rn(acc, c32_term(x0.z, x0.w, fs, fg[c0.y]));
      acc2 = __fadd_rn(acc2, c32_term(x1.z, x1.w, fs, fg[c1.y]));
      acc = __fadd_rn(acc, c32_term(y0.x, y0.y, fs, fg[c0.z]));
      acc2 = __fadd_rn(acc2, c32_term(y1.x, y1.y, fs, fg[c1.z]));
      acc = __fadd_rn(acc, c32_term(y0.z, y0.w, fs, fg[c0.w]));
      acc2 = __fadd_rn(acc2, c32_term(y1.z, y1.w, fs, fg[c1.w]));
    }
    if (g < ng) {
      const long long q0 = g0 + g;
      const uint4 c0 = partners4(colp, q0);
      const float4 x0 = __ldcs(C4 + 2 * q0), y0 = __ldcs(C4 + 2 * q0 + 1);
      acc = __fadd_rn(acc, c32_term(x0.x, x0.y, fs, fg[c0.x]));
      acc = __fadd_rn(acc, c32_term(x0.z, x0.w, fs, fg[c0.y]));
      acc = __fadd_rn(acc, c32_term(y0.x, y0.y, fs, fg[c0.z]));
      acc = __fadd_rn(acc, c32_term(y0.z, y0.w, fs, fg[c0.w]));
    }
    acc = __fadd_rn(acc, acc2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, o));
    if (lane == 0) part[it] = make_part4((double)acc, 0.0, 0.0, 0.0);
  }
}

// C[e] = rounded (P_in, P_out) of n branch-merged float-float entries (A = P_in, B = D)
__global__ void k_pairs_c32(const float2 *__restrict__ A, const float2 *__restrict__ B, long long n,
                            float2 *__restrict__ C) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const double pin = ff_to_double(A[e].x, A[e].y);
    C[e] = c32_round_pair(pin, pin + ff_to_double(B[e].x, B[e].y));
  }
}

// Epilogue of the net-term sweeps (PT = float: C32; float2: the float-float half-tile sweep, whose
// next input is (f, 1 - f)): a 256-thread CTA takes SPC states; each warp adds the block
// partials of SPC / 8 states (lanes over the blocks in float-float, then one 32-lane float-float
// reduce-scatter of the SPC / 8 values), and warp 0 applies the prefactor and the RK4 stage
// arithmetic in FP64, one lane per state.
// prow, pmap: as TileSrc.  RATE: 1/tau = c (R - sum) for the float-float sweep (partials of B), c sum
// for C32 (partials of the summands themselves).
__device__ __forceinline__ float2 as_ff(float v) { return make_float2(v, 0.f); }
__device__ __forceinline__ float2 as_ff(float2 v) { return v; }
template <typename PT, int STAGE, bool RATE, int SPC, bool PDL>
__global__ void __launch_bounds__(256) k_fin_net(const PT *tp, const int2 *__restrict__ prow,
                                                 const int *__restrict__ pmap, int ns, double c,
                                                 const double *__restrict__ R, double *out, double *f, double *acc,
                                                 double *y, float2 *yff, double dt) {
  constexpr int SPW = SPC / 8, LPV = 32 / SPW;  // states per warp, lanes per state after the reduce-scatter
  __shared__ float2 tot[SPC];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int base = blockIdx.x * SPC;
  const int r0 = base + lane;
  FinIn in{0.0, 0.0, 0.0, 0.0};
  int ry = 0;
  int2 pr[SPW];
  auto load_rows = [&] {
#pragma unroll
    for (int q = 0; q < SPW; ++q) {
      const int r = base + SPW * wid + q;
      pr[q] = r < ns ? prow[r] : make_int2(0, 0);
    }
  };
  if (PDL) {
    load_rows();
    pdl_wait();
  }
  double Rr = 0.0;
  if (RATE && R && wid == 0 && lane < SPC && r0 < ns) Rr = R[r0];
  if (!RATE && wid == 0 && lane < SPC && r0 < ns) {
    if (STAGE >= 0) in.f = f[r0];
    if (STAGE >= 1) in.acc = acc[r0];
    if (STAGE >= 0) ry = pmap[r0];
  }
  float2 v[SPW];
  if (!PDL) load_rows();
#pragma unroll
  for (int q = 0; q < SPW; ++q) {
    v[q] = make_float2(0.f, 0.f);
    for (int k = lane; k < pr[q].y; k += 32) v[q] = ff_add(v[q], as_ff(__ldcg(tp + pr[q].x + k)));
  }
  if (PDL) pdl_trigger();
  ff_reduce_scatter<SPW, 16>(v, lane);
  if ((lane & (LPV - 1)) == 0) tot[SPW * wid + lane / LPV] = v[0];
  __syncthreads();
  if (wid != 0 || lane >= SPC || r0 >= ns) return;
  const float2 Tt = tot[lane];
  if (RATE) {
    out[r0] = c * (R ? Rr - ff_to_double(Tt.x, Tt.y) : ff_to_double(Tt.x, Tt.y));
    return;
  }
  const double I = c * ff_to_double(Tt.x, Tt.y);
  fin_stage<STAGE, sizeof(PT) == sizeof(float) ? OUT_FF : OUT_FG>(r0, I, in, out, f, acc, y, yff, dt, ry);
}

}  // namespace dev
}  // namespace pb
