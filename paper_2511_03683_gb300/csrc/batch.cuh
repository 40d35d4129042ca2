// Batched rt-BTE: many independent e-ph systems (different grids, bands, modes,
// temperatures) advanced together.  Included at the end of device.cu (one translation unit).
//
// All instances' channel lists are concatenated (rows padded to 8 channels) with |g|^2 in
// FP32, one padded FP32 phonon table per instance, one 16-byte record per state, and a single
// work-item list whose items carry an instance id.  One persistent launch per RK4 stage
// sweeps every instance: each CTA takes a contiguous range of items (mostly one instance, so
// the partner records it gathers stay in L1), evaluates the literal per-channel form of
// Eq. 2 in FP32 with Kahan lane sums, and one finaliser applies each state's prefactor and
// the FP64 RK4 stage arithmetic.  A CUDA graph of the 8 launches replays each step.  The item
// size and CTAs per SM come from a small autotuner that times candidate launch shapes.
//
// With pb_batch_opts.precision = 1 the batch streams FP64-accurate coefficients instead:
// every instance's per-channel P_in and D are computed once in FP64 (its own grid, bands,
// phonons, T and sigma), summed over the branches of each state pair and scaled by the
// instance's 2 pi / (hbar N_q), then concatenated; the sweep and the RK4 stage epilogues are
// the single-system float-float kernels run over all instances at once.
//
// With precision = 2 the same branch-merged coefficients are rounded once to FP32 pairs
// (P_in, P_out) with their ratio kept, 8 bytes per state pair, and the row stream forms each
// entry's net term in FP32 with an exact leading product and the first-order terms in the low
// part of f (tiles32.cuh): df/dt within about 1e-6 of Eq. 2.
//
// Symmetric tiles (precision 1 and 2, every instance's channel list verified closed under
// reversal): each instance takes a run of 64-state blocks of one padded state space, its states in
// energy order (precision 2: in state order, all tiles of the triangle), and the tiles of its upper
// block triangle within reach of a phonon are stored as
// 64 x 64 tiles (zero where a state pair has no channel), as in the single-system sweeps, so each
// unordered state pair is streamed once for both of its directions and the pairs whose coefficients
// are zero by their distance in energy are not streamed at all.  One launch of the single-system
// tile kernel sweeps every instance's tiles; the epilogues map each state to its padded row.

namespace pb {
namespace dev {

struct BInst {
  const float2 *tab;  // this instance's padded phonon table
  int cpad;           // L(N1,N2,N3) * nmodes of the instance
  float k2;           // -log2(e) / (2 sigma^2)
  int soff;           // first global state of the instance
  int ns;             // states of the instance
  long long doff;     // dense form: the instance's first value in g2d
  long long poff;     // its first slot in pidx
  long long moff;     // its first entry in the slot map
  int nm, pad;        // branches
};

template <int MODE>
__global__ void __launch_bounds__(512) k_stream_gbatch(const Item *__restrict__ items,
                                                       const int *__restrict__ item_inst, int nitems,
                                                       const BInst *__restrict__ inst,
                                                       const uint32_t *__restrict__ col,
                                                       const float *__restrict__ g2v,
                                                       const uint4 *__restrict__ gstate, Part4 *__restrict__ part) {
  const int per = (nitems + gridDim.x - 1) / gridDim.x;
  const int begin = blockIdx.x * per;
  const int end = min(nitems, begin + per);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint4 *__restrict__ col4 = (const uint4 *)col;
  for (int it = begin + wib; it < end; it += nw) {
    const Item I = items[it];
    const BInst B = inst[item_inst[it]];
    GGeom g;
    g.col = col;
    g.tabp = B.tab;
    g.cpad = B.cpad;
    g.k2 = B.k2;
    const uint4 ss = __ldg(gstate + I.row);
    const int base = B.cpad - rec_lnm(ss);
    const uint4 *__restrict__ gsi = gstate + B.soff;
    const long long g0 = I.start >> 2;
    const int ng = I.len >> 2;
    float sum = 0.f, comp = 0.f;
    uint4 c = make_uint4(0u, 0u, 0u, 0u);
    float4 gv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < ng) {
      c = __ldcs(col4 + g0 + lane);
      gv = load_g2x4(g2v, g0 + lane);
    }
    for (int q = lane; q < ng; q += 32) {
      uint4 cn = make_uint4(0u, 0u, 0u, 0u);
      float4 gn = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q + 32 < ng) {
        cn = __ldcs(col4 + g0 + q + 32);
        gn = load_g2x4(g2v, g0 + q + 32);
      }
      const float t0 = g_term<MODE>(g, ss, __ldg(gsi + (c.x & 0xFFFFFFu)), c.x, base, gv.x);
      const float t1 = g_term<MODE>(g, ss, __ldg(gsi + (c.y & 0xFFFFFFu)), c.y, base, gv.y);
      const float t2 = g_term<MODE>(g, ss, __ldg(gsi + (c.z & 0xFFFFFFu)), c.z, base, gv.z);
      const float t3 = g_term<MODE>(g, ss, __ldg(gsi + (c.w & 0xFFFFFFu)), c.w, base, gv.w);
      kahan_add(sum, comp, t0);
      kahan_add(sum, comp, t1);
      kahan_add(sum, comp, t2);
      kahan_add(sum, comp, t3);
      c = cn;
      gv = gn;
    }
    const double v = warp_sum((double)sum - (double)comp);
    if (lane == 0) part[it] = make_part4(v, 0.0, 0.0, 0.0);
  }
}

// Dense pair-major form of the FP32 batch sweep (as k_stream_g_dense, per instance): every
// instance's pairs in reach have one slot each, their branches together at g2d[doff + slot * nm],
// their partners (numbered within the instance) at pidx[poff + slot].  An item is a bundle of 32
// chains of the global row I.row, its slots numbered within the instance (LanePlan); partner records
// come through L1 (CTA b takes the items [cbeg[b], cbeg[b + 1]), ranges of about equal work, mostly
// of one instance: rows differ tenfold in length over the instances).  The per-pair arithmetic is
// k_stream_g_dense's (the bracket collected per pair).  pidx: as there, with 32-bit words (the top bit the
// gap, the next the padding).
constexpr uint32_t kPadBit32 = 0x40000000u;
__global__ void __launch_bounds__(512, 2) k_stream_gbatch_dense(const Item *__restrict__ items,
                                                             const int *__restrict__ item_inst,
                                                             const int *__restrict__ cbeg,
                                                             const BInst *__restrict__ inst,
                                                             const float *__restrict__ g2d,
                                                             const uint32_t *__restrict__ pidx,
                                                             const uint4 *__restrict__ gstate,
                                                             Part4 *__restrict__ part) {
  const int begin = cbeg[blockIdx.x], end = cbeg[blockIdx.x + 1];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int it = begin + wib; it < end; it += nw) {
    const Item I = items[it];
    const BInst B = inst[item_inst[it]];
    const uint4 ss = __ldg(gstate + I.row);
    const float2 *__restrict__ tab = B.tab + (B.cpad - rec_lnm(ss));
    const uint4 *__restrict__ gsi = gstate + B.soff;
    const int nm = B.nm;
    const float *__restrict__ gq = g2d + B.doff + (I.start + lane) * nm;  // the pair's nm branches
    const uint32_t *__restrict__ pr = pidx + B.poff + I.start + lane;
    const float fs = __uint_as_float(ss.z), fsl = rec_f_lo(ss), es = __uint_as_float(ss.x), esl = rec_eps_lo(ss);
    float sum = 0.f, comp = 0.f;
    uint32_t pn = pr[0];  // the next pair's partner, loaded a step ahead
#pragma unroll 1
    for (int left = I.len; left > 0; --left) {
      const bool gap = pn >> 31;
      const int p = (int)(pn & (kPadBit32 - 1));
      pr += 32;
      if (left > 1) pn = pr[0];
      const uint4 sp = __ldg(gsi + p);
      const float dh = __fsub_rn(es, __uint_as_float(sp.x));
      const float dl = __fsub_rn(esl, rec_eps_lo(sp));
      const float fp = __uint_as_float(sp.z), fpl = rec_f_lo(sp);
      const float P = fs * fp, A = fs - P, Bq = fp - P;
      const float delta = fmaf(fsl, fp, fpl * fs);
      const float alpha = (fs - fp) + (fsl - fpl);
      const float betap = (A + fsl) - delta, gammap = (Bq + fpl) - delta;
      const float2 *__restrict__ tr = tab + rec_lnm(sp);
      auto term = [&](float gv, float2 t) {
        const float a = (dh + t.x) + dl;  // x + w
        const float e = (dh - t.x) + dl;  // x - w
        const float Ga = ex2_approx(a * a * B.k2);
        const float Ge = ex2_approx(e * e * B.k2);
        const float na = alpha * t.y;
        return gv * fmaf(Ge, na + betap, Ga * (na - gammap));
      };
      float acc = 0.f;
      if (nm <= kDenseBranches) {
        // the pair's loads first; even nm: slot offsets are even (doff too: slots come in bundles of 32)
        float gv[kDenseBranches];
        float2 tv[kDenseBranches];
        if ((nm & 1) == 0) {
#pragma unroll
          for (int k = 0; k < kDenseBranches / 2; ++k)
            if (2 * k < nm) {
              const float2 v = __ldcs(reinterpret_cast<const float2 *>(gq) + k);
              gv[2 * k] = v.x;
              gv[2 * k + 1] = v.y;
            }
        } else {
#pragma unroll
          for (int nu = 0; nu < kDenseBranches; ++nu)
            if (nu < nm) gv[nu] = __ldcs(gq + nu);
        }
#pragma unroll
        for (int nu = 0; nu < kDenseBranches; ++nu)
          if (nu < nm) tv[nu] = __ldg(tr + nu);
#pragma unroll
        for (int nu = 0; nu < kDenseBranches; ++nu)
          if (nu < nm) acc += term(gv[nu], tv[nu]);
      } else {
        for (int nu = 0; nu < nm; ++nu) acc += term(__ldcs(gq + nu), __ldg(tr + nu));
      }
      kahan_add(sum, comp, acc);
      if (gap) kahan_add(sum, comp, 0.f);
      gq += 32 * nm;
    }
    const double v = warp_sum_ff(make_float2(sum, -comp));
    if (lane == 0) part[it] = make_part4(v, 0.0, 0.0, 0.0);
  }
}

// smap[moff + local row * ns + p] = the slot of every pair of the items (the map holds ~0 elsewhere)
__global__ void __launch_bounds__(kBlock) k_slot_map_batch(const Item *__restrict__ items,
                                                           const int *__restrict__ item_inst, int nitems,
                                                           const BInst *__restrict__ inst,
                                                           const uint32_t *__restrict__ pidx,
                                                           uint32_t *__restrict__ smap) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int it = warp; it < nitems; it += nwarps) {
    const Item I = items[it];
    const BInst B = inst[item_inst[it]];
    for (int j = 0; j < I.len; ++j) {
      const long long slot = I.start + 32 * j + lane;
      const uint32_t p = pidx[B.poff + slot];
      if (!(p & kPadBit32)) smap[B.moff + (long long)(I.row - B.soff) * B.ns + (p & (kPadBit32 - 1))] = (uint32_t)slot;
    }
  }
}

// g2d values of every stored channel of the batch that has a slot (the array is cleared before)
__global__ void __launch_bounds__(kBlock) k_dense_g2_batch(const Item *__restrict__ items,
                                                           const int *__restrict__ item_inst, int nitems,
                                                           const BInst *__restrict__ inst,
                                                           const uint32_t *__restrict__ col,
                                                           const float *__restrict__ g2,
                                                           const uint32_t *__restrict__ smap,
                                                           float *__restrict__ g2d) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int it = warp; it < nitems; it += nwarps) {
    const Item I = items[it];
    const BInst B = inst[item_inst[it]];
    const uint32_t *__restrict__ sr = smap + B.moff + (long long)(I.row - B.soff) * B.ns;
    for (int j = lane; j < I.len; j += 32) {
      const long long c = I.start + j;
      const float v = g2[c];
      if (v == 0.f) continue;  // row padding (and channels with |g|^2 = 0, whose slot stays 0)
      const unsigned cw = col[c];
      const uint32_t slot = sr[cw & 0xFFFFFFu];
      if (slot != ~0u) g2d[B.doff + (long long)slot * B.nm + (cw >> 24)] = v;
    }
  }
}

// I_r = -cs[r] * (row sum); cs = (2 pi / hbar N_q) / (sqrt(2 pi) sigma) of the row's instance.
// STAGE < 0 writes I; STAGE 0..3 does the RK4 stage arithmetic as k_fin_coll does.
template <int STAGE>
__global__ void k_fin_gbatch(const int *__restrict__ item_ptr, const Part4 *__restrict__ part, int ns,
                             const double *__restrict__ cs, const double *__restrict__ ysrc, double *__restrict__ out,
                             double *__restrict__ f, double *__restrict__ acc, double *__restrict__ y,
                             uint4 *__restrict__ gstate, double dt) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= ns) return;
  double S = 0.0;
  for (int i = item_ptr[r]; i < item_ptr[r + 1]; ++i) S += part[i].x;
  const double I = -cs[r] * S;
  (void)ysrc;
  if (STAGE < 0) {
    out[r] = I;
    return;
  }
  const double fr = f[r];
  double yn;
  if (STAGE == 0) {
    acc[r] = I;
    yn = fr + 0.5 * dt * I;
  } else if (STAGE == 1) {
    acc[r] += 2.0 * I;
    yn = fr + 0.5 * dt * I;
  } else if (STAGE == 2) {
    acc[r] += 2.0 * I;
    yn = fr + dt * I;
  } else {
    yn = fr + dt / 6.0 * (acc[r] + I);
    f[r] = yn;
  }
  y[r] = yn;
  rec_set_f(gstate + r, yn);
}

}  // namespace dev
}  // namespace pb

struct pb_batch {
  int n = 0;
  int64_t ns = 0, nchp = 0, nitems = 0, nitems_cap = 0;
  int sm_count = 0, item_ch = 2048, ctas = 2;
  std::vector<int64_t> soff;       // [n+1] state offsets
  std::vector<int64_t> lenp;       // padded length of every global row
  std::vector<int32_t> row_inst;   // instance of every global row
  std::vector<int64_t> nch;        // [n] stored channels per instance
  // dense pair-major FP32 form (precision 0): |g|^2 of the pairs in reach in slots; the instances'
  // energies and reaches are kept for the plans of other item sizes (the channel lists may be gone)
  bool dense = false;
  float *g2d = nullptr;
  uint32_t *pidx0 = nullptr, *smap = nullptr;
  int32_t *cbeg = nullptr;         // item ranges of the CTAs, one table per CTAs-per-SM choice
  int64_t slot_cap = 0, value_cap = 0, map_size = 0;
  std::vector<double> heps, reach;           // [ns], [n]
  std::vector<pb::dev::BInst> hinst;         // [n]
  char *arena = nullptr;
  size_t bytes = 0;
  Item *items = nullptr;
  int32_t *item_inst = nullptr, *item_ptr = nullptr;
  uint32_t *col = nullptr;
  float *g2 = nullptr;
  uint4 *gstate = nullptr;
  float2 *tabs = nullptr;
  pb::dev::BInst *inst = nullptr;
  double *cs = nullptr;
  Part4 *part = nullptr;
  double *acc = nullptr, *y = nullptr;
  // precision 1 (FP64-accurate, branch-merged): per-entry coefficients and global partner
  // indices, per-state R (with the instance's prefactor folded in) and float-float stage input
  int prec = 0;
  float2 *pA = nullptr, *pB = nullptr, *yff = nullptr;
  float2 *pC = nullptr;  // precision 2: rounded FP32 (P_in, P_out) per entry
  uint32_t *pidx = nullptr;
  double *Rg = nullptr;
  // symmetric tiles (precision >= 1; TilePlan): tnt tiles; launch shape tshape (float-float: CTAs
  // per SM of the half-tile ring, 2 or 3; FP32 pairs: the C32 shape number 2..8)
  bool tiles = false;
  int tnt = 0, tshape = 0;
  int rev = 0;  // the next tile sweep takes the tile list from its end (alternating RK4 stages)
  pb::dev::TileD *tl = nullptr;
  int *pmap = nullptr;
  int2 *prow = nullptr, *tbase = nullptr;
  long long *srp = nullptr;
  void *tc = nullptr, *tp = nullptr;
  int *err = nullptr;
  cudaStream_t cap = nullptr;
  cudaGraphExec_t exec = nullptr;
  double *rk_f = nullptr;
  double rk_dt = 0.0;
};

namespace {

struct BatchPlan {
  std::vector<Item> items;
  std::vector<int32_t> item_inst, item_ptr;
};

void batch_plan(const pb_batch *b, int item_ch, BatchPlan &P) {
  P.items.clear();
  P.item_inst.clear();
  P.item_ptr.assign(b->ns + 1, 0);
  int64_t off = 0;
  for (int64_t r = 0; r < b->ns; ++r) {
    P.item_ptr[r] = (int32_t)P.items.size();
    const int64_t lenp = b->lenp[r];
    if (lenp > 0) {
      const int64_t chunks = lenp / kRowPad;
      const int64_t np = std::max<int64_t>(1, (lenp + item_ch - 1) / item_ch);
      int64_t o = 0;
      for (int64_t k = 0; k < np; ++k) {
        const int64_t c = chunks / np + (k < chunks % np ? 1 : 0);
        if (c > 0) {
          Item it;
          it.start = off + o;
          it.len = (int)(c * kRowPad);
          it.row = (int)r;
          P.items.push_back(it);
          P.item_inst.push_back(b->row_inst[r]);
        }
        o += c * kRowPad;
      }
    }
    off += lenp;
  }
  P.item_ptr[b->ns] = (int32_t)P.items.size();
}

int64_t batch_items_count(const std::vector<int64_t> &lenp, int item_ch) {
  int64_t n = 0;
  for (int64_t l : lenp)
    if (l > 0) n += std::max<int64_t>(1, (l + item_ch - 1) / item_ch);
  return n;
}

// Dense pair-major FP32 batch (pb_batch_opts.layout 0 with precision 0): used when the stored
// channels fill at least 85% of all instances' (state, partner, branch) slots; npp = nstate
// rounded up to 32.  A piece of a row (LanePlan) takes item_ch / 4 partners (at least 32).
int64_t batch_npp(int64_t ns) { return (ns + 31) / 32 * 32; }
bool batch_dense_for(const pb_channels *const *chs, int32_t n, const pb_batch_opts &o) {
  if (o.precision != 0 || o.layout != 0) return false;
  int64_t nch = 0, slots = 0;
  for (int i = 0; i < n; ++i) {
    if (chs[i]->nstate > 60000) return false;  // slots (at most 1.1 per pair) are numbered in 32 bits
    nch += chs[i]->nch;
    slots += chs[i]->nstate * batch_npp(chs[i]->nstate) * chs[i]->nmodes;
  }
  return (double)nch >= 0.85 * (double)slots;
}
int batch_dense_part(int item_ch) { return std::max(32, item_ch / 4 / 8 * 8); }
// What the arena reserves, for the autotuner's item sizes and the batch's own: a row's bundles hold its
// pairs in reach and, since each is as long as its longest chain, at most 32 times the longest chain
// more; nor can they hold more than the pieces do with every lane as long as the piece's longest (the
// chains sorted by length never need more steps than piece by piece).
struct BatchDenseCaps {
  int64_t items = 0, slots = 0, values = 0, map = 0;
};
BatchDenseCaps batch_dense_caps(const pb_channels *const *chs, int32_t n, int item_ch) {
  BatchDenseCaps C;
  for (int i = 0; i < n; ++i) {
    const int64_t ns = chs[i]->nstate, npp = batch_npp(ns);
    std::vector<double> e(chs[i]->eps.begin(), chs[i]->eps.begin() + ns);
    std::sort(e.begin(), e.end());
    const double reach = energy_reach_f32(chs[i]);
    std::vector<int64_t> near((size_t)ns);  // pairs in reach of every state, in energy order
    for (int64_t r = 0, a = 0, b = 0; r < ns; ++r) {
      while (e[r] - e[a] > reach) ++a;
      while (b < ns && e[b] - e[r] <= reach) ++b;
      near[r] = b - a;
    }
    int64_t slots = 0;
    for (const int item : {1024, 2048, 4096, item_ch}) {
      if (item <= 0) continue;
      int64_t longest = 0, pieces = 0, s = 0;  // 32 times the longest lane of any piece, of all pieces
      for (const int64_t n : lane_pieces(npp, batch_dense_part(item))) {
        longest = std::max(longest, (n + 31) / 32 * 32);
        pieces += (n + 31) / 32 * 32;
      }
      for (const int64_t p : near) s += std::min(p + longest, pieces);
      slots = std::max(slots, s);
    }
    C.items += ns * std::max<int64_t>(1, (npp + batch_dense_part(1024) - 1) / batch_dense_part(1024));
    C.slots += slots;
    C.values += slots * chs[i]->nmodes;
    C.map += ns * ns;
  }
  return C;
}

constexpr int kBatchMinItem = 1024;  // smallest item size the arena is planned for

struct BatchLayout {
  size_t items, item_inst, item_ptr, col, g2, gstate, tabs, inst, cs, part, acc, y, omega_tmp, tab_tmp, eps_tmp,
      kc_tmp, g2d, pidx, smap, cbeg, total;
};

BatchLayout batch_layout(const pb_channels *const *chs, int n, int64_t ns, int64_t nchp, int64_t nitems_cap,
                         const BatchDenseCaps &dc, int sm) {
  BatchLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + std::max<size_t>(bytes, 1));
    return at;
  };
  size_t tab = 0, maxq = 0, maxs = 0;
  for (int i = 0; i < n; ++i) {
    size_t r = 1;
    for (int a = 0; a < 3; ++a) r *= (size_t)(chs[i]->nk[a] > 1 ? 2 * chs[i]->nk[a] : 1);
    tab += align_up(sizeof(float2) * r * chs[i]->nmodes);
    maxq = std::max(maxq, (size_t)chs[i]->nq * chs[i]->nmodes);
    maxs = std::max(maxs, (size_t)chs[i]->nstate);
  }
  L.items = take(sizeof(Item) * nitems_cap);
  L.item_inst = take(sizeof(int32_t) * nitems_cap);
  L.item_ptr = take(sizeof(int32_t) * (ns + 1));
  L.col = take(sizeof(uint32_t) * nchp);
  L.g2 = take(sizeof(float) * nchp);
  L.gstate = take(sizeof(uint4) * ns);
  L.tabs = take(tab);
  L.inst = take(sizeof(pb::dev::BInst) * n);
  L.cs = take(sizeof(double) * ns);
  L.part = take(sizeof(Part4) * nitems_cap);
  L.acc = take(sizeof(double) * ns);
  L.y = take(sizeof(double) * ns);
  L.omega_tmp = take(sizeof(double) * maxq);
  L.tab_tmp = take(sizeof(double2) * maxq);
  L.eps_tmp = take(sizeof(double) * maxs);
  L.kc_tmp = take(sizeof(short4) * maxs);
  L.g2d = take(sizeof(float) * (size_t)dc.values);
  L.pidx = take(sizeof(uint32_t) * (size_t)dc.slots);
  L.smap = take(sizeof(uint32_t) * (size_t)dc.map);
  L.cbeg = take(dc.slots ? sizeof(int32_t) * 4 * ((size_t)sm * 4 + 1) : 0);
  L.total = o;
  return L;
}

// Sweep entries per row of the FP64-accurate batch: one per run of equal partner (state pair),
// padded to kRowPad.
std::vector<int64_t> batch_pair_lenp(const pb_channels *const *chs, int32_t n) {
  int64_t total = 0;
  for (int i = 0; i < n; ++i) total += chs[i]->nstate;
  std::vector<int64_t> lenp((size_t)total);
  int64_t off = 0;
  for (int i = 0; i < n; ++i) {
    const pb_channels *ch = chs[i];
#pragma omp parallel for schedule(dynamic, 16)
    for (int64_t r = 0; r < ch->nstate; ++r) {
      int64_t runs = 0;
      for (int64_t c = ch->row_ptr[r]; c < ch->row_ptr[r + 1]; ++c)
        if (c == ch->row_ptr[r] || ch->col[c] != ch->col[c - 1]) ++runs;
      lenp[off + r] = (runs + kRowPad - 1) / kRowPad * kRowPad;
    }
    off += ch->nstate;
  }
  return lenp;
}

// The symmetric-tile form of a precision >= 1 batch (layout 2: always; layout 0: taken when every instance's
// channel list was verified closed (the tile entry of (s, p) serves the reverse pair with
// P_in and P_out swapped) and the tiles stream at most 0.7 of the rows' bytes (the row stream
// runs closer to the copy bandwidth; sparse rows, or many instances much smaller than a
// 64-state block, fill the tiles with zeros).
struct BatchTiles : TilePlan {
  bool on = false;
};
// nent: the padded pair entries of all rows; lenp: those of every row (batch_pair_lenp)
BatchTiles batch_tiles_for(const pb_channels *const *chs, int32_t n, int prec, int layout,
                           const std::vector<int64_t> &lenp, int sm) {
  BatchTiles T;
  if (prec < 1 || layout == 1) return T;
  int64_t nent = 0, so = 0;
  for (const int64_t l : lenp) nent += l;
  for (int i = 0; i < n; ++i)
    if (!chs[i]->closed) return T;
  for (int i = 0; i < n; ++i) {
    const pb_channels *ch = chs[i];
    // rows as long as complete ones (up to the padding): the reach alone bounds the tiles
    bool complete = true;
    const int64_t full = (ch->nstate + kRowPad - 1) / kRowPad * kRowPad;
    for (int64_t r = 0; r < ch->nstate; ++r) complete = complete && lenp[so + r] == full;
    so += ch->nstate;
    tile_plan_add(ch, prec == 1, complete, energy_reach(ch, ch->g2_max), T);
  }
  const int64_t nt = (int64_t)T.tiles.size();
  if (nt == 0 || nt >= INT32_MAX / 2 || T.npart >= INT32_MAX) return T;
  const double row_bytes = (double)nent * (prec == 2 ? 12.0 : 20.0);
  auto pay = [&](int64_t tiles) {
    return (double)tiles * dev::kTile * dev::kTile * (prec == 2 ? 8.0 : 16.0) <= 0.7 * row_bytes;
  };
  T.band = layout != 2 && !pay(T.nt_full);
  T.on = !T.band || pay(nt);
  if (T.on && prec == 1 && chain_pdl(nt, sm)) tile_plan_halve(T);
  return T;
}

struct BatchLayoutFF {
  size_t items, item_inst, item_ptr, pA, pB, pC, pidx, Rg, yff, part, acc, y, tcol, tg2, tcA, tcB, titems, titem_ptr,
      tpart, tR, tpcst, tpcnt, omega_tmp, tab_tmp, eps_tmp, kc_tmp, srp, tl, pmap, prow, tbase, tc, tp, err, total;
};

constexpr int kBatchSetupItem = 2048;  // channels per work item of the per-instance coefficient setup

// c32: precision 2 (the rounded FP32 pairs of the rows, or FP32 tiles); T: the tile form;
// lenp: the padded pair entries of every row (batch_pair_lenp)
BatchLayoutFF batch_layout_ff(const pb_channels *const *chs, int n, int64_t ns, int64_t nent, int64_t nitems_cap,
                              bool c32, const BatchTiles &T, const std::vector<int64_t> &lenp) {
  BatchLayoutFF L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + std::max<size_t>(bytes, 1));
    return at;
  };
  size_t maxq = 0, maxs = 0, maxc = 0, maxp = 0, maxi = 0;
  int64_t so = 0;
  for (int i = 0; i < n; ++i) {
    const pb_channels *ch = chs[i];
    size_t c = 0, p = 0, it = 0;
    for (int64_t r = 0; r < ch->nstate; ++r) {
      const int64_t len = ch->row_ptr[r + 1] - ch->row_ptr[r], lp = (len + kRowPad - 1) / kRowPad * kRowPad;
      c += (size_t)lp;
      if (lp > 0) it += (size_t)std::max<int64_t>(1, (lp + kBatchSetupItem - 1) / kBatchSetupItem);
      p += (size_t)lenp[so + r];
    }
    so += ch->nstate;
    maxq = std::max(maxq, (size_t)ch->nq * ch->nmodes);
    maxs = std::max(maxs, (size_t)ch->nstate);
    maxc = std::max(maxc, c);
    maxp = std::max(maxp, p);
    maxi = std::max(maxi, it);
  }
  L.items = take(sizeof(Item) * nitems_cap);
  L.item_inst = take(sizeof(int32_t) * nitems_cap);
  L.item_ptr = take(sizeof(int32_t) * (ns + 1));
  L.pA = take(sizeof(float2) * nent);
  L.pB = take(sizeof(float2) * nent);
  L.pC = take(c32 && !T.on ? sizeof(float2) * nent : 0);
  L.pidx = take(sizeof(uint32_t) * nent);
  L.Rg = take(sizeof(double) * ns);
  L.yff = take(T.on ? sizeof(float4) * T.nsp : sizeof(float2) * ns);  // tiles: the padded state space
  L.part = take(sizeof(Part4) * nitems_cap);
  L.acc = take(sizeof(double) * ns);
  L.y = take(sizeof(double) * ns);
  L.tcol = take(sizeof(uint32_t) * maxc);
  L.tg2 = take(sizeof(double) * maxc);
  L.tcA = take(sizeof(float2) * maxc);
  L.tcB = take(sizeof(float2) * maxc);
  L.titems = take(sizeof(Item) * maxi);
  L.titem_ptr = take(sizeof(int32_t) * (maxs + 1));
  L.tpart = take(sizeof(Part4) * maxi);
  L.tR = take(sizeof(double) * maxs);
  L.tpcst = take(sizeof(int64_t) * maxp);
  L.tpcnt = take(maxp);
  L.omega_tmp = take(sizeof(double) * maxq);
  L.tab_tmp = take(sizeof(double2) * maxq);
  L.eps_tmp = take(sizeof(double) * maxs);
  L.kc_tmp = take(sizeof(short4) * maxs);
  const size_t te = c32 ? sizeof(float2) : sizeof(float4), pe = c32 ? sizeof(float) : sizeof(float4);
  L.srp = take(T.on ? sizeof(int64_t) * (ns + 1) : 0);
  L.tl = take(T.on ? sizeof(dev::TileD) * T.tiles.size() : 0);
  L.pmap = take(T.on ? sizeof(int32_t) * ns : 0);
  L.prow = take(T.on ? sizeof(int2) * ns : 0);
  L.tbase = take(T.on ? sizeof(int2) * T.nb : 0);
  L.tc = take(T.on ? te * (size_t)T.tiles_reserved() * dev::kTile * dev::kTile : 0);
  L.tp = take(T.on ? T.part_bytes(pe) : 0);
  L.err = take(sizeof(int));
  L.total = o;
  return L;
}

int batch_check(const pb_channels *const *chs, int32_t n, int64_t *ns, int64_t *nchp) {
  if (!chs || n <= 0) return set_error(PB_EINVAL, "pb_batch: need at least one channel list");
  int64_t s = 0, c = 0;
  for (int i = 0; i < n; ++i) {
    if (!chs[i]) return set_error(PB_EINVAL, "pb_batch: channel list %d is null", i);
    s += chs[i]->nstate;
    for (int64_t r = 0; r < chs[i]->nstate; ++r)
      c += (chs[i]->row_ptr[r + 1] - chs[i]->row_ptr[r] + kRowPad - 1) / kRowPad * kRowPad;
  }
  if (s >= INT32_MAX / 4) return set_error(PB_EINVAL, "pb_batch: too many states");
  *ns = s;
  *nchp = c;
  return PB_OK;
}

std::vector<int64_t> batch_lenp(const pb_channels *const *chs, int32_t n) {
  std::vector<int64_t> lenp;
  for (int i = 0; i < n; ++i)
    for (int64_t r = 0; r < chs[i]->nstate; ++r)
      lenp.push_back((chs[i]->row_ptr[r + 1] - chs[i]->row_ptr[r] + kRowPad - 1) / kRowPad * kRowPad);
  return lenp;
}

int batch_dense_grid(int64_t nitems, int sm_count, int ctas) {
  const int64_t need = (nitems * 32 + 511) / 512;
  return (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sm_count * ctas));
}

int batch_upload_items(pb_batch *b, const BatchPlan &P, int item_ch, cudaStream_t st) {
  if ((int64_t)P.items.size() > b->nitems_cap)
    return set_error(PB_EINVAL, "pb_batch: item size %d needs more items than the arena holds", item_ch);
  PB_CUDA(cudaMemcpyAsync(b->items, P.items.data(), sizeof(Item) * P.items.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->item_inst, P.item_inst.data(), sizeof(int32_t) * P.item_inst.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->item_ptr, P.item_ptr.data(), sizeof(int32_t) * P.item_ptr.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaStreamSynchronize(st));  // the plan vectors are released on return
  b->nitems = (int64_t)P.items.size();
  b->item_ch = item_ch;
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  return PB_OK;
}

// The dense form's plan for an item size: the instances' lane plans, the slot map, the |g|^2 values
// scattered into the slots from the channel list, and the CTAs' item ranges.  Everything that can fail
// on the host comes before the first change on the device: after an error the plan before it is whole.
int batch_upload_dense(pb_batch *b, int item_ch, cudaStream_t st) {
  BatchPlan D, C;
  std::vector<uint32_t> pidx;
  std::vector<pb::dev::BInst> inst = b->hinst;
  int64_t values = 0, map = 0;
  for (int i = 0; i < b->n; ++i) {
    const int64_t s0 = b->soff[i], ns = b->soff[i + 1] - s0;
    LanePlan<uint32_t> P;
    lane_plan(b->heps.data() + s0, ns, batch_npp(ns), batch_dense_part(item_ch), b->reach[i], true, P);
    auto &B = inst[i];
    B.doff = values;
    B.poff = (long long)pidx.size();
    B.moff = map;
    values += P.slots * B.nm;
    map += ns * ns;
    pidx.insert(pidx.end(), P.pidx.begin(), P.pidx.end());
    for (int64_t r = 0; r < ns; ++r) D.item_ptr.push_back((int32_t)D.items.size() + P.item_ptr[r]);
    for (Item it : P.items) {
      it.row += (int)s0;
      D.items.push_back(it);
      D.item_inst.push_back(i);
    }
  }
  D.item_ptr.push_back((int32_t)D.items.size());
  if ((int64_t)pidx.size() > b->slot_cap || values > b->value_cap)
    return set_error(PB_EINVAL, "pb_batch: item size %d needs more slots than the arena holds", item_ch);
  batch_plan(b, 2048, C);  // the channel list's own items, for the scatter
  const int64_t nitems = (int64_t)D.items.size();
  if (std::max(nitems, (int64_t)C.items.size()) > b->nitems_cap)
    return set_error(PB_EINVAL, "pb_batch: item size %d needs more items than the arena holds", item_ch);
  // per CTAs-per-SM choice, item ranges of about equal work (steps times branches)
  std::vector<int64_t> cost((size_t)nitems + 1, 0);
  for (int64_t i = 0; i < nitems; ++i)
    cost[i + 1] = cost[i] + (int64_t)D.items[i].len * (2 + inst[D.item_inst[i]].nm) + 4;
  const int stride = b->sm_count * 4 + 1;
  std::vector<int32_t> cb((size_t)4 * stride, (int32_t)nitems);
  for (int c = 1; c <= 4; ++c) {
    const int g = batch_dense_grid(nitems, b->sm_count, c);
    for (int k = 0; k <= g; ++k)
      cb[(size_t)(c - 1) * stride + k] =
          (int32_t)(std::lower_bound(cost.begin(), cost.end(), cost[nitems] * k / g) - cost.begin());
  }
  b->hinst.swap(inst);
  int rc;
  PB_CUDA(cudaMemcpyAsync(b->inst, b->hinst.data(), sizeof(pb::dev::BInst) * b->hinst.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->pidx0, pidx.data(), sizeof(uint32_t) * pidx.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemsetAsync(b->smap, 0xFF, sizeof(uint32_t) * (size_t)b->map_size, st));
  PB_CUDA(cudaMemsetAsync(b->g2d, 0, sizeof(float) * (size_t)values, st));
  auto grid = [&] {
    const int64_t need = (b->nitems * 32 + dev::kBlock - 1) / dev::kBlock;
    return (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)b->sm_count * 8));
  };
  if ((rc = batch_upload_items(b, D, item_ch, st))) return rc;
  dev::k_slot_map_batch<<<grid(), dev::kBlock, 0, st>>>(b->items, b->item_inst, (int)b->nitems, b->inst, b->pidx0, b->smap);
  PB_LAUNCHED("k_slot_map_batch");
  if ((rc = batch_upload_items(b, C, 2048, st))) return rc;
  dev::k_dense_g2_batch<<<grid(), dev::kBlock, 0, st>>>(b->items, b->item_inst, (int)b->nitems, b->inst, b->col, b->g2,
                                                        b->smap, b->g2d);
  PB_LAUNCHED("k_dense_g2_batch");
  PB_CUDA(cudaStreamSynchronize(st));
  if ((rc = batch_upload_items(b, D, item_ch, st))) return rc;
  PB_CUDA(cudaMemcpyAsync(b->cbeg, cb.data(), sizeof(int32_t) * cb.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaStreamSynchronize(st));
  return PB_OK;
}

int batch_upload_plan(pb_batch *b, int item_ch, cudaStream_t st) {
  try {
    if (b->dense) return batch_upload_dense(b, item_ch, st);
    BatchPlan P;
    batch_plan(b, item_ch, P);
    return batch_upload_items(b, P, item_ch, st);
  } catch (const std::bad_alloc &) {
    return set_error(PB_ENOMEM, "pb_batch: out of host memory");
  }
}

// the tile sweep of every instance in one launch (the single-system kernels)
int batch_sweep_tiles(pb_batch *b, cudaStream_t st) {
  const int nt = b->tnt;
  const bool chain = chain_pdl(nt, b->sm_count);
  if (b->prec == 1)
    launch_half_tiles<dev::MODE_COLL>(chain, b->tshape, b->sm_count, b->tl, nt, (const float4 *)b->tc, b->yff, b->tp,
                                      b->err, b->rev, st);
  else
    with_bool(chain, [&](auto pdl) {
      with_c32_shape(b->tshape, [&](auto nst, auto cps, auto half) {
        const int gs = (int)std::max<int64_t>(1, std::min<int64_t>(nt, (int64_t)b->sm_count * cps()));
        const float2 *tc = (const float2 *)b->tc;
        float *tp = (float *)b->tp;
        if constexpr (decltype(half)::value)
          launch_pdl(pdl(), dev::k_stream_c32_half<dev::MODE_COLL, nst(), cps(), pdl()>, gs, dev::kC32Threads,
                     dev::c32_half_smem<nst()>(), st, b->tl, nt, tc, b->yff, tp, b->err, b->rev);
        else
          launch_pdl(pdl(), dev::k_stream_c32<dev::MODE_COLL, nst(), cps(), pdl()>, gs, dev::kC32Threads,
                     dev::c32_smem<nst()>(), st, b->tl, nt, tc, b->yff, tp, b->err, b->rev);
      });
    });
  PB_LAUNCHED("tile sweep (batch)");
  return PB_OK;
}

int batch_sweep(pb_batch *b, cudaStream_t st) {
  if (b->tiles) return batch_sweep_tiles(b, st);
  if (b->prec == 2) {
    const int64_t need = (b->nitems * 32 + dev::kBlock - 1) / dev::kBlock;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)b->sm_count * b->ctas));
    pb::dev::k_stream_c32_rows<uint32_t><<<grid, dev::kBlock, 0, st>>>(b->items, (int)b->nitems,
                                                                        (const float4 *)b->pC, b->pidx, b->yff,
                                                                        b->part);
    PB_LAUNCHED("k_stream_c32_rows (batch)");
    return PB_OK;
  }
  if (b->prec == 1) {
    const int64_t need = (b->nitems * 32 + dev::kBlock - 1) / dev::kBlock;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)b->sm_count * b->ctas));
    pb::dev::k_stream_ff<dev::MODE_COLL, false, uint32_t><<<grid, dev::kBlock, 0, st>>>(
        b->items, (int)b->nitems, (const float4 *)b->pA, (const float4 *)b->pB, b->pidx, b->yff, (int)b->ns, b->part);
    PB_LAUNCHED("k_stream_ff (batch)");
    return PB_OK;
  }
  const int grid = batch_dense_grid(b->nitems, b->sm_count, b->ctas);  // of 512 threads
  if (b->dense) {
    pb::dev::k_stream_gbatch_dense<<<grid, 512, 0, st>>>(b->items, b->item_inst,
                                                          b->cbeg + (size_t)(b->ctas - 1) * (b->sm_count * 4 + 1),
                                                          b->inst, b->g2d, b->pidx0, b->gstate, b->part);
    PB_LAUNCHED("k_stream_gbatch_dense");
    return PB_OK;
  }
  pb::dev::k_stream_gbatch<dev::MODE_COLL><<<grid, 512, 0, st>>>(b->items, b->item_inst, (int)b->nitems, b->inst,
                                                                 b->col, b->g2, b->gstate, b->part);
  PB_LAUNCHED("k_stream_gbatch");
  return PB_OK;
}

// src: the stage input (f for STAGE <= 0, y after), read by the FP64-accurate epilogue
template <int STAGE>
int batch_fin(pb_batch *b, double *out, double *f, double dt, cudaStream_t st, const double *src) {
  if (b->tiles) {
    // the instances' prefactors are folded into the tiles: c = 1; states index f, y and the
    // outputs, their padded rows the partials and the next stage's float-float input
    const int ns = (int)b->ns;
    with_bool(chain_pdl(b->tnt, b->sm_count), [&](auto pdl) {
      with_bool(fin_small(ns, b->sm_count), [&](auto small) {
        constexpr int SPC = small() ? 8 : 32;
        const int grid = (ns + SPC - 1) / SPC;
        if (b->prec == 2)
          launch_pdl(pdl(), dev::k_fin_net<float, STAGE, false, SPC, pdl()>, grid, 256, 0, st, (const float *)b->tp,
                     b->prow, b->pmap, ns, 1.0, nullptr, out, f, b->acc, b->y, b->yff, dt);
        else
          launch_pdl(pdl(), dev::k_fin_net<float2, STAGE, false, SPC, pdl()>, grid, 256, 0, st, (const float2 *)b->tp,
                     b->prow, b->pmap, ns, 1.0, nullptr, out, f, b->acc, b->y, b->yff, dt);
      });
    });
    PB_LAUNCHED("tile epilogue (batch)");
    return PB_OK;
  }
  if (b->prec == 2) {
    // the partials are sums of t (prefactors folded in): the plain-sum epilogue with c = -1 gives
    // I = -c A = A; it writes the next stage's float-float input like the FF batch
    pb::dev::k_fin_coll<true, STAGE><<<(int)((b->ns + 255) / 256), 256, 0, st>>>(
        pb::dev::ItemSrc{b->item_ptr, b->part}, (int)b->ns, -1.0, nullptr, src, out, f, b->acc, b->y, b->yff, dt);
    PB_LAUNCHED("k_fin_coll (batch, FP32 pairs)");
    return PB_OK;
  }
  if (b->prec == 1) {
    pb::dev::k_fin_coll<false, STAGE><<<(int)((b->ns + 255) / 256), 256, 0, st>>>(
        pb::dev::ItemSrc{b->item_ptr, b->part}, (int)b->ns, 1.0, b->Rg, src, out, f, b->acc, b->y, b->yff, dt);
    PB_LAUNCHED("k_fin_coll (batch)");
    return PB_OK;
  }
  (void)src;
  pb::dev::k_fin_gbatch<STAGE><<<(int)((b->ns + 255) / 256), 256, 0, st>>>(b->item_ptr, b->part, (int)b->ns, b->cs,
                                                                            nullptr, out, f, b->acc, b->y, b->gstate, dt);
  PB_LAUNCHED("k_fin_gbatch");
  return PB_OK;
}

int batch_stage_input(pb_batch *b, const double *f, cudaStream_t st) {
  if (b->tiles) {
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((b->ns + 255) / 256, 1024));
    if (b->prec == 1) dev::k_f0_map<<<grid, 256, 0, st>>>(f, (int)b->ns, b->pmap, (float4 *)b->yff);
    else dev::k_to_ff_map<<<grid, 256, 0, st>>>(f, (int)b->ns, b->pmap, b->yff);
    PB_LAUNCHED("stage input (batch tiles)");
    return PB_OK;
  }
  if (b->prec >= 1) {
    dev::k_to_ff<<<(int)std::max<int64_t>(1, std::min<int64_t>((b->ns + 255) / 256, 1024)), 256, 0, st>>>(
        f, (long long)b->ns, b->yff);
    PB_LAUNCHED("k_to_ff (batch)");
    return PB_OK;
  }
  dev::k_gstate_f<<<(int)((b->ns + 255) / 256), 256, 0, st>>>(f, (int)b->ns, b->gstate);
  PB_LAUNCHED("k_gstate_f");
  return PB_OK;
}

// the tile sweeps of stages 2 and 4 take the tile list from its end (each starts on the tiles
// the sweep before it left in L2)
int batch_rk4_stages(pb_batch *b, double *f, double dt, cudaStream_t st) {
  int rc;
  b->rev = 0;
  if ((rc = batch_sweep(b, st)) || (rc = batch_fin<0>(b, nullptr, f, dt, st, f))) return rc;
  b->rev = 1;
  if ((rc = batch_sweep(b, st)) || (rc = batch_fin<1>(b, nullptr, f, dt, st, b->y))) return rc;
  b->rev = 0;
  if ((rc = batch_sweep(b, st)) || (rc = batch_fin<2>(b, nullptr, f, dt, st, b->y))) return rc;
  b->rev = 1;
  if ((rc = batch_sweep(b, st)) || (rc = batch_fin<3>(b, nullptr, f, dt, st, b->y))) return rc;
  return PB_OK;
}

int batch_rk4_launches(pb_batch *b, double *f, double dt, cudaStream_t st) {
  const int rc = batch_rk4_stages(b, f, dt, st);
  b->rev = 0;
  return rc;
}

}  // namespace

namespace {

// Precision 1: per instance, the per-channel coefficients in FP64 on its own geometry
// (k_coef over temporaries), R_s, the branch sums scaled by its prefactor into the shared
// arrays, and the global partner indices.
int batch_setup_ff(pb_batch *b, const pb_channels *const *chs, int n, const BatchLayoutFF &L, cudaStream_t st) {
  char *A = b->arena;
  uint32_t *tcol = (uint32_t *)(A + L.tcol);
  double *tg2 = (double *)(A + L.tg2);
  float2 *tcA = (float2 *)(A + L.tcA), *tcB = (float2 *)(A + L.tcB);
  Item *titems = (Item *)(A + L.titems);
  int32_t *titem_ptr = (int32_t *)(A + L.titem_ptr);
  Part4 *tpart = (Part4 *)(A + L.tpart);
  double *tR = (double *)(A + L.tR);
  int64_t *tpcst = (int64_t *)(A + L.tpcst);
  uint8_t *tpcnt = (uint8_t *)(A + L.tpcnt);
  double *om = (double *)(A + L.omega_tmp);
  double2 *tt = (double2 *)(A + L.tab_tmp);
  double *ep = (double *)(A + L.eps_tmp);
  short4 *kc = (short4 *)(A + L.kc_tmp);
  int64_t poff = 0;  // first sweep entry of the instance
  for (int i = 0; i < n; ++i) {
    const pb_channels *ch = chs[i];
    const int64_t ns_i = ch->nstate, so = b->soff[i];
    if (ch->nk[0] > 32767 || ch->nk[1] > 32767 || ch->nk[2] > 32767)
      return set_error(PB_EINVAL, "pb_batch_create: instance %d grid dimension above 32767", i);
    // host: padded channel layout, setup items, pair entries
    std::vector<int64_t> rp((size_t)ns_i + 1, 0);
    for (int64_t r = 0; r < ns_i; ++r)
      rp[r + 1] = rp[r] + (ch->row_ptr[r + 1] - ch->row_ptr[r] + kRowPad - 1) / kRowPad * kRowPad;
    const int64_t nc = rp[ns_i];
    // first pair entry of every row, then the rows filled in parallel (each writes only its own
    // ranges; the arrays are filled, not zeroed first)
    std::vector<int64_t> pe((size_t)ns_i + 1, 0);
    for (int64_t r = 0; r < ns_i; ++r) pe[r + 1] = pe[r] + b->lenp[so + r];
    const int64_t np = pe[ns_i];
    std::unique_ptr<uint32_t[]> hcol(new uint32_t[(size_t)nc]);
    std::unique_ptr<double[]> hg2(new double[(size_t)nc]);
    std::unique_ptr<uint32_t[]> hpidx(new uint32_t[(size_t)np]);
    std::unique_ptr<int64_t[]> hcst(new int64_t[(size_t)np]);
    std::unique_ptr<uint8_t[]> hcnt(new uint8_t[(size_t)np]);
#pragma omp parallel for schedule(dynamic, 16)
    for (int64_t r = 0; r < ns_i; ++r) {
      const int64_t a = ch->row_ptr[r], len = ch->row_ptr[r + 1] - a;
      for (int64_t k = 0; k < len; ++k) {
        hcol[rp[r] + k] = (uint32_t)ch->col[a + k] | ((uint32_t)ch->nu[a + k] << kPartnerBits);
        hg2[rp[r] + k] = ch->g2[a + k];
      }
      for (int64_t k = len; k < rp[r + 1] - rp[r]; ++k) {
        hcol[rp[r] + k] = (uint32_t)r;
        hg2[rp[r] + k] = 0.0;
      }
      int64_t e = pe[r];
      for (int64_t k = 0; k < len; ++k) {
        if (k > 0 && ch->col[a + k] == ch->col[a + k - 1]) {
          ++hcnt[e - 1];
          continue;
        }
        hpidx[e] = (uint32_t)(so + ch->col[a + k]);
        hcst[e] = rp[r] + k;
        hcnt[e] = 1;
        ++e;
      }
      for (; e < pe[r + 1]; ++e) {
        hpidx[e] = (uint32_t)(so + r);
        hcst[e] = 0;
        hcnt[e] = 0;
      }
    }
    std::vector<Item> hit;
    std::vector<int32_t> hptr;
    plan_items(rp, kBatchSetupItem, hit, hptr);
    std::vector<short4> hkc((size_t)ns_i);
    const int N2 = ch->nk[1], N3 = ch->nk[2];
    for (int64_t r = 0; r < ns_i; ++r) {
      const int ik = ch->kidx[r];
      hkc[r] = make_short4((short)(ik / (N2 * N3)), (short)((ik / N3) % N2), (short)(ik % N3), 0);
    }
    const size_t nq = (size_t)ch->nq * ch->nmodes;
    PB_CUDA(cudaMemcpyAsync(tcol, hcol.get(), sizeof(uint32_t) * nc, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(tg2, hg2.get(), sizeof(double) * nc, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(titems, hit.data(), sizeof(Item) * hit.size(), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(titem_ptr, hptr.data(), sizeof(int32_t) * hptr.size(), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(tpcst, hcst.get(), sizeof(int64_t) * np, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(tpcnt, hcnt.get(), np, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(b->pidx + poff, hpidx.get(), sizeof(uint32_t) * np, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(om, ch->omega.data(), sizeof(double) * nq, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(ep, ch->eps.data(), sizeof(double) * ns_i, cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(kc, hkc.data(), sizeof(short4) * ns_i, cudaMemcpyHostToDevice, st));
    dev::k_table<<<(int)std::min<size_t>((nq + 255) / 256, 4096), 256, 0, st>>>(om, (long long)nq, kBoltz * ch->T, tt);
    PB_LAUNCHED("k_table (batch)");
    dev::ChanGeom g;
    g.col = tcol;
    g.g2 = tg2;
    g.eps = ep;
    g.kc = kc;
    g.tab = tt;
    g.N1 = ch->nk[0];
    g.N2 = ch->nk[1];
    g.N3 = ch->nk[2];
    g.nmodes = ch->nmodes;
    g.inv2s2 = 1.0 / (2.0 * ch->sigma * ch->sigma);
    g.norm = 1.0 / (std::sqrt(2.0 * kPi) * ch->sigma);
    const int nit = (int)hit.size();
    if (nit > 0) {
      const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)nit * 32 + dev::kBlock - 1) / dev::kBlock,
                                                                   (int64_t)b->sm_count * 8));
      dev::k_coef<true><<<grid, dev::kBlock, 0, st>>>(titems, nit, g, tcA, tcB, tpart);
      PB_LAUNCHED("k_coef (batch)");
    }
    const double c = 2.0 * kPi / (kHbar * (double)ch->nq);
    if (ns_i > 0) {
      dev::k_rowsum<<<(int)((ns_i + 255) / 256), 256, 0, st>>>(titem_ptr, tpart, (int)ns_i, tR);
      PB_LAUNCHED("k_rowsum (batch)");
      dev::k_scale_copy<<<(int)((ns_i + 255) / 256), 256, 0, st>>>(tR, (int)ns_i, c, b->Rg + so);
      PB_LAUNCHED("k_scale_copy (batch)");
    }
    if (np > 0) {
      dev::k_pair_coef<true><<<(int)std::min<int64_t>((np + 255) / 256, 8192), 256, 0, st>>>(
          (const long long *)tpcst, tpcnt, (long long)np, tcA, tcB, b->pA + poff, b->pB + poff, c, nullptr);
      PB_LAUNCHED("k_pair_coef (batch)");
    }
    PB_CUDA(cudaStreamSynchronize(st));  // the temporaries are reused by the next instance
    poff += np;
  }
  return PB_OK;
}

// CTAs per SM of a tile launch shape
int batch_tile_cps(const pb_batch *b) {
  if (b->prec != 2) return b->tshape;
  int c = 0;
  with_c32_shape(b->tshape, [&](auto, auto cps, auto) { c = cps(); });
  return c;
}

// The tile form: the plan's tables uploaded, then the tiles zeroed and every stored pair scattered
// into them from the instances' branch-merged pair rows (prefactors folded in).
int batch_setup_tiles(pb_batch *b, const TilePlan &T, cudaStream_t st) {
  std::vector<long long> srp((size_t)b->ns + 1, 0);
  for (int64_t r = 0; r < b->ns; ++r) srp[r + 1] = srp[r] + b->lenp[r];
  PB_CUDA(cudaMemcpyAsync(b->srp, srp.data(), sizeof(long long) * srp.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->tl, T.tiles.data(), sizeof(dev::TileD) * T.tiles.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->pmap, T.pmap.data(), sizeof(int32_t) * T.pmap.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->prow, T.prow.data(), sizeof(int2) * T.prow.size(), cudaMemcpyHostToDevice, st));
  PB_CUDA(cudaMemcpyAsync(b->tbase, T.tbase.data(), sizeof(int2) * T.tbase.size(), cudaMemcpyHostToDevice, st));
  const size_t tbytes = (size_t)b->tnt * dev::kTile * dev::kTile * (b->prec == 2 ? sizeof(float2) : sizeof(float4));
  PB_CUDA(cudaMemsetAsync(b->tc, 0, tbytes, st));
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((b->ns * 32 + 255) / 256, (int64_t)b->sm_count * 8));
  if (b->prec == 2)
    dev::k_tiles_scatter<true, uint32_t><<<grid, 256, 0, st>>>(b->srp, (int)b->ns, b->pidx, b->pA, b->pB, b->pmap,
                                                               b->tbase, b->tc);
  else
    dev::k_tiles_scatter<false, uint32_t><<<grid, 256, 0, st>>>(b->srp, (int)b->ns, b->pidx, b->pA, b->pB, b->pmap,
                                                                b->tbase, b->tc);
  PB_LAUNCHED("k_tiles_scatter (batch)");
  PB_CUDA(cudaStreamSynchronize(st));  // the host tables are released on return
  // dynamic shared memory of every launch shape the autotuner may pick
  if (b->prec == 2)
    for (int shape : {2, 3, 4, 7, 8}) set_c32_smem(shape);
  else
    set_half_smem();
  PB_CUDA(cudaGetLastError());
  return PB_OK;
}

}  // namespace

extern "C" int pb_batch_arena_bytes(const pb_channels *const *chs, int32_t n, const pb_batch_opts *opts,
                                    size_t *bytes) {
  clear_error();
  if (!bytes) return set_error(PB_EINVAL, "pb_batch_arena_bytes: null argument");
  int64_t ns = 0, nchp = 0;
  int rc = batch_check(chs, n, &ns, &nchp);
  if (rc) return rc;
  const int prec = opts ? opts->precision : 0;
  if (prec < 0 || prec > 2) return set_error(PB_EINVAL, "pb_batch: precision must be 0, 1 or 2");
  const int layout = opts ? opts->layout : 0;
  if (layout < 0 || layout > (prec >= 1 ? 2 : 1))
    return set_error(PB_EINVAL, "pb_batch: layout must be 0 or 1 (precision 0), 0..2 (precision 1, 2)");
  if (layout == 2)
    for (int i = 0; i < n; ++i)
      if (!chs[i]->closed)
        return set_error(PB_EINVAL, "pb_batch: layout 2 (symmetric tiles) needs channel lists built with the "
                                    "closure check (list %d was not)", i);
  int sm = 152, devid = 0;
  if (cudaGetDevice(&devid) == cudaSuccess) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, devid);
  else cudaGetLastError();
  try {
    if (prec >= 1) {
      const std::vector<int64_t> lenp = batch_pair_lenp(chs, n);
      int64_t nent = 0;
      for (int64_t l : lenp) nent += l;
      const BatchTiles T = batch_tiles_for(chs, n, prec, opts ? opts->layout : 0, lenp, sm);
      *bytes = batch_layout_ff(chs, n, ns, nent, batch_items_count(lenp, kBatchMinItem), prec == 2, T, lenp).total;
    } else {
      pb_batch_opts o{};
      if (opts) o = *opts;
      const bool dense = batch_dense_for(chs, n, o);
      const BatchDenseCaps dc = dense ? batch_dense_caps(chs, n, o.item_channels) : BatchDenseCaps{};
      const int64_t cap = std::max(batch_items_count(batch_lenp(chs, n), kBatchMinItem), dc.items);
      *bytes = batch_layout(chs, n, ns, nchp, cap, dc, sm).total;
    }
  } catch (const std::bad_alloc &) {
    return set_error(PB_ENOMEM, "pb_batch_arena_bytes: out of host memory");
  }
  return PB_OK;
}

extern "C" int pb_batch_create(const pb_channels *const *chs, int32_t n, const pb_batch_opts *opts, void *arena,
                               size_t bytes, void *stream, pb_batch **out) {
  clear_error();
  if (!arena || !out) return set_error(PB_EINVAL, "pb_batch_create: null argument");
  *out = nullptr;
  if (((uintptr_t)arena) % kAlign) return set_error(PB_EINVAL, "pb_batch_create: arena must be 256-byte aligned");
  int sm = 0;
  int rc = check_device(&sm);
  if (rc) return rc;
  int64_t ns = 0, nchp = 0;
  if ((rc = batch_check(chs, n, &ns, &nchp))) return rc;
  pb_batch_opts o{};
  if (opts) o = *opts;
  if (o.item_channels < 0 || (o.item_channels && (o.item_channels % 64 || o.item_channels < kBatchMinItem)))
    return set_error(PB_EINVAL, "pb_batch_create: item_channels must be 0 or a multiple of 64 >= %d", kBatchMinItem);
  if (o.ctas_per_sm < 0 || o.ctas_per_sm > 4) return set_error(PB_EINVAL, "pb_batch_create: ctas_per_sm must be 0..4");
  if (o.precision < 0 || o.precision > 2) return set_error(PB_EINVAL, "pb_batch: precision must be 0, 1 or 2");
  if (o.layout < 0 || o.layout > (o.precision >= 1 ? 2 : 1))
    return set_error(PB_EINVAL, "pb_batch: layout must be 0 or 1 (precision 0), 0..2 (precision 1, 2)");
  if (o.layout == 2)
    for (int i = 0; i < n; ++i)
      if (!chs[i]->closed)
        return set_error(PB_EINVAL, "pb_batch: layout 2 (symmetric tiles) needs channel lists built with the "
                                    "closure check (list %d was not)", i);
  cudaStream_t st = (cudaStream_t)stream;
  pb_batch *b = new (std::nothrow) pb_batch();
  if (!b) return set_error(PB_ENOMEM, "pb_batch_create: out of host memory");
  int status = PB_OK;
  try {
    b->n = n;
    b->ns = ns;
    b->nchp = nchp;
    b->sm_count = sm;
    b->prec = o.precision;
    b->lenp = b->prec >= 1 ? batch_pair_lenp(chs, n) : batch_lenp(chs, n);
    b->nitems_cap = batch_items_count(b->lenp, kBatchMinItem);
    b->dense = batch_dense_for(chs, n, o);
    const BatchDenseCaps dc = b->dense ? batch_dense_caps(chs, n, o.item_channels) : BatchDenseCaps{};
    b->nitems_cap = std::max(b->nitems_cap, dc.items);
    b->slot_cap = dc.slots;
    b->value_cap = dc.values;
    b->map_size = dc.map;
    b->soff.assign(n + 1, 0);
    for (int i = 0; i < n; ++i) {
      b->soff[i + 1] = b->soff[i] + chs[i]->nstate;
      b->nch.push_back(chs[i]->nch);
      for (int64_t r = 0; r < chs[i]->nstate; ++r) b->row_inst.push_back(i);
    }
    if (b->prec >= 1) {
      int64_t nent = 0;
      for (int64_t l : b->lenp) nent += l;
      const BatchTiles T = batch_tiles_for(chs, n, b->prec, o.layout, b->lenp, sm);
      const BatchLayoutFF LF = batch_layout_ff(chs, n, ns, nent, b->nitems_cap, b->prec == 2, T, b->lenp);
      if (bytes < LF.total) {
        delete b;
        return set_error(PB_ENOMEM, "pb_batch_create: arena of %zu bytes is smaller than the %zu needed", bytes,
                         LF.total);
      }
      char *A = (char *)arena;
      b->arena = A;
      b->bytes = bytes;
      b->items = (Item *)(A + LF.items);
      b->item_inst = (int32_t *)(A + LF.item_inst);
      b->item_ptr = (int32_t *)(A + LF.item_ptr);
      b->pA = (float2 *)(A + LF.pA);
      b->pB = (float2 *)(A + LF.pB);
      if (b->prec == 2) b->pC = (float2 *)(A + LF.pC);
      b->pidx = (uint32_t *)(A + LF.pidx);
      b->Rg = (double *)(A + LF.Rg);
      b->yff = (float2 *)(A + LF.yff);
      b->part = (Part4 *)(A + LF.part);
      b->acc = (double *)(A + LF.acc);
      b->y = (double *)(A + LF.y);
      b->err = (int *)(A + LF.err);
      if (T.on) {
        b->tiles = true;
        b->tnt = (int)T.tiles.size();
        b->tshape = b->prec == 2 ? 2 : 3;  // 2 stages x 3 CTAs per SM for both
        b->srp = (long long *)(A + LF.srp);
        b->tl = (dev::TileD *)(A + LF.tl);
        b->pmap = (int32_t *)(A + LF.pmap);
        b->prow = (int2 *)(A + LF.prow);
        b->tbase = (int2 *)(A + LF.tbase);
        b->tc = A + LF.tc;
        b->tp = A + LF.tp;
      }
      {
        // the error word; the padding of the stage input stays zero
        cudaError_t e = cudaMemsetAsync(b->err, 0, sizeof(int), st);
        if (e == cudaSuccess && T.on) e = cudaMemsetAsync(b->yff, 0, sizeof(float4) * (size_t)T.nsp, st);
        if (e != cudaSuccess) status = cuda_fail(e, "pb_batch_create: clear");
      }
      if (status == PB_OK) status = batch_setup_ff(b, chs, n, LF, st);
      if (status == PB_OK && b->tiles) status = batch_setup_tiles(b, T, st);
      if (status == PB_OK && !b->tiles && b->prec == 2 && nent > 0) {
        dev::k_pairs_c32<<<(int)std::min<int64_t>((nent + 255) / 256, 8192), 256, 0, st>>>(b->pA, b->pB,
                                                                                           (long long)nent, b->pC);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) status = cuda_fail(e, "k_pairs_c32 (batch)");
      }
      if (status == PB_OK) {
        b->ctas = o.ctas_per_sm ? o.ctas_per_sm : 4;  // of 256 threads
        status = batch_upload_plan(b, o.item_channels ? o.item_channels : 2048, st);
      }
      if (status != PB_OK) {
        delete b;
        return status;
      }
      *out = b;
      return PB_OK;
    }
    const BatchLayout L = batch_layout(chs, n, ns, nchp, b->nitems_cap, dc, sm);
    if (bytes < L.total) {
      delete b;
      return set_error(PB_ENOMEM, "pb_batch_create: arena of %zu bytes is smaller than the %zu needed", bytes, L.total);
    }
    char *A = (char *)arena;
    b->arena = A;
    b->bytes = bytes;
    b->items = (Item *)(A + L.items);
    b->item_inst = (int32_t *)(A + L.item_inst);
    b->item_ptr = (int32_t *)(A + L.item_ptr);
    b->col = (uint32_t *)(A + L.col);
    b->g2 = (float *)(A + L.g2);
    b->gstate = (uint4 *)(A + L.gstate);
    b->tabs = (float2 *)(A + L.tabs);
    b->inst = (pb::dev::BInst *)(A + L.inst);
    b->cs = (double *)(A + L.cs);
    b->part = (Part4 *)(A + L.part);
    b->acc = (double *)(A + L.acc);
    b->y = (double *)(A + L.y);
    if (b->dense) {
      b->g2d = (float *)(A + L.g2d);
      b->pidx0 = (uint32_t *)(A + L.pidx);
      b->smap = (uint32_t *)(A + L.smap);
      b->cbeg = (int32_t *)(A + L.cbeg);
      for (int i = 0; i < n; ++i) {
        b->heps.insert(b->heps.end(), chs[i]->eps.begin(), chs[i]->eps.begin() + chs[i]->nstate);
        b->reach.push_back(energy_reach_f32(chs[i]));
      }
    }
    double *om = (double *)(A + L.omega_tmp);
    double2 *tt = (double2 *)(A + L.tab_tmp);
    double *ep = (double *)(A + L.eps_tmp);
    short4 *kc = (short4 *)(A + L.kc_tmp);

    // per-instance tables, records and prefactors; channel words and FP32 |g|^2
    std::vector<pb::dev::BInst> hin(n);
    std::vector<double> hcs((size_t)ns);
    std::vector<uint32_t> hcol((size_t)nchp);
    std::vector<float> hg2((size_t)nchp, 0.f);
    size_t tab_off = 0;  // in float2
    int64_t coff = 0;
    for (int i = 0; i < n && status == PB_OK; ++i) {
      const pb_channels *ch = chs[i];
      int rad[3];
      size_t r = 1;
      for (int a = 0; a < 3; ++a) {
        rad[a] = ch->nk[a] > 1 ? 2 * ch->nk[a] : 1;
        r *= (size_t)rad[a];
      }
      const int64_t nt = (int64_t)r * ch->nmodes;
      if ((double)nt >= (double)(1 << dev::kRecLnmBits))
        status = set_error(PB_EINVAL, "pb_batch_create: instance %d needs (2 N1)(2 N2)(2 N3) nmodes < 2^27", i);
      if (ch->nk[0] > 32767 || ch->nk[1] > 32767 || ch->nk[2] > 32767)
        status = set_error(PB_EINVAL, "pb_batch_create: instance %d grid dimension above 32767", i);
      if (status) break;
      const double c = 2.0 * kPi / (kHbar * (double)ch->nq);
      const double norm = 1.0 / (std::sqrt(2.0 * kPi) * ch->sigma);
      const int n1 = rad[0] > 1 ? ch->nk[0] : 0, n2 = rad[1] > 1 ? ch->nk[1] : 0, n3 = rad[2] > 1 ? ch->nk[2] : 0;
      hin[i].tab = b->tabs + tab_off;
      hin[i].cpad = ((n1 * rad[1] + n2) * rad[2] + n3) * ch->nmodes;
      hin[i].k2 = (float)(-1.4426950408889634 / (2.0 * ch->sigma * ch->sigma));
      hin[i].soff = (int)b->soff[i];
      hin[i].ns = (int)ch->nstate;
      hin[i].nm = ch->nmodes;
      for (int64_t s = 0; s < ch->nstate; ++s) hcs[b->soff[i] + s] = c * norm;
      // the instance's rows in parallel from their first padded channel (hg2 is zero-filled)
      std::vector<int64_t> rs((size_t)ch->nstate + 1, coff);
      for (int64_t s = 0; s < ch->nstate; ++s) rs[s + 1] = rs[s] + b->lenp[b->soff[i] + s];
#pragma omp parallel for schedule(dynamic, 16)
      for (int64_t s = 0; s < ch->nstate; ++s) {
        const int64_t a = ch->row_ptr[s], len = ch->row_ptr[s + 1] - a, c0 = rs[s], lp = rs[s + 1] - c0;
        for (int64_t k = 0; k < len; ++k) {
          hcol[c0 + k] = (uint32_t)ch->col[a + k] | ((uint32_t)ch->nu[a + k] << kPartnerBits);
          hg2[c0 + k] = (float)ch->g2[a + k];
        }
        for (int64_t k = len; k < lp; ++k) hcol[c0 + k] = (uint32_t)s;
      }
      coff = rs[ch->nstate];
      // device: (w, N) table, padded FP32 table, state records
      std::vector<short4> hkc((size_t)ch->nstate);
      const int N2 = ch->nk[1], N3 = ch->nk[2];
      for (int64_t s = 0; s < ch->nstate; ++s) {
        const int ik = ch->kidx[s];
        hkc[s] = make_short4((short)(ik / (N2 * N3)), (short)((ik / N3) % N2), (short)(ik % N3), 0);
      }
      const size_t nq = (size_t)ch->nq * ch->nmodes;
      cudaError_t e = cudaMemcpyAsync(om, ch->omega.data(), sizeof(double) * nq, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(ep, ch->eps.data(), sizeof(double) * ch->nstate, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(kc, hkc.data(), sizeof(short4) * ch->nstate, cudaMemcpyHostToDevice, st);
      if (e != cudaSuccess) {
        status = cuda_fail(e, "pb_batch_create: upload");
        break;
      }
      dev::k_table<<<(int)std::min<size_t>((nq + 255) / 256, 4096), 256, 0, st>>>(om, (long long)nq, kBoltz * ch->T, tt);
      dev::k_tab_padded<<<(int)std::min<int64_t>((nt + 255) / 256, 8192), 256, 0, st>>>(
          tt, ch->nk[0], ch->nk[1], ch->nk[2], rad[0], rad[1], rad[2], ch->nmodes, b->tabs + tab_off);
      dev::k_gstate_init<<<(int)((ch->nstate + 255) / 256), 256, 0, st>>>(ep, kc, (int)ch->nstate, rad[1], rad[2],
                                                                         ch->nmodes, b->gstate + b->soff[i]);
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // temporaries are reused by the next instance
      if (e != cudaSuccess) {
        status = cuda_fail(e, "pb_batch_create: instance setup");
        break;
      }
      tab_off += align_up(sizeof(float2) * (size_t)nt) / sizeof(float2);
    }
    if (status == PB_OK) {
      cudaError_t e = cudaMemcpyAsync(b->inst, hin.data(), sizeof(pb::dev::BInst) * n, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(b->cs, hcs.data(), sizeof(double) * ns, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(b->col, hcol.data(), sizeof(uint32_t) * nchp, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaMemcpyAsync(b->g2, hg2.data(), sizeof(float) * nchp, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) status = cuda_fail(e, "pb_batch_create: upload");
    }
    b->hinst = hin;
    if (status == PB_OK) {
      b->ctas = o.ctas_per_sm ? o.ctas_per_sm : 2;
      status = batch_upload_plan(b, o.item_channels ? o.item_channels : 2048, st);
    }
  } catch (const std::bad_alloc &) {
    status = set_error(PB_ENOMEM, "pb_batch_create: out of host memory");
  }
  if (status != PB_OK) {
    delete b;
    return status;
  }
  *out = b;
  return PB_OK;
}

extern "C" void pb_batch_destroy(pb_batch *b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->cap) cudaStreamDestroy(b->cap);
  delete b;
}

extern "C" int pb_batch_get_info(const pb_batch *b, int64_t *nstate, int64_t *nchannels, int64_t *state_offsets,
                                 int32_t *item_channels, int32_t *ctas_per_sm) {
  clear_error();
  if (!b) return set_error(PB_EINVAL, "pb_batch_get_info: null handle");
  if (nstate) *nstate = b->ns;
  if (nchannels) {
    int64_t s = 0;
    for (int64_t c : b->nch) s += c;
    *nchannels = s;
  }
  if (state_offsets) std::memcpy(state_offsets, b->soff.data(), sizeof(int64_t) * (b->n + 1));
  if (item_channels) *item_channels = b->tiles ? 0 : b->item_ch;
  if (ctas_per_sm) *ctas_per_sm = b->tiles ? batch_tile_cps(b) : b->ctas;
  return PB_OK;
}

extern "C" int pb_batch_check(pb_batch *b, void *stream) {
  clear_error();
  if (!b) return set_error(PB_EINVAL, "pb_batch_check: null argument");
  if (!b->err) return PB_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int h = 0;
  PB_CUDA(cudaMemcpyAsync(&h, b->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  PB_CUDA(cudaStreamSynchronize(st));
  if (h) {
    PB_CUDA(cudaMemsetAsync(b->err, 0, sizeof(int), st));  // reported once
    PB_CUDA(cudaStreamSynchronize(st));
    return set_error(PB_ETIMEOUT, "a bounded device-side wait gave up (error word %d)", h);
  }
  return PB_OK;
}

extern "C" int pb_batch_collision(pb_batch *b, const double *f, double *dfdt, void *stream) {
  clear_error();
  if (!b || !f || !dfdt) return set_error(PB_EINVAL, "pb_batch_collision: null argument");
  cudaStream_t st = (cudaStream_t)stream;
  int rc;
  if ((rc = batch_stage_input(b, f, st)) || (rc = batch_sweep(b, st))) return rc;
  return batch_fin<-1>(b, dfdt, nullptr, 0.0, st, f);
}

extern "C" int pb_batch_rk4_step(pb_batch *b, double *f, double dt, int32_t nsteps, void *stream) {
  clear_error();
  if (!b || !f) return set_error(PB_EINVAL, "pb_batch_rk4_step: null argument");
  if (nsteps < 0 || !std::isfinite(dt)) return set_error(PB_EINVAL, "pb_batch_rk4_step: bad dt or nsteps");
  if (nsteps == 0) return PB_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (!(b->exec && b->rk_f == f && b->rk_dt == dt)) {
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    if (!b->cap) PB_CUDA(cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
    PB_CUDA(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
    int rc = batch_rk4_launches(b, f, dt, b->cap);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(b->cap, &graph);
    if (rc) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&b->exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      b->exec = nullptr;
      return cuda_fail(e, "cudaGraphInstantiate");
    }
    b->rk_f = f;
    b->rk_dt = dt;
  }
  int rc = batch_stage_input(b, f, st);
  if (rc) return rc;
  for (int32_t i = 0; i < nsteps; ++i) PB_CUDA(cudaGraphLaunch(b->exec, st));
  return PB_OK;
}

extern "C" int pb_batch_autotune(pb_batch *b, const double *f, void *stream, int32_t *best_item, int32_t *best_ctas,
                                 double *best_ms) {
  clear_error();
  if (!b || !f) return set_error(PB_EINVAL, "pb_batch_autotune: null argument");
  cudaStream_t st = (cudaStream_t)stream;
  if (b->tiles) {
    // the tile form: the launch shapes of the tile ring (stages x CTAs per SM).  A small float-float list
    // takes no ring but one CTA per half-tile, three per SM whatever the shape.
    static constexpr int kC32Shapes[] = {2, 3, 4, 7, 8}, kFFShapes[] = {3, 2};
    const int *shapes = b->prec == 2 ? kC32Shapes : kFFShapes;
    const int nshapes = b->prec == 2 ? 5 : chain_pdl(b->tnt, b->sm_count) ? 1 : 2;
    int bs = b->tshape;
    float best = 1e30f;
    cudaEvent_t e0, e1;
    PB_CUDA(cudaEventCreate(&e0));
    PB_CUDA(cudaEventCreate(&e1));
    int rc = batch_stage_input(b, f, st);
    for (int a = 0; a < nshapes && rc == PB_OK; ++a) {
      b->tshape = shapes[a];
      if ((rc = batch_sweep(b, st))) break;  // warm-up
      cudaEventRecord(e0, st);
      for (int k = 0; k < 3 && rc == PB_OK; ++k) rc = batch_sweep(b, st);
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) {
        best = ms;
        bs = shapes[a];
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->tshape = bs;
    if (b->exec) {  // the captured step holds the previous shape
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    if (rc) return rc;
    if (best_item) *best_item = 0;
    if (best_ctas) *best_ctas = batch_tile_cps(b);
    if (best_ms) *best_ms = best / 3.0;
    return PB_OK;
  }
  const int items[3] = {1024, 2048, 4096};
  const int ctas[3] = {2, 3, 4};
  int bi = b->item_ch, bc = b->ctas;
  float best = 1e30f;
  cudaEvent_t e0, e1;
  PB_CUDA(cudaEventCreate(&e0));
  PB_CUDA(cudaEventCreate(&e1));
  int rc = batch_stage_input(b, f, st);
  for (int a = 0; a < 3 && rc == PB_OK; ++a) {
    if ((rc = batch_upload_plan(b, items[a], st))) break;
    for (int c = 0; c < 3 && rc == PB_OK; ++c) {
      b->ctas = ctas[c];
      if ((rc = batch_sweep(b, st))) break;  // warm-up
      cudaEventRecord(e0, st);
      for (int k = 0; k < 3 && rc == PB_OK; ++k) rc = batch_sweep(b, st);
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) {
        best = ms;
        bi = items[a];
        bc = ctas[c];
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  b->ctas = bc;
  if ((rc = batch_upload_plan(b, bi, st))) return rc;
  if (best_item) *best_item = bi;
  if (best_ctas) *best_ctas = bc;
  if (best_ms) *best_ms = best / 3.0;
  return PB_OK;
}
