"""What sizing a device or a batch costs and reserves (host only, no GPU)."""
import ctypes
import time

import synth
import paper_2511_03683_gb300 as pb


def arena(lists, prec, layout=0, item=0):
    arr = (ctypes.c_void_p * len(lists))(*[c._h.value for c in lists])
    o, n = pb._BatchOpts(item, 0, prec, layout), ctypes.c_size_t(0)
    t = time.perf_counter()
    rc = pb.lib().pb_batch_arena_bytes(arr, len(lists), ctypes.byref(o), ctypes.byref(n))
    t = time.perf_counter() - t
    assert rc == pb.PB_OK, pb.lib().pb_last_error().decode()
    return n.value, t


def test_sizing_a_tiled_batch_does_not_walk_every_coupling():
    """The tile plan needs each list's largest |g|^2, which is kept with the list: sizing (and
    creating) a tiled batch costs about what the row form does (1.2 times here; one serial pass over
    the 1.4e7 couplings made it 15 times)."""
    lists = [pb.Channels.from_model(synth.make_window4(n)) for n in (24, 25)]
    rows = min(arena(lists, 1, layout=1)[1] for _ in range(7))
    for prec in (1, 2):
        assert min(arena(lists, prec)[1] for _ in range(7)) <= 4 * rows


def dev_arena(ch, **kw):
    o, n = pb._DevOpts(), ctypes.c_size_t(0)
    for k, v in kw.items():
        setattr(o, k, v)
    assert pb.lib().pb_dev_arena_bytes(ch._h, ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
    return n.value


def test_lists_that_take_the_tiles_for_their_reach_reserve_the_stored_tiles():
    """A cutoff list whose whole upper triangle would not pay (28^3: 325 tiles, 21 MB) but whose
    hundred tiles in reach do reserves those and not the triangle, alone and in a batch; forced tiles
    reserve the triangle, a size that follows from the number of states."""
    ch = pb.Channels.from_model(synth.make_window4(28), g2_min=1e-5, delta_nsigma=6.0)
    nb = (ch.nstate + 63) // 64
    triangle = 16 * 4096 * nb * (nb + 1) // 2
    assert 0 < dev_arena(ch) - dev_arena(ch, dense_rows=2) < triangle // 2
    assert dev_arena(ch, dense_rows=3) - dev_arena(ch, dense_rows=2) >= triangle
    assert 0 < arena([ch, ch], 1)[0] - arena([ch, ch], 1, layout=1)[0] < triangle
    assert arena([ch, ch], 1, layout=2)[0] - arena([ch, ch], 1, layout=1)[0] >= 2 * triangle


def test_dense_batch_reserves_no_more_slots_than_pairs():
    """The default FP32 batch: per (state, partner) slot 8 bytes of list and 4 of dense |g|^2 per branch,
    4 of partner and 4 of slot map, each grid's padded phonon table and a few hundred bytes per state; its
    chains never need more slots than there are partners (rounded up to 32 in each piece of a row)."""
    ns = (16, 18, 20, 22)
    lists = [pb.Channels.from_model(synth.make_window4(n)) for n in ns]
    slots = sum(c.nstate * ((c.nstate + 31) // 32 * 32) for c in lists)
    tables = sum((2 * n) ** 3 * 6 * 8 for n in ns)
    assert arena(lists, 0)[0] <= slots * (12 * 6 + 8) + tables + 400 * sum(c.nstate for c in lists) + (1 << 20)
