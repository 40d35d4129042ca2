"""Host side of the batched forms: what sizing a batch costs and reserves (no GPU)."""
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
