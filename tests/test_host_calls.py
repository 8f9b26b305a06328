"""The host side of the C entry points, on a stand-in for the CUDA runtime (fake_runtime)."""
import ctypes

import pytest

from paper_1201_2501_gb300 import sfft
from tests import fake_runtime as fr

STREAM = ctypes.c_void_p(0xABC000)


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fr.load(tmp_path_factory.mktemp("fake"))


def _outputs():
    return ctypes.c_void_p(0x1000), ctypes.c_void_p(0x2000), 64, ctypes.c_void_p(0x3000), ctypes.c_void_p(0x4000)


def _run_mixed(L):
    plans = [fr.plan(L, 1 << 14, 8), fr.plan(L, 1 << 16, 512)]  # one of each kind of decode
    assert [s for s, _ in plans] == [0, 0]
    handles = (ctypes.c_void_p * 2)(*[h for _, h in plans])
    bp = ctypes.c_void_p()
    assert L.sfft_batch_plan_create(handles, 2, 4, ctypes.byref(bp)) == 0
    table = (sfft.SfftRequest * 2)()
    for r in range(2):
        table[r].d_x = 0x10000
    call = lambda: L.sfft_batch_execute(bp, (ctypes.c_uint32 * 2)(0, 1), table, 2, STREAM, *_outputs())
    return call, lambda: (L.sfft_batch_plan_destroy(bp), [L.sfft_plan_destroy(h) for _, h in plans])


def _run_groups(L, mode):
    s, h = fr.plan(L, 1 << 14, 8, mode, batch=16, streams=4)
    assert s == 0
    call = lambda: L.sfft_execute(h, ctypes.c_void_p(0x10000), 16, ctypes.c_uint64(5), STREAM, *_outputs())
    return call, lambda: L.sfft_plan_destroy(h)


@pytest.mark.parametrize("what", ["mixed", "exact", "general"])
def test_a_launch_that_fails_leaves_nothing_running_unordered(L, what):
    """A call that spreads its work over streams and fails at any of its launches returns SFFT_ERR_CUDA, and
    the caller's stream still waits for every launch made before: the caller may free its arrays behind it."""
    call, close = _run_mixed(L) if what == "mixed" else _run_groups(L, {"exact": 0, "general": 1}[what])
    L.fake_reset()
    assert call() == 0
    st = hex(STREAM.value)
    total = sum(c[0] == "launch" for c in fr.log(L))
    assert total >= 2 and len({c[2] for c in fr.log(L) if c[0] == "launch"}) >= 2  # on several streams
    assert fr.unordered(fr.log(L), st) == []
    for good in range(total):
        L.fake_reset()
        L.fake_fail_launch(good)
        assert call() == sfft.SFFT_ERR_CUDA
        assert b"a call made to fail" in L.sfft_last_error()
        assert sum(c[0] == "launch" for c in fr.log(L)) == good
        assert fr.unordered(fr.log(L), st) == [], good
    L.fake_reset()
    close()


# per request of max_batch, the most device memory a general plan may take: what it took when the rounds
# gathered one after another (bytes: (log2 n, k, fields) -> one request)
GENERAL_BYTES = [(16, 16, dict(alpha0=0.25), 967_600), (15, 16, dict(bins_per_k=4.0), 529_600), (16, 64, {}, 2_520_700)]


@pytest.mark.parametrize("m,k,fields,per", GENERAL_BYTES)
def test_a_general_plan_takes_the_memory_of_one_round_where_it_has_to(L, m, k, fields, per):
    """A plan for as many requests as fit when rounds take turns in the memory of one is built, by the size of
    the plan alone or because other users hold the rest of the device, and runs; a smaller plan keeps one
    gather for all rounds."""
    def gathers(h, batch):
        L.fake_reset()
        assert L.sfft_execute(h, ctypes.c_void_p(0x10000), batch, ctypes.c_uint64(5), STREAM, *_outputs()) == 0
        names = [c[1] for c in fr.log(L) if c[0] == "launch"]
        assert sum("k_gen_select" in n for n in names) == L.sfft_plan_rounds(h)
        return sum("k_gen_gather" in n for n in names)

    L.fake_reset()
    st, h = fr.plan(L, 1 << m, k, sfft.SFFT_GENERAL, batch=64, **fields)
    at_once, rounds = L.fake_bytes(), L.sfft_plan_rounds(h)
    assert st == 0 and gathers(h, 1) == 1 and rounds > 1
    L.sfft_plan_destroy(h)
    for batch, memory in (((1 << 38) // per, 1 << 38), (64, min(64 * per + (1 << 20), at_once - 1))):
        L.fake_reset()
        L.fake_memory(ctypes.c_size_t(memory))
        st, h = fr.plan(L, 1 << m, k, sfft.SFFT_GENERAL, batch=batch, **fields)
        assert st == 0, batch
        assert L.fake_bytes() <= batch * per + (1 << 20)  # (the tables are the plan's, not a request's)
        assert gathers(h, 1) == rounds
        L.sfft_plan_destroy(h)
    L.fake_reset()


def test_the_wait_check_reads_what_the_channel_slots_report(L):
    """sfft_persistent_wait_check answers SFFT_ERR_TIMEOUT only when the channel gather's wait gave up and the
    decode of every slot reported it: not when the wait ended, nor when the slots hold something else."""
    gave_up = fr.LAUNCH_FN(lambda kernel, args: ctypes.memset(ctypes.cast(args[1], ctypes.POINTER(ctypes.c_void_p))[0], 1, 4)
                           if b"wait_check" in kernel else None)
    L.fake_reset()
    assert L.sfft_persistent_wait_check(STREAM) == 0
    assert not any("k_chan_decode" in c[1] for c in fr.log(L))
    L.fake_reset()
    L.fake_on_launch(gave_up)
    assert L.sfft_persistent_wait_check(STREAM) == sfft.SFFT_ERR_CUDA
    assert b"slot" in L.sfft_last_error()
    assert any("k_chan_decode" in c[1] for c in fr.log(L))
    L.fake_reset()
