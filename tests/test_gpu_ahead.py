"""The draw-ahead form of a sweep call (csrc/ahead.cu), which a handle without a set
launch configuration takes for calls that are long enough: lattice and every sample
equal the oracle's bit for bit, at the edges of its plans (one warp, one CTA, tiles
with halos; 2, 4 and 8 rows a thread; words per row that divide nothing), over block
remainders and sample spacings; and the paths around it."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TC = 2.269185


@pytest.fixture(scope="module")
def P():
    import paper_1007_3726_gb300 as P

    P.build()
    P.load()
    return P


def _compare(orc, lat, s, t, n, rec, seed, sid, thr):
    got = lat.sweep(n, rec, collect=bool(rec))
    Mo, Eo = orc.run(s, n, seed, sid, *thr, t0=t)
    if rec:
        k0 = (rec - 1 - t) % rec
        assert np.array_equal(got[0], Mo[k0::rec]) and np.array_equal(got[1], Eo[k0::rec]), (n, rec)
    d = lat.measure()
    assert (d["M"], d["E"]) == (Mo[-1], Eo[-1]), (n, rec)
    assert np.array_equal(lat.spins(), s), (n, rec)


# calls: lengths around the plans' blocks (256, 32, 16, 8 and 4 sweeps) with every
# remainder of 4, sample spacings that cross the calls, none
SMALL = ((200, 1), (203, 3), (321, 0), (514, 7))
MIDDLE = ((10, 1), (33, 3), (64, 0), (71, 7))
LARGE = ((5, 1), (12, 3), (18, 0), (23, 1))


@pytest.mark.parametrize("L,calls", [(64, SMALL), (128, SMALL), (192, SMALL + MIDDLE), (256, MIDDLE), (320, MIDDLE),
                                     (448, MIDDLE), (512, MIDDLE), (704, MIDDLE), (960, MIDDLE), (1024, MIDDLE),
                                     (1088, MIDDLE), (2048, LARGE), (2112, LARGE), (4096, LARGE), (4160, LARGE),
                                     (8192, ((5, 1), (8, 2)))])
def test_sizes_blocks_and_records_bit_exact(P, orc, L, calls):
    T, seed, sid = TC, L + 3, 5
    lat = P.Lattice(L, T, seed=seed, stream_id=sid, init="hot", word_bits=64 if L % 128 == 0 else 32)
    s, t, thr = orc.init_hot(L, seed, sid), 0, orc.thresholds(T)
    for n, rec in calls:
        _compare(orc, lat, s, t, n, rec, seed, sid, thr)
        t += n
    lat.close()


@pytest.mark.parametrize("T", [0.05, 0.8, 3.5, 1e12])
def test_temperatures_and_changes_between_calls(P, orc, T):
    """Thresholds from 0 to 2^32 - 1; a short call, a call in a field and a set
    configuration between long ones keep one trajectory."""
    L, seed = 384, 11
    lat = P.Lattice(L, T, seed=seed, init="hot")
    s = orc.init_hot(L, seed, 0)
    _compare(orc, lat, s, 0, 21, 2, seed, 0, orc.thresholds(T))
    _compare(orc, lat, s, 21, 1, 1, seed, 0, orc.thresholds(T))
    lat.set_field(0.3)
    M, E = lat.sweep(4, 1, collect=True)
    Mo, Eo = orc.run_field(s, 4, seed, 0, T, 0.3, t0=22)
    assert np.array_equal(M, Mo) and np.array_equal(E, Eo)
    lat.set_field(0.0)
    lat.set_temperature(2.0)
    _compare(orc, lat, s, 26, 18, 1, seed, 0, orc.thresholds(2.0))
    lat.set_launch(proc_bits=32, regcap=0, insert=0, block=128, rows_per_item=4, grid=0)
    _compare(orc, lat, s, 44, 6, 1, seed, 0, orc.thresholds(2.0))
    lat.close()


# neighbour sums strictly inside, on and outside the field's zeros: 0 to 5 thresholds a sign
@pytest.mark.parametrize("H", [0.1, -0.1, 2.0, -2.0, 3.0, -3.5, 4.0, -4.0, 7.25, 1e-300, -1e3])
@pytest.mark.parametrize("L", [64, 320])
def test_field_classes_bit_exact(P, orc, L, H):
    T, seed, sid = 2.1, 9, 3
    lat = P.Lattice(L, T, seed=seed, stream_id=sid, init="hot", H=H)
    s, t = orc.init_hot(L, seed, sid), 0
    for n, rec in ((205, 1), (34, 3)) if L == 64 else ((34, 1), (37, 3)):
        M, E = lat.sweep(n, rec, collect=True)
        Mo, Eo = orc.run_field(s, n, seed, sid, T, H, t0=t)
        k0 = (rec - 1 - t) % rec
        assert np.array_equal(M, Mo[k0::rec]) and np.array_equal(E, Eo[k0::rec]), (n, rec)
        assert np.array_equal(lat.spins(), s)
        t += n
    lat.close()


@pytest.mark.parametrize("L", [64, 128, 192, 256, 448, 704, 1024, 1088, 2048, 2112, 4096, 4160])
def test_field_sizes_bit_exact(P, orc, L):
    T, H, seed = TC, -0.4, L
    lat = P.Lattice(L, T, seed=seed, init="hot")
    s, t = orc.init_hot(L, seed, 0), 0
    n = 210 if L <= 128 else 12
    _compare(orc, lat, s, 0, n, 2, seed, 0, orc.thresholds(T))  # scratch of the smaller form first
    lat.set_field(H)
    M, E = lat.sweep(n + 5, 3, collect=True)
    Mo, Eo = orc.run_field(s, n + 5, seed, 0, T, H, t0=n)
    k0 = (2 - n) % 3
    assert np.array_equal(M, Mo[k0::3]) and np.array_equal(E, Eo[k0::3])
    assert np.array_equal(lat.spins(), s)
    lat.close()


def test_late_sweep_indices_and_high_stream(P, orc):
    """Sweep indices next to 2^32 and the largest stream id in the Philox counter."""
    L, seed, sid, t = 128, 2 ** 63 + 5, 2 ** 31 - 1, 2 ** 32 - 300
    lat = P.Lattice(L, TC, seed=seed, stream_id=sid, init="hot", first_sweep=t)
    s = orc.init_hot(L, seed, sid)
    _compare(orc, lat, s, t, 260, 9, seed, sid, orc.thresholds(TC))
    lat.close()


@pytest.mark.parametrize("hold", [6, 390, 400])
def test_masks_that_never_arrive_are_reported(P, monkeypatch, hold):
    """L = 64 waits for masks on their way: a step whose masks never arrive ends the
    wait, the call reports ISING_ERR_TIMEOUT and the GPU stays usable."""
    lat = P.Lattice(64, 2.0, seed=1, init="hot")
    monkeypatch.setenv("ISING_TINY_HOLD_STEP", str(hold))
    with pytest.raises(P.IsingError) as ei:
        lat.sweep(200, 1, collect=True)
    assert ei.value.status == P.ERR_TIMEOUT
    monkeypatch.delenv("ISING_TINY_HOLD_STEP")
    with pytest.raises(P.IsingError) as ei:
        lat.sweep(1, 1)
    assert ei.value.status == P.ERR_STATE
    lat.close()
    ok = P.Lattice(64, 2.0, seed=1, init="hot")
    ok.sweep(200, 1)
    assert ok.measure()["sweeps_done"] == 200
    ok.close()


@pytest.mark.parametrize("L", [64, 512])
def test_without_scratch_memory_the_call_still_runs(P, orc, L):
    import torch

    taken = {}
    refuse = []

    def alloc(n, s):
        if refuse and n > 2 * L * L:  # the scratch, not the staging of a read-back
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        taken[p] = n
        return p

    def release(p, s):
        taken.pop(p)
        torch.cuda.caching_allocator_delete(p)

    P.ising_set_allocator(alloc, release)
    try:
        lat = P.Lattice(L, TC, seed=4, init="hot")
        s, thr = orc.init_hot(L, 4, 0), orc.thresholds(TC)
        held = len(taken)
        refuse.append(1)
        _compare(orc, lat, s, 0, 210, 4, 4, 0, thr)
        assert len(taken) == held
        refuse.clear()
        _compare(orc, lat, s, 210, 210, 4, 4, 0, thr)
        assert len(taken) == held + 1  # one allocation, kept by the handle
        lat.close()
        assert not taken
    finally:
        P.ising_set_allocator(None)


def test_handles_on_streams_and_threads(P, orc):
    """Handles of several sizes, each on its own stream and thread, at the same time."""
    import torch

    sizes = (64, 256, 512, 1024)
    out = {}

    def work(L):
        st = torch.cuda.Stream()
        lat = P.Lattice(L, TC, seed=L, init="hot", stream=st)
        r = [lat.sweep(220, 5, collect=True) for _ in range(3)]
        out[L] = (np.concatenate([m for m, _ in r]), np.concatenate([e for _, e in r]), lat.spins())
        lat.close()

    th = [threading.Thread(target=work, args=(L,)) for L in sizes]
    for x in th:
        x.start()
    for x in th:
        x.join()
    for L in sizes:
        s = orc.init_hot(L, L, 0)
        Mo, Eo = orc.run(s, 660, L, 0, *orc.thresholds(TC))
        M, E, spins = out[L]
        assert np.array_equal(M, Mo[4::5]) and np.array_equal(E, Eo[4::5]) and np.array_equal(spins, s), L
