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
LONG = MIDDLE + ((130, 1), (203, 3), (514, 1), (193, 0))
LARGE = ((10, 1), (12, 3), (18, 0), (23, 1), (33, 5))


@pytest.mark.parametrize("L,calls", [(64, SMALL), (128, SMALL), (192, SMALL + MIDDLE), (256, MIDDLE), (320, LONG),
                                     (384, LONG), (448, LONG), (512, LONG), (704, MIDDLE), (960, MIDDLE), (1024, MIDDLE),
                                     (1088, MIDDLE), (2048, LARGE), (2112, LARGE), (4096, LARGE), (4160, LARGE),
                                     (8192, ((10, 1), (13, 2))), (8256, ((4, 1), (11, 2))), (9984, ((9, 1), (8, 0))),
                                     (16384, ((7, 3), (4, 1)))])
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


@pytest.mark.parametrize("L", [64, 128, 192, 256, 448, 704, 1024, 1088, 2048, 2112, 4096, 4160, 8256])
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


@pytest.mark.parametrize("L,hold", [(64, 6), (64, 390), (64, 400), (448, 6), (512, 390), (512, 400)])
def test_masks_that_never_arrive_are_reported(P, monkeypatch, L, hold):
    """L = 64 and the clusters (L = 320 .. 512) wait for masks on their way: a step whose
    masks never arrive ends the wait, the call reports ISING_ERR_TIMEOUT and the GPU stays
    usable."""
    lat = P.Lattice(L, 2.0, seed=1, init="hot")
    monkeypatch.setenv("ISING_TINY_HOLD_STEP", str(hold))
    with pytest.raises(P.IsingError) as ei:
        lat.sweep(200, 1, collect=True)
    assert ei.value.status == P.ERR_TIMEOUT
    monkeypatch.delenv("ISING_TINY_HOLD_STEP")
    with pytest.raises(P.IsingError) as ei:
        lat.sweep(1, 1)
    assert ei.value.status == P.ERR_STATE
    lat.close()
    ok = P.Lattice(L, 2.0, seed=1, init="hot")
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


# (L, H, sweeps): tiles of every kind, blocks of 4 .. 64 sweeps with remainders, odd and
# even numbers of blocks, lattices that end before the others
BATCHES = [
    [(64, 0.0, 61), (128, 0.0, 9), (192, 0.0, 40), (256, 0.0, 13), (64, 0.0, 8)],
    [(320, 0.0, 17), (448, 0.0, 24), (512, 0.0, 9), (704, 0.0, 12), (1088, 0.0, 10)],
    [(1024, 0.0, 21), (2048, 0.0, 9), (4096, 0.0, 8), (2112, 0.0, 11), (960, 0.0, 1)],
    [(64, 0.3, 30), (192, -2.0, 19), (256, 0.1, 22), (512, 0.0, 14), (320, 4.0, 9), (1024, -0.2, 8), (2048, 0.5, 9)],
    [(1024, 0.0, 37)],
]


@pytest.mark.parametrize("record_every", [0, 1, 3])
@pytest.mark.parametrize("k", range(len(BATCHES)))
def test_batch_equals_the_strips(P, k, record_every):
    """Runs of a batch without launch options against the same runs in strips."""
    make = lambda: [P.Lattice(L, 2.0 + 0.05 * i, seed=7 + i, stream_id=i, init="hot", H=H)  # noqa: E731
                    for i, (L, H, _) in enumerate(BATCHES[k])]
    a, b = make(), make()
    sweeps = [n for _, _, n in BATCHES[k]]
    with P.Batch(a, sweeps, record_every, use_graph=k == 0) as x, P.Batch(b, sweeps, record_every, block=512) as y:
        x.run(1)
        y.run(1)
        a[0].sweep(3, record_every)  # another form in between
        b[0].sweep(3, record_every)
        x.run(2)
        y.run(2)
    for l, r in zip(a, b):
        assert np.array_equal(l.spins(), r.spins()), l.L
        assert np.array_equal(np.stack(l.samples()), np.stack(r.samples())), l.L
        dl, dr = l.measure(), r.measure()
        assert (dl["M"], dl["E"], dl["sweeps_done"]) == (dr["M"], dr["E"], dr["sweeps_done"])


def test_batch_against_the_oracle(P, orc):
    specs = [(256, 0.0), (512, 0.2), (1024, 0.0)]
    lats = [P.Lattice(L, TC, seed=L, stream_id=2, init="hot", H=H) for L, H in specs]
    with P.Batch(lats, [14, 9, 12], 2) as b:
        b.run(1)
    for (L, H), n, lat in zip(specs, (14, 9, 12), lats):
        s = orc.init_hot(L, L, 2)
        Mo, Eo = orc.run_field(s, n, L, 2, TC, H) if H else orc.run(s, n, L, 2, *orc.thresholds(TC))
        M, E = lat.samples()
        assert np.array_equal(M, Mo[1::2]) and np.array_equal(E, Eo[1::2]) and np.array_equal(lat.spins(), s), L


def test_batch_without_scratch_memory_runs_in_strips(P):
    import torch

    taken, refused = {}, []

    def alloc(n, s):
        if n > 8 << 20:  # the masks of a block
            refused.append(n)
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        taken[p] = n
        return p

    def release(p, s):
        taken.pop(p)
        torch.cuda.caching_allocator_delete(p)

    P.ising_set_allocator(alloc, release)
    try:
        a = [P.Lattice(512, TC, seed=1, stream_id=i, init="hot") for i in range(4)]
        with P.Batch(a, [20] * 4, 2) as x:
            x.run(1)
        got = [(l.spins(), l.samples()) for l in a]
        for l in a:
            l.close()
        assert refused and not taken
    finally:
        P.ising_set_allocator(None)
    for i, (spins, samples) in enumerate(got):
        l = P.Lattice(512, TC, seed=1, stream_id=i, init="hot")
        M, E = l.sweep(20, 2, collect=True)
        assert np.array_equal(l.spins(), spins) and np.array_equal(samples[0], M) and np.array_equal(samples[1], E)


def test_second_counter_word_within_a_row(P):
    """Above 2^35 sites the Philox group index needs its second word, which changes
    inside a row of this size: the band form against the step kernels."""
    L = 185408
    out = []
    for legacy in (True, False):
        with P.Lattice(L, TC, seed=5, init="hot") as lat:
            if legacy:
                lat.set_launch(**lat.launch)
            out.append(lat.sweep(6, 1, collect=True))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("L", [320, 448, 512])
def test_cluster_counts_every_sweep_while_its_buffers_turn(P, orc, L):
    """Calls of many blocks with M/E after every sweep: both snapshot buffers and both
    mask buffers are used over and over, by launches that start beside the update before,
    and what an earlier call left in them is counted by none."""
    seed, calls = 5, (1030, 700)
    lat = P.Lattice(L, TC, seed=seed, init="cold_up")
    s, t = orc.init_cold(L, 1), 0
    for n in calls:
        _compare(orc, lat, s, t, n, 1, seed, 0, orc.thresholds(TC))
        t += n
    lat.close()
