"""Runtime pieces around the sweep: checkpoint / resume, the allocator hook
(PyTorch's caching allocator, and an injected allocation failure), handle
errors."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1007_3726_gb300 as P

    P.build()
    P.load()
    return P


@pytest.mark.parametrize("word_bits", [32, 64])
def test_checkpoint_resume_is_bit_exact(P, tmp_path, word_bits):
    L, T = 512, 2.269185
    ref = P.Lattice(L, T, seed=21, stream_id=4, init="hot", word_bits=word_bits)
    Ma, Ea = ref.sweep(10, 2, collect=True)
    path = str(tmp_path / "ckpt.npz")
    ref.save(path)
    Mb, Eb = ref.sweep(15, 2, collect=True)
    res = P.Lattice.load(path)
    assert res.sweeps_done == 10
    M0, E0 = res.restored_samples
    assert np.array_equal(M0, Ma) and np.array_equal(E0, Ea)
    Mc, Ec = res.sweep(15, 2, collect=True)
    assert np.array_equal(Mb, Mc) and np.array_equal(Eb, Ec)
    assert np.array_equal(ref.spins(), res.spins())
    assert res.measure()["sweeps_done"] == 25


def test_torch_caching_allocator_hook(P):
    import torch

    P.use_torch_allocator()
    try:
        a = P.Lattice(256, 2.0, seed=3, init="hot")
        Ma, Ea = a.sweep(12, 1, collect=True)
        sa = a.spins()
        a.close()
    finally:
        P.ising_set_allocator(None)
    b = P.Lattice(256, 2.0, seed=3, init="hot")
    Mb, Eb = b.sweep(12, 1, collect=True)
    assert np.array_equal(Ma, Mb) and np.array_equal(Ea, Eb) and np.array_equal(sa, b.spins())
    torch.cuda.synchronize()


def test_injected_allocation_failure(P):
    """An allocator that fails: creation reports ISING_ERR_OOM, frees what it took,
    and the library keeps working once a working allocator is back."""
    import torch

    taken = {}

    def alloc(n, s):
        if n > 4096:  # the lattice and staging buffers fail, small ones succeed
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        taken[p] = n
        return p

    def release(p, s):
        taken.pop(p, None)
        torch.cuda.caching_allocator_delete(p)

    P.ising_set_allocator(alloc, release)
    try:
        with pytest.raises(P.IsingError) as ei:
            P.Lattice(1024, 2.0, seed=1)
        assert ei.value.status == P.ERR_OOM
        assert not taken  # nothing left allocated
    finally:
        P.ising_set_allocator(None)
    ok = P.Lattice(1024, 2.0, seed=1)
    ok.sweep(2)
    assert ok.measure()["sweeps_done"] == 2


def test_invalid_first_sweep_and_counter_limit(P):
    with pytest.raises(P.IsingError):
        P.Lattice(256, 2.0, first_sweep=2 ** 32 - 1)
    lat = P.Lattice(256, 2.0, first_sweep=2 ** 32 - 3)
    lat.sweep(1)
    with pytest.raises(P.IsingError) as ei:
        lat.sweep(1)
    assert ei.value.status == P.ERR_INVALID


def test_scratch_of_many_handles_is_bounded_and_given_back(P, orc, monkeypatch):
    """Handles swept in turn keep scratch up to a bound together (here 100 MB; one of these
    takes 25 MB): all run the draw-ahead form, and lattices and samples are the oracle's
    although a handle's scratch was another's a call before.  Scratch also gives way to a
    lattice that would not fit beside it."""
    import torch

    monkeypatch.setenv("ISING_SCRATCH_MB", "100")
    taken, most, room = {}, [0], [1 << 40]

    def alloc(n, s):
        if sum(taken.values()) + n > room[0]:
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        taken[p] = n
        most[0] = max(most[0], sum(v for v in taken.values() if v > 20 << 20))
        return p

    def release(p, s):
        taken.pop(p)
        torch.cuda.caching_allocator_delete(p)

    L, n, k = 512, 200, 7
    for hook in (True, False):
        if hook:
            P.ising_set_allocator(alloc, release)
        try:
            streams = [torch.cuda.Stream() for _ in range(k)]
            lats = [P.Lattice(L, 2.2 + 0.02 * i, seed=i, init="hot", stream=streams[i]) for i in range(k)]
            for _ in range(2):
                for lat in lats:
                    lat.sweep(n, 4)  # queued only
                    assert lat.form == "ahead_cluster"
            for i, lat in enumerate(lats):
                s = orc.init_hot(L, i, 0)
                Mo, Eo = orc.run(s, 2 * n, i, 0, *orc.thresholds(2.2 + 0.02 * i))
                M, E = lat.samples()
                assert np.array_equal(M, Mo[3::4]) and np.array_equal(E, Eo[3::4]) and np.array_equal(lat.spins(), s)
            if hook:
                assert 20 << 20 < most[0] <= 100 << 20
                room[0] = sum(taken.values()) + (20 << 20)
                with P.Lattice(16384, 2.0, seed=1) as big:  # 32 MB
                    assert big.sweeps_done == 0
                room[0] = 1 << 40
            P.ising_release_scratch()
            assert not hook or not any(v > 20 << 20 for v in taken.values())
            lats[0].sweep(n, 4)
            assert lats[0].form == "ahead_cluster"
            for lat in lats:
                lat.close()
            assert not taken
        finally:
            if hook:
                P.ising_set_allocator(None)


def test_scratch_is_taken_from_handles_on_other_threads(P, orc, monkeypatch):
    """Threads with a handle each, on streams of their own, that take one another's idle
    scratch all the time (a bound of two)."""
    import threading

    import torch

    monkeypatch.setenv("ISING_SCRATCH_MB", "52")
    L, n, out = 512, 192, {}

    def work(i):
        st = torch.cuda.Stream()
        with P.Lattice(L, 2.25, seed=i, init="hot", stream=st) as lat:
            r = []
            for _ in range(6):
                r.append(lat.sweep(n, 3, collect=True))
            out[i] = (np.concatenate([m for m, _ in r]), np.concatenate([e for _, e in r]), lat.spins())

    th = [threading.Thread(target=work, args=(i,)) for i in range(5)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert len(out) == 5
    for i, (M, E, spins) in out.items():
        s = orc.init_hot(L, i, 0)
        Mo, Eo = orc.run(s, 6 * n, i, 0, *orc.thresholds(2.25))
        assert np.array_equal(M, Mo[2::3]) and np.array_equal(E, Eo[2::3]) and np.array_equal(spins, s)
