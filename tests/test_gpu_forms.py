"""Which form a call takes, and the forms that the draw-ahead form has replaced as the
default: they remain what runs where it does not apply, and what a set configuration runs."""
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


# the edges of the plans' ranges: (L, H, sweeps) and the form
DEFAULTS = [
    (64, 0.0, 199, "one_launch"), (64, 0.0, 200, "ahead"), (128, 0.0, 99, "one_launch"), (128, 0.0, 100, "ahead"),
    (192, 0.0, 2, "steps"), (192, 0.0, 3, "ahead"), (256, 0.0, 9, "one_launch"), (256, 0.0, 10, "ahead"),
    (320, 0.0, 191, "ahead"), (320, 0.0, 192, "ahead_cluster"), (512, 0.0, 2, "one_launch"), (512, 0.0, 3, "ahead"),
    (512, 0.0, 192, "ahead_cluster"), (576, 0.0, 200, "ahead"), (1024, 0.0, 4, "steps"), (1024, 0.0, 5, "ahead"),
    (1472, 0.0, 5, "ahead"), (1536, 0.0, 5, "steps"), (1536, 0.0, 6, "ahead"), (1856, 0.0, 8, "steps"), (1856, 0.0, 9, "ahead"),
    (2048, 0.0, 9, "steps"), (2048, 0.0, 10, "ahead"), (8192, 0.0, 10, "ahead"), (8256, 0.0, 3, "steps"),
    (8256, 0.0, 4, "ahead_bands"), (185408, 0.0, 6, "ahead_bands"),
    (64, 0.3, 4, "one_launch"), (64, 0.3, 5, "ahead"), (320, 0.3, 1, "ahead"), (512, -2.0, 200, "ahead"),
    (2048, 0.3, 1, "ahead"), (4096, 0.3, 3, "steps"), (4096, 0.3, 4, "ahead"), (4160, 0.3, 3, "steps"), (4160, 0.3, 4, "ahead_bands"),
]


@pytest.mark.parametrize("L,H,n,form", DEFAULTS)
def test_form_of_a_default_call(P, L, H, n, form):
    with P.Lattice(L, TC, seed=1, init="hot", H=H) as lat:
        assert lat.form == "none"
        lat.sweep(n, 1)
        assert lat.form == form


def test_a_set_configuration_is_what_runs(P):
    with P.Lattice(512, TC, seed=1) as lat:
        for cfg, form in ((dict(lat.launch), "one_launch"),
                          (dict(proc_bits=32, regcap=0, insert=0, block=256, rows_per_item=4, grid=0), "steps"),
                          (dict(proc_bits=32, regcap=0, insert=0, block=256, rows_per_item=4, grid=0, persistent=1), "cooperative")):
            lat.set_launch(**cfg)
            lat.sweep(200, 1)
            assert lat.form == form


def test_the_way_back_to_the_default_form(P, orc):
    with P.Lattice(512, TC, seed=3, init="hot") as lat:
        default = lat.launch
        M, forms = [], []
        for change in (lambda: None, lambda: lat.set_launch(**default), lat.clear_launch,
                       lambda: lat.set_launch(proc_bits=32, regcap=0, insert=0, block=128, rows_per_item=4, grid=0), lat.clear_launch):
            change()
            M.append(lat.sweep(30, 1, collect=True)[0])
            forms.append(lat.form)
        assert forms == ["ahead", "one_launch", "ahead", "steps", "ahead"] and lat.launch == default
        s = orc.init_hot(512, 3, 0)
        Mo, _ = orc.run(s, 150, 3, 0, *orc.thresholds(TC))
        assert np.array_equal(np.concatenate(M), Mo) and np.array_equal(lat.spins(), s)


def test_form_of_a_batch(P):
    lats = [P.Lattice(L, TC, seed=L) for L in (64, 512)]
    for n, opts, form in ((20, {}, "ahead"), (20, dict(use_graph=True), "ahead"), (4, {}, "strips"), (20, dict(block=512), "strips"),
                          (20, dict(wait_ms=100.0), "strips")):
        with P.Batch(lats, [n, n], 1, **opts) as b:
            assert b.form == form
            b.run(1)


# one-launch forms on whole calls of the plain method's length, as they were the default
@pytest.mark.parametrize("L,n", [(64, 1000), (128, 400), (256, 200), (512, 60)])
def test_one_launch_forms_on_long_calls(P, orc, L, n):
    lat = P.Lattice(L, TC, seed=1, init="cold_up")
    lat.set_launch(**lat.launch)
    M, E = lat.sweep(n, 1, collect=True)
    assert lat.form == "one_launch"
    s = orc.init_cold(L, 1)
    Mo, Eo = orc.run(s, n, 1, 0, *orc.thresholds(TC))
    assert np.array_equal(M, Mo) and np.array_equal(E, Eo) and np.array_equal(lat.spins(), s)
    lat.close()


@pytest.mark.parametrize("L,H", [(64, 0.0), (128, 0.0), (256, 0.0), (512, 0.0), (64, 0.3), (256, -2.0)])
def test_one_launch_forms_in_several_launches(P, orc, monkeypatch, L, H):
    """Calls longer than a launch's bound: a launch hands its sample slots to the next."""
    T, seed, sid, t = 2.1, 23, 2, 0
    lat = P.Lattice(L, T, seed=seed, stream_id=sid, init="hot", H=H)
    lat.set_launch(**lat.launch)
    monkeypatch.setenv("ISING_TINY_MAX_SWEEPS", "7")
    s = orc.init_hot(L, seed, sid)
    for n, rec in ((50, 3), (15, 0), (22, 1)):
        got = lat.sweep(n, rec, collect=bool(rec))
        assert lat.form == "one_launch"
        Mo, Eo = orc.run_field(s, n, seed, sid, T, H, t0=t) if H else orc.run(s, n, seed, sid, *orc.thresholds(T), t0=t)
        if rec:
            k0 = (rec - 1 - t) % rec
            assert np.array_equal(got[0], Mo[k0::rec]) and np.array_equal(got[1], Eo[k0::rec]), (n, rec)
        d = lat.measure()
        assert (d["M"], d["E"]) == (Mo[-1], Eo[-1])
        t += n
    assert np.array_equal(lat.spins(), s)
    lat.close()


@pytest.mark.parametrize("L,H,n", [(4096, 0.0, 12), (4096, 0.25, 6), (32768, 0.0, 6)])
def test_step_kernels_on_larger_lattices(P, orc, L, H, n):
    """The whole lattice and every sample, in the step kernels' default configuration."""
    lat = P.Lattice(L, TC, seed=7, init="hot", H=H)
    lat.set_launch(**lat.launch)
    M, E = lat.sweep(n, 1, collect=True)
    assert lat.form == "steps"
    s = orc.init_hot(L, 7, 0)
    Mo, Eo = orc.run_field(s, n, 7, 0, TC, H) if H else orc.run(s, n, 7, 0, *orc.thresholds(TC), check=False)
    assert np.array_equal(M, Mo) and np.array_equal(E, Eo) and np.array_equal(lat.spins(), s)
    lat.close()


def test_step_kernels_on_L524288(P, orc):
    """Rows of four windows (both ends, the middle) after 5 sweeps, against the oracle's
    light-cone evolution, and the fused M/E against a recount."""
    import torch

    if torch.cuda.mem_get_info()[0] < 40 * 2 ** 30:
        pytest.skip("needs 40 GiB of free device memory")
    L, T, seed, k = 524288, 2.0, 5, 5
    lat = P.Lattice(L, T, seed=seed, init="cold_up", word_bits=64)
    lat.set_launch(**lat.launch)
    M, E = lat.sweep(k, 1, collect=True)
    assert lat.form == "steps"
    margin = 2 * k + 1
    for row0 in (0, L - 40, L // 2 + 17, 123456):
        w = np.ones((64 + 2 * margin, L), dtype=np.int8)
        orc.run_window(w, L, (row0 - margin) % L, k, seed, 0, *orc.thresholds(T))
        assert np.array_equal(lat.spins(row0, 64), w[margin:margin + 64]), row0
    assert (int(M[-1]), int(E[-1])) == lat.recount()
    lat.close()


def test_autotune_without_scratch_leaves_the_default_form(P):
    """Where the draw-ahead form's scratch is refused while a handle is tuned, the form is
    not timed and stays the default, for the handle and for later ones."""
    import torch

    L, refused = 832, []

    def alloc(n, s):
        if n > 1 << 20:  # the masks, not the lattice or its copy
            refused.append(n)
            return None
        return torch.cuda.caching_allocator_alloc(n)

    P.ising_set_allocator(alloc, lambda p, s: torch.cuda.caching_allocator_delete(p))
    try:
        with P.Lattice(L, TC, seed=1) as lat:
            lat.autotune(reps=1)
            assert refused
            lat.sweep(20, 1)
            assert lat.form != "ahead"  # refused here too
    finally:
        P.ising_set_allocator(None)
    with P.Lattice(L, TC, seed=1) as lat:
        lat.sweep(20, 1)
        assert lat.form == "ahead"


def test_autotune_returns_the_time_of_the_configuration_it_returns(P, monkeypatch, capfd):
    monkeypatch.setenv("ISING_AUTOTUNE_LOG", "1")
    with P.Lattice(448, TC, seed=1) as lat:
        cfg, us = lat.autotune(reps=2)
        log = [ln for ln in capfd.readouterr().err.splitlines() if ln.startswith("autotune L=448")]
        times = [float(ln.split(": ")[1].split()[0]) for ln in log if "draw-ahead" not in ln]
        assert len(times) == len(P.ising_launch_candidates(448)) and len(log) == len(times) + 1
        assert abs(us - min(times)) < 0.01
        # what was not timed stays: calls in a field, and long ones in a cluster
        lat.sweep(200, 1)
        assert lat.form == "ahead_cluster"
        lat.set_field(0.2)
        lat.sweep(20, 1)
        assert lat.form == "ahead"


@pytest.mark.parametrize("probe", [0, 4])
def test_batch_tune_weighs_the_default_form_too(P, probe):
    """Where the runs take the draw-ahead form without options, it is one of the
    candidates (and by far the fastest on 32 of 512^2); with an option that asks for the
    strips, or for runs too short for it, it is none."""
    lats = [P.Lattice(512, 2.0 + 0.02 * i, seed=i) for i in range(32)]
    before = [l.packed() for l in lats]
    opts, ms = P.ising_batch_tune(lats, [1000] * 32, probe)
    assert opts["block"] == opts["ctas_per_sm"] == opts["rows_per_item"] == 0 and ms > 0
    with P.Batch(lats, [20] * 32, 1, **opts) as b:
        assert b.form == "ahead"
    for kw, n in ((dict(wait_ms=500.0), 1000), ({}, 6)):
        opts, _ = P.ising_batch_tune(lats, [n] * 32, probe, **kw)
        assert opts["block"] in (128, 256, 512) and opts["wait_ms"] == kw.get("wait_ms", 0.0)
        with P.Batch(lats, [n] * 32, 1, **opts) as b:
            assert b.form == "strips"
    for l, p in zip(lats, before):
        assert np.array_equal(l.packed(), p) and l.sweeps_done == 0


def test_command_line_batch_runs_the_default_form(P, capsys):
    import json

    from paper_1007_3726_gb300 import __main__ as cli

    for argv, form in (([], "ahead"), (["--block", "256", "--ctas-per-sm", "4"], "strips")):
        assert cli.main(["fss-batch", "--sweeps", "20", *argv]) == 0
        assert json.loads(capsys.readouterr().out)["form"] == form


@pytest.mark.parametrize("L,n,what", [(64, 20, "one-launch"), (64, 200, "draw-ahead"), (512, 200, "draw-ahead")])
def test_a_wait_that_runs_out_names_the_form(P, monkeypatch, L, n, what):
    with P.Lattice(L, 2.0, seed=1) as lat:
        monkeypatch.setenv("ISING_TINY_HOLD_STEP", "6")
        with pytest.raises(P.IsingError) as ei:
            lat.sweep(n, 1, collect=True)
        assert ei.value.status == P.ERR_TIMEOUT and what in str(ei.value)


def test_small_lattices_in_blocks_of_a_thousand_sweeps(P, orc):
    """L = 64, calls of several blocks, whole and partial ones."""
    s, t, lat = orc.init_hot(64, 3, 0), 0, P.Lattice(64, TC, seed=3, init="hot")
    for n, rec in ((1030, 1), (2500, 7), (1024, 0), (203, 3), (2049, 1)):
        got = lat.sweep(n, rec, collect=bool(rec))
        assert lat.form == "ahead"
        Mo, Eo = orc.run(s, n, 3, 0, *orc.thresholds(TC), t0=t)
        if rec:
            k0 = (rec - 1 - t) % rec
            assert np.array_equal(got[0], Mo[k0::rec]) and np.array_equal(got[1], Eo[k0::rec]), n
        d = lat.measure()
        assert (d["M"], d["E"]) == (Mo[-1], Eo[-1]) and np.array_equal(lat.spins(), s)
        t += n
    lat.close()


def test_small_lattices_on_many_streams(P, orc):
    """L = 64: calls of handles on more than eight streams are one launch each, whatever was
    queued before; lattices and samples do not depend on it."""
    import torch

    streams = [torch.cuda.Stream() for _ in range(9)]
    lats = [P.Lattice(64, 2.2, seed=i, init="hot", stream=streams[i % 8]) for i in range(10)]

    def call(form):
        for lat in lats:
            lat.sweep(250, 5)
            assert lat.form == form

    call("ahead")
    lats.append(P.Lattice(64, 2.2, seed=10, init="hot", stream=streams[8]))
    call("one_launch")
    with P.Lattice(64, 2.2, seed=1, H=0.1) as f, P.Lattice(128, 2.2, seed=1) as g:
        f.sweep(200)
        g.sweep(200)
        assert f.form == g.form == "ahead"
    last = lats.pop()
    last.close()  # while its call may still run
    call("ahead")
    for i, lat in enumerate(lats):
        s = orc.init_hot(64, i, 0)
        Mo, Eo = orc.run(s, 750, i, 0, *orc.thresholds(2.2))
        M, E = lat.samples()
        assert np.array_equal(M, Mo[4::5]) and np.array_equal(E, Eo[4::5]) and np.array_equal(lat.spins(), s)
        lat.close()
