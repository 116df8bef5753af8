"""The calls a user of the framework makes, as cases whose time is measured.

Every case goes through the public entry points of ``paper_1007_3726_gb300``:
``Lattice`` (one simulated lattice), ``Batch`` (many lattices in one launch) and
``Server`` (a request stream).  The outputs are the recorded samples M, E and
the whole lattice afterwards; all of them are whole numbers.

Kinds of case:

* ``chain``   one ``Lattice.sweep`` call that records M and E, at the sizes and
              sample spacings of the workloads and tests: the small lattices of a
              finite-size-scaling run (64 .. 512), lattices that are not a power
              of two (320), the middle range (1024, 4096: the paper's Table 1
              shape) and a lattice far larger than L2; with ``H`` in a field.
* ``anneal``  one temperature of an annealing schedule: ``set_temperature`` and a
              few sweeps of a small lattice, the smallest call there is.
* ``buffer``  a configuration that the user holds on the host as int8 +1/-1: upload,
              a few sweeps, read back.
* ``batch``   lattices of several sizes and temperatures in one persistent launch.
* ``served``  a burst of requests to the server, submitted, awaited and read out.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1007_3726_gb300 as ising

TC = 2.269185
FSS_SIZES = (256, 512, 1024, 2048)


def listed():
    return [
        # one temperature of an annealing run on the smallest lattice: latency
        dict(name="anneal_L64", kind="anneal", L=64, sweeps=5),
        # the smallest workload of the repository: L = 64, M and E every sweep
        dict(name="chain_L64", kind="chain", L=64, T=TC, H=0.0, init="cold", sweeps=1000, record_every=1),
        # a lattice of a finite-size-scaling run
        dict(name="chain_L256", kind="chain", L=256, T=2.27, H=0.0, init="cold", sweeps=1000, record_every=10),
        # a size that is no power of two
        dict(name="chain_L320", kind="chain", L=320, T=2.3, H=0.0, init="hot", sweeps=500, record_every=1),
        # the larger lattice of the U4 crossing pair
        dict(name="chain_L512", kind="chain", L=512, T=2.25, H=0.0, init="cold", sweeps=1000, record_every=100),
        # the middle range, where one lattice does not fill the GPU
        dict(name="chain_L1024", kind="chain", L=1024, T=2.26, H=0.0, init="hot", sweeps=500, record_every=10),
        # a magnetisation curve in an external field
        dict(name="field_L2048", kind="chain", L=2048, T=TC, H=0.1, init="hot", sweeps=200, record_every=1),
        # the paper's Table 1 shape
        dict(name="paper_L4096", kind="chain", L=4096, T=0.99 * TC, H=0.0, init="hot", sweeps=200, record_every=1),
        # a lattice far larger than the L2 cache (512 MiB, 64-bit words)
        dict(name="large_L65536", kind="chain", L=65536, T=2.0, H=0.0, init="cold", sweeps=4, record_every=1),
        # the finite-size-scaling batch: four sizes at 32 temperatures
        dict(name="fss_batch", kind="batch", sizes="256,512,1024,2048", temps=32, sweeps=100, record_every=10),
        # a burst of requests of mixed size, temperature and length
        dict(name="served_mix", kind="served", requests=24, mix=4, Lmax=4096, sweeps_max=2000),
        # a host configuration taken through a few sweeps and back
        dict(name="buffer_L2048", kind="buffer", L=2048, T=2.2, sweeps=10),
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _some_L(rng: random.Random, lo: int, hi: int) -> int:
    """A lattice size (a multiple of 64), every other one a power of two."""
    if rng.random() < 0.5:
        return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))
    return max(lo, min(hi, 64 * round(_log_uniform(rng, lo, hi) / 64)))


def draw(rng: random.Random):
    kind = rng.choice(("chain", "chain", "chain", "chain", "chain", "anneal", "buffer", "batch", "served"))
    T = round(rng.uniform(1.5, 3.5), 3)
    if kind == "chain":
        H = round(rng.uniform(-0.5, 0.5), 3) if rng.random() < 0.25 else 0.0
        L = _some_L(rng, 64, 32768 if H else 65536)
        most = max(1, min(1000, int(1.2e10 / (L * L))))
        return dict(kind="chain", L=L, T=T, H=H, init=rng.choice(("hot", "cold")),
                    sweeps=max(1, round(_log_uniform(rng, max(1, most / 10), most))),
                    record_every=rng.choice((0, 1, 1, 3, 10)))
    if kind == "anneal":
        return dict(kind="anneal", L=_some_L(rng, 64, 512), sweeps=rng.randint(1, 20))
    if kind == "buffer":
        return dict(kind="buffer", L=_some_L(rng, 256, 4096), T=T, sweeps=rng.randint(1, 20))
    if kind == "batch":
        sizes = sorted(rng.sample((64, 128, 192, 256, 320, 512, 704, 1024, 1088, 2048), rng.randint(2, 4)))
        temps = rng.randint(3, 32)
        per_sweep = temps * sum(L * L for L in sizes)
        sweeps = max(10, min(200, int(1.5e10 / per_sweep)))
        return dict(kind="batch", sizes=",".join(map(str, sizes)), temps=temps, sweeps=sweeps,
                    record_every=rng.choice((1, 10)))
    return dict(kind="served", requests=rng.randint(6, 24), mix=rng.randint(0, 999), Lmax=rng.choice((512, 1024, 2048, 4096)),
                sweeps_max=rng.choice((300, 500, 1000)))


def _requests(case):
    """Size, temperature, length and sample spacing of each request (the seeds come from prepare)."""
    r = random.Random(1000 + case["mix"])
    Ls = [L for L in (64, 128, 256, 512, 1024, 2048, 4096) if L <= case["Lmax"]]
    return [dict(L=r.choice(Ls), T=round(r.uniform(1.5, 3.5), 4),
                 nsweeps=round(_log_uniform(r, 100, case["sweeps_max"])), record_every=10)
            for _ in range(case["requests"])]


def _batch_lattices(case):
    n = case["temps"]
    return [dict(L=int(L), T=2.20 + i * 0.15 / (n - 1), stream_id=n * k + i)
            for k, L in enumerate(case["sizes"].split(",")) for i in range(n)]


def _host_spins(L: int, seed: int) -> np.ndarray:
    bits = np.random.Generator(np.random.PCG64(seed)).integers(0, 2, (L, L), dtype=np.int8)
    return (2 * bits - 1).astype(np.int8)


ANNEAL_T = (3.0, 2.75, 2.5, 2.4, 2.3, 2.25, 2.2, 2.1, 2.0, 1.8)


class _Spins:
    """A lattice's packed rows on the device, for torch."""

    def __init__(self, lat: ising.Lattice):
        self.lat = lat
        ptr, _ = ising.ising_device_spins(lat.handle)
        self.__cuda_array_interface__ = dict(shape=(lat.L, lat.L // 8), typestr="|u1", data=(ptr, False), version=2)


def _spins(lat: ising.Lattice) -> torch.Tensor:
    return torch.as_tensor(_Spins(lat), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        lat = ising.Lattice(case["L"], case["T"], seed=seed, init=case["init"], H=case["H"])
        return dict(case=case, lat=lat, spins=_spins(lat))
    if kind == "anneal":
        lat = ising.Lattice(case["L"], ANNEAL_T[0], seed=seed, init="hot")
        return dict(case=case, lat=lat, spins=_spins(lat), k=0)
    if kind == "buffer":
        return dict(case=case, seed=seed, host=_host_spins(case["L"], seed))
    if kind == "batch":
        lats = [ising.Lattice(d["L"], d["T"], seed=seed, stream_id=d["stream_id"], init="hot")
                for d in _batch_lattices(case)]
        batch = ising.Batch(lats, [case["sweeps"]] * len(lats), case["record_every"])
        n = case["temps"]
        spins = [[_spins(l) for l in lats[i:i + n]] for i in range(0, len(lats), n)]
        return dict(case=case, lats=lats, batch=batch, spins=spins, seen=0)
    reqs = _requests(case)
    seeds = np.random.Generator(np.random.PCG64(seed)).integers(0, 2 ** 63, len(reqs))
    for r, s in zip(reqs, seeds):
        r["seed"] = int(s)
    return dict(case=case, reqs=reqs, server=ising.Server(keep_samples=True))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "chain":
        M, E = state["lat"].sweep(case["sweeps"], case["record_every"], collect=True)
        return dict(M=M, E=E, spins=state["spins"])
    if kind == "anneal":
        lat = state["lat"]
        lat.set_temperature(ANNEAL_T[state["k"] % len(ANNEAL_T)])
        state["k"] += 1
        M, E = lat.sweep(case["sweeps"], 1, collect=True)
        return dict(M=M, E=E, spins=state["spins"])
    if kind == "buffer":
        with ising.Lattice(case["L"], case["T"], seed=state["seed"], spins=state["host"]) as lat:
            M, E = lat.sweep(case["sweeps"], 1, collect=True)
            return dict(M=M, E=E, spins=lat.spins())
    if kind == "batch":
        state["batch"].run()
        samples = [l.samples(state["seen"], case["sweeps"]) for l in state["lats"]]
        state["seen"] += len(samples[0][0])
        return dict(M=np.stack([m for m, _ in samples]), E=np.stack([e for _, e in samples]),
                    spins=[torch.stack(s) for s in state["spins"]])
    server = state["server"]
    ids = [server.submit(init="hot", **r) for r in state["reqs"]]
    left = len(ids)
    while left:
        left -= len(server.poll(wait_s=1.0))
    samples = [server.samples(i) for i in ids]
    return dict(M=np.concatenate([m for m, _ in samples]), E=np.concatenate([e for _, e in samples]))


def _sites_and_attempts(case):
    """(sites that the call holds, attempted spin updates, recorded samples) of one pass."""
    kind = case["kind"]
    if kind == "served":
        reqs = _requests(case)
        return (sum(r["L"] ** 2 for r in reqs), sum(r["L"] ** 2 * r["nsweeps"] for r in reqs),
                sum(r["nsweeps"] // r["record_every"] for r in reqs))
    if kind == "batch":
        lats = _batch_lattices(case)
        sites = sum(d["L"] ** 2 for d in lats)
        return sites, sites * case["sweeps"], len(lats) * (case["sweeps"] // case["record_every"])
    every = case.get("record_every", 1)
    sites = case["L"] ** 2
    return sites, sites * case["sweeps"], case["sweeps"] // every if every else 0


def work(case):
    """The lattice read and written once (a bit per spin; a byte where the host's configuration has one), the samples
    written; 16 integer operations per attempted update: a quarter of the ten rounds of Philox4x32 (two widening
    multiplications and two three-input XORs each), the counter, two comparisons, the bit logic and the masked flip."""
    sites, attempts, samples = _sites_and_attempts(case)
    return {"bytes": (2 * sites if case["kind"] == "buffer" else sites / 4) + 16 * samples, "flops": 16 * attempts}


# ------------------------------------------------------------- plain torch --
MASK = 0xFFFFFFFF
CHUNK = 1 << 25  # sites updated at a time


def _philox(x0, x1, x2, x3, seed):
    """Philox4x32-10 in 64-bit integers."""
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        pa, pb = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = ((pb >> 32) & MASK) ^ x1 ^ k0, pb & MASK, ((pa >> 32) & MASK) ^ x3 ^ k1, pa & MASK
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return torch.stack((x0, x1, x2, x3), dim=-1)


def _hot(L, seed, stream_id, dev):
    g = torch.arange(L * L // 128, dtype=torch.int64, device=dev)
    w = _philox(g & MASK, g >> 32, torch.full_like(g, MASK), torch.full_like(g, stream_id << 1), seed)
    bits = (w[..., None] >> torch.arange(32, device=dev)) & 1
    return bits.to(torch.int8).reshape(L, L)


def _threshold_table(T, H, dev):
    """Acceptance thresholds of the classes (S, anti-aligned neighbours), 2^32 where a flip is always taken."""
    tab = []
    for S in (-1, 1):
        for c in range(5):
            dE = 2.0 * S * (S * (4 - 2 * c) + H)
            tab.append(2 ** 32 if dE <= 0 else min(MASK, math.floor(math.ldexp(math.exp(-dE / T), 32))))
    return torch.tensor(tab, dtype=torch.int64, device=dev)


def _step(s, tab, t, p, seed, stream_id):
    """One checkerboard step of the lattice s (0 / 1 per site) in place."""
    L, dev = s.shape[0], s.device
    rows = max(1, min(L, CHUNK // L))
    for y0 in range(0, L, rows):
        y = torch.arange(y0, min(L, y0 + rows), dtype=torch.int64, device=dev)
        cur = s[y0:y0 + len(y)]
        g = (y[:, None] * (L // 8) + torch.arange(L // 8, device=dev)).reshape(-1)
        u = _philox(g & MASK, g >> 32, torch.full_like(g, t), torch.full_like(g, stream_id << 1 | p), seed)
        u = u.reshape(len(y), L // 2).repeat_interleave(2, dim=1)
        anti = (cur ^ s[(y - 1) % L]) + (cur ^ s[(y + 1) % L]) + (cur ^ cur.roll(1, 1)) + (cur ^ cur.roll(-1, 1))
        mine = ((y[:, None] + torch.arange(L, device=dev)) & 1) == p
        flip = mine & (u < tab[(5 * cur + anti).to(torch.int64)])
        cur ^= flip.to(torch.int8)


def _observables(s):
    L = s.shape[0]
    up = int(s.sum(dtype=torch.int64))
    anti = int((s ^ s.roll(1, 0)).sum(dtype=torch.int64) + (s ^ s.roll(1, 1)).sum(dtype=torch.int64))
    return 2 * up - L * L, 2 * anti - 2 * L * L


def _packed(s):
    out = torch.zeros((s.shape[0], s.shape[1] // 8), dtype=torch.uint8, device=s.device)
    for b in range(8):
        out |= s[:, b::8].to(torch.uint8) << b
    return out


def _simulate(s, T, H, seed, stream_id, sweeps, record_every):
    M, E = [], []
    tab = _threshold_table(T, H, s.device)
    for t in range(sweeps):
        for p in (0, 1):
            _step(s, tab, t, p, seed, stream_id)
        if record_every and (t + 1) % record_every == 0:
            m, e = _observables(s)
            M.append(m)
            E.append(e)
    return np.array(M, dtype=np.int64), np.array(E, dtype=np.int64)


def exact(case, seed):
    """A pass on a new state in plain torch: the update rule, the random-number contract and the observables of
    include/ising.h on one byte per spin."""
    kind = case["kind"]
    sites, attempts, _ = _sites_and_attempts(case)
    if kind == "served":
        lats = [dict(r, stream_id=0) for r in _requests(case)]
        seeds = [int(x) for x in np.random.Generator(np.random.PCG64(seed)).integers(0, 2 ** 63, len(lats))]
    elif kind == "batch":
        lats = [dict(d, nsweeps=case["sweeps"], record_every=case["record_every"]) for d in _batch_lattices(case)]
        seeds = [seed] * len(lats)
    else:
        T = ANNEAL_T[0] if kind == "anneal" else case["T"]
        lats = [dict(L=case["L"], T=T, nsweeps=case["sweeps"], record_every=case.get("record_every", 1), stream_id=0)]
        seeds = [seed]
    if sum(4e-3 * d["nsweeps"] for d in lats) + attempts / 1.5e9 > 15 or not torch.cuda.is_available():
        return None
    dev = torch.device("cuda")
    out = []
    for d, sd in zip(lats, seeds):
        L = d["L"]
        if kind == "buffer":
            s = torch.from_numpy((_host_spins(L, sd) > 0).astype(np.int8)).to(dev)
        elif case.get("init", "hot") == "hot":
            s = _hot(L, sd, d["stream_id"], dev)
        else:
            s = torch.ones((L, L), dtype=torch.int8, device=dev)
        M, E = _simulate(s, d["T"], case.get("H", 0.0), sd, d["stream_id"], d["nsweeps"], d["record_every"])
        out.append((M, E, s))
    if kind == "served":
        return dict(M=np.concatenate([m for m, _, _ in out]), E=np.concatenate([e for _, e, _ in out]))
    if kind == "batch":
        n = case["temps"]
        return dict(M=np.stack([m for m, _, _ in out]), E=np.stack([e for _, e, _ in out]),
                    spins=[torch.stack([_packed(s) for _, _, s in out[i:i + n]]) for i in range(0, len(out), n)])
    M, E, s = out[0]
    return dict(M=M, E=E, spins=(2 * s.cpu().numpy() - 1).astype(np.int8) if kind == "buffer" else _packed(s))
