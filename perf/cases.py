"""What a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain numbers and texts; its "do" names the kind of work:

  sweep      Monte-Carlo sweeps of one lattice, then (if asked) its exact energy
  observe    one measurement interval of a production run: energy and
             Warren-Cowley SRO of the configuration, then the sweeps to the next
  anneal     one temperature of an annealing schedule: sweeps with the exact
             energy recorded after each, reduced to <E>, Var(E) and C_V
  qsro       sweeps under the qSRO model, and the energy under it
  replicas   many lattices of uneven sizes and temperatures in one launch
  fluct      fluctuation sums of every replica of a batch, then its sweeps
  fit        one step of fitting the EPI table: pair counts of a batch of
             configurations, their energies, the loss and its gradient
  clusters   local-energy classes, clusters and the summary of the largest

Lattices live in tensors that the program holds (Lattice.wrap), so a case's
configuration after the sweeps is the program's own buffer.  Every trajectory
is an exact function of the seeds, so configurations, energies and counts have
to come out the same bit for bit; the few floating results have a tolerance.
"""
import math

import numpy as np
import torch

from paper_2503_12591_gb300 import diff, smcx
from paper_2503_12591_gb300.inputs import batched_edges, epi_gaussian, log_temperatures

BCC, FCC = smcx.BCC, smcx.FCC
SITE, TILE, BLOCK = smcx.PROPOSAL_SITE, smcx.PROPOSAL_TILE, smcx.PROPOSAL_BLOCK
# compositions: equiatomic up to four species, the five-species alloy's own
COMP5 = [0.3, 0.25, 0.2, 0.15, 0.1]


def listed():
    return [
        # the smallest call: a lattice of 8,192 sites, as in a first try or a
        # finite-size study; latency and launches count
        dict(name="bcc16", do="sweep", kind="bcc", nx=16, ny=16, nz=16, M=4, K=4, storage="int8", proposal="site",
             T=1000.0, sweeps=2, energy=1),
        # edges that nothing divides: ragged tiles, rows that straddle words
        dict(name="bcc_ragged", do="sweep", kind="bcc", nx=301, ny=257, nz=203, M=4, K=4, storage="packed4",
             proposal="site", T=1500.0, sweeps=1, energy=0),
        # the plain throughput run: 33.5M sites at one temperature, energy and
        # SRO at intervals, with the schedule that tuning gives for this size
        dict(name="bcc256_observe", do="observe", kind="bcc", nx=256, ny=256, nz=256, M=4, K=4, storage="int8",
             proposal="site", T=1500.0, sweeps=4, L=3, tile=15),
        # the largest run: a billion sites, one direction per tile and phase
        dict(name="bcc800", do="sweep", kind="bcc", nx=800, ny=800, nz=800, M=4, K=4, storage="packed4",
             proposal="tile", T=1200.0, sweeps=1, energy=0),
        # one temperature of an annealing run with a two-shell model
        dict(name="bcc320_anneal", do="anneal", kind="bcc", nx=320, ny=320, nz=320, M=4, K=2, storage="packed4",
             proposal="site", T=1600.0, sweeps=6),
        # the five-species FCC alloy at 256M sites
        dict(name="fcc400", do="sweep", kind="fcc", nx=400, ny=400, nz=400, M=5, K=3, storage="packed4",
             proposal="tile", T=1200.0, sweeps=1, energy=0),
        # a ragged FCC box annealed with a direction per trial
        dict(name="fcc_ragged_anneal", do="anneal", kind="fcc", nx=151, ny=180, nz=133, M=5, K=3, storage="int8",
             proposal="site", T=1400.0, sweeps=3),
        # the qSRO model on 6.9M sites
        dict(name="fcc120_qsro", do="qsro", kind="fcc", nx=120, ny=120, nz=120, M=5, K=3, storage="packed4", T=1000.0,
             sweeps=1),
        # temperature parallelism: 64 lattices with edges of 24 to 96 cells
        dict(name="replicas64", do="replicas", R=64, lo=24, hi=96, proposal="tile", sweeps=4, L=3, tile=18),
        # thermal derivatives: fluctuation sums between the sweeps of 64 replicas
        dict(name="fluct64", do="fluct", R=64, n=48, T=1000.0, sweeps=1),
        # one step of fitting the EPI table to reference energies
        dict(name="fit4096", do="fit", kind="bcc", n=8, M=4, K=4, B=4096),
        # nanostructure analysis of a 16M-site FCC configuration
        dict(name="fcc160_clusters", do="clusters", kind="fcc", nx=160, ny=160, nz=160, M=5, K=3, storage="packed4",
             quantile=0.2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, lo, hi):
    """Three edges around a cube whose cell count is log-uniform in [lo^3, hi^3]."""
    e = _log(rng, lo, hi)
    return [max(8, min(hi, int(round(e * rng.uniform(0.85, 1.18))))) for _ in range(3)]


def draw(rng):
    do = rng.choice(["sweep"] * 6 + ["observe", "anneal", "anneal", "qsro", "replicas", "fluct", "fit", "clusters"])
    T = round(_log(rng, 600.0, 2500.0), 1)
    storage = rng.choice(["int8", "packed4"])
    kind = rng.choice(["bcc", "bcc", "fcc"])
    if do == "sweep":
        nx, ny, nz = _dims(rng, 16, 700) if kind == "bcc" else _dims(rng, 14, 360)
        proposal = rng.choice(["site", "site", "tile", "tile", "block"])
        K = (4 if proposal != "site" else rng.choice([2, 3, 4, 4])) if kind == "bcc" else rng.choice([2, 3, 3])
        M = rng.choice([2, 3, 4, 4, 4]) if kind == "bcc" else rng.choice([3, 4, 5, 5])
        if kind == "fcc" and proposal != "site":
            K = 3
        return dict(do=do, kind=kind, nx=nx, ny=ny, nz=nz, M=M, K=K, storage=storage, proposal=proposal, T=T,
                    sweeps=rng.choice([1, 1, 2]), energy=rng.choice([0, 1]) if nx * ny * nz < 10 ** 7 else 0)
    if do in ("observe", "anneal"):
        nx, ny, nz = _dims(rng, 16, 280) if kind == "bcc" else _dims(rng, 14, 150)
        K = rng.choice([2, 4]) if kind == "bcc" else rng.choice([2, 3])
        M = 4 if kind == "bcc" else rng.choice([4, 5])
        c = dict(do=do, kind=kind, nx=nx, ny=ny, nz=nz, M=M, K=K, storage=storage, proposal="site", T=T,
                 sweeps=rng.randint(2, 5))
        if do == "observe" and kind == "bcc":
            c.update(K=4, L=rng.choice([3, 4]), tile=rng.choice([12, 14, 15, 16, 18, 20]))
        return c
    if do == "qsro":
        nx, ny, nz = _dims(rng, 16, 130)
        return dict(do=do, kind="fcc", nx=nx, ny=ny, nz=nz, M=rng.choice([4, 5]), K=rng.choice([2, 3]), storage=storage,
                    T=T, sweeps=1)
    if do == "replicas":
        L = rng.choice([3, 4])
        return dict(do=do, R=rng.choice([8, 16, 33, 64]), lo=rng.randint(16, 30), hi=rng.randint(40, 96),
                    proposal=rng.choice(["site", "tile", "block"]), sweeps=rng.randint(1, 4), L=L,
                    tile=rng.choice([12, 14, 15, 16, 18]))
    if do == "fluct":
        return dict(do=do, R=rng.choice([8, 24, 64]), n=rng.randint(16, 56), T=T, sweeps=rng.choice([1, 2]))
    if do == "fit":
        n = rng.randint(4, 16) if kind == "bcc" else rng.randint(3, 12)
        return dict(do=do, kind=kind, n=n, M=rng.choice([2, 3, 4, 5]), K=rng.choice([2, 3, 4]) if kind == "bcc" else 3,
                    B=max(64, min(8192, int(_log(rng, 64.0, 2.0e6 / n ** 3 + 65.0)))))
    nx, ny, nz = _dims(rng, 16, 150)
    return dict(do=do, kind=kind, nx=nx, ny=ny, nz=nz, M=4 if kind == "bcc" else 5, K=3, storage=storage,
                quantile=round(rng.uniform(0.05, 0.4), 3))


# ---- inputs ---------------------------------------------------------------
def _kind(case):
    return FCC if case.get("kind") == "fcc" else BCC


def _per_cell(kind):
    return 4 if kind == FCC else 2


def _species(gen, n, M):
    """n random species ids (uint8) at the alloy's composition."""
    if M != 5:
        return torch.randint(0, M, (n,), dtype=torch.uint8, device="cuda", generator=gen)
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    edges = torch.tensor(np.cumsum(COMP5)[:-1], dtype=torch.float32, device="cuda")
    for i in range(0, n, 1 << 26):  # in pieces: random floats of the whole lattice would not be small
        u = torch.rand(min(1 << 26, n - i), device="cuda", generator=gen)
        out[i:i + u.numel()] = torch.bucketize(u, edges, right=True).to(torch.uint8)
    return out


def _store(gen, n, M, storage):
    """A lattice store of n random species: ids, or two per byte (n is even)."""
    if storage == "int8":
        return _species(gen, n, M)
    out = torch.empty(n // 2, dtype=torch.uint8, device="cuda")
    for i in range(0, n, 1 << 27):
        s = _species(gen, min(1 << 27, n - i), M).view(-1, 2)
        out[i // 2:i // 2 + s.shape[0]] = s[:, 0] | (s[:, 1] << 4)
    return out


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _proposal(case):
    return {"site": SITE, "tile": TILE, "block": BLOCK}[case.get("proposal", "site")]


def _epi(kind, K, M, seed):
    return epi_gaussian(K, M, 30.0 if kind == FCC else 20.0, seed)


def _tiles(dims, L, tile):
    """A schedule of link cells of L and tiles of at most `tile` cells."""
    nt = []
    for n in dims:
        t = 2
        while -(-n // t) > tile and n // (t + 2) >= 3:
            t += 2
        nt.append(t)
    return L, tuple(nt)


def _lattice(case, seed, gen, stream, V=None):
    kind, dims = _kind(case), (case["nx"], case["ny"], case["nz"])
    n = dims[0] * dims[1] * dims[2] * _per_cell(kind)
    store = _store(gen, n, case["M"], case["storage"])
    torch.cuda.synchronize()
    lat = smcx.Lattice.wrap(kind, dims, case["M"], store.data_ptr(), store.numel(),
                            smcx.INT8 if case["storage"] == "int8" else smcx.PACKED4, stream=stream, owner=store)
    lat.set_epi(_epi(kind, case["K"], case["M"], seed) if V is None else V)
    if "L" in case:
        lat.set_schedule(_tiles(dims, case["L"], case["tile"]))
    lat.set_proposal(_proposal(case))
    return lat, store


def _edges(case):
    if "n" in case:
        return [case["n"]] * case["R"]
    return [int(n) for n in batched_edges(case["R"], case["lo"], case["hi"])]


def _replicas(case, seed, gen, stream):
    """R cubic BCC lattices in one buffer, and the batch over them."""
    V = _epi(BCC, 4, 4, seed)
    edges = _edges(case)
    at, total = [], 0
    for n in edges:
        at.append(total)
        total += -(-2 * n ** 3 // 256) * 256
    store = _store(gen, total, 4, "int8")
    torch.cuda.synchronize()
    lats = []
    for r, (n, o) in enumerate(zip(edges, at)):
        lat = smcx.Lattice.wrap(BCC, (n, n, n), 4, store.data_ptr() + o, 2 * n ** 3, smcx.INT8, stream=stream,
                                owner=store)
        lat.set_epi(V)
        if "L" in case:
            lat.set_schedule(_tiles((n, n, n), case["L"], case["tile"]))
        lat.set_proposal(_proposal(case))
        lat.set_replica(r)
        lats.append(lat)
    return smcx.Batch(lats, stream), store


def _seed(seed):
    return 1 + (int(seed) * 2654435761) % (1 << 31)


def prepare(case, seed):
    do, gen = case["do"], _gen(seed)
    st = dict(case=case, seed=_seed(seed), stream=torch.cuda.Stream())
    if do == "fit":
        kind, n = _kind(case), case["n"]
        N = n ** 3 * _per_cell(kind)
        st["configs"] = _species(gen, case["B"] * N, case["M"]).view(torch.int8).view(case["B"], N)
        shape = (case["K"], case["M"], case["M"])
        V = _epi(kind, case["K"], case["M"], seed) / 100.0
        # the table as the fit has it (meV), and per-site reference energies
        rough = np.random.default_rng(int(seed)).normal(0.0, 2.0, shape)
        st["V"] = torch.tensor(V + rough + rough.transpose(0, 2, 1), dtype=torch.float32, device="cuda")
        st["target"] = torch.randn(case["B"], device="cuda", generator=gen) * 20.0
        return st
    if do in ("replicas", "fluct"):
        st["batch"], st["store"] = _replicas(case, seed, gen, st["stream"])
        R = case["R"]
        st["T"] = log_temperatures(R) if do == "replicas" else np.full(R, case["T"])
        if do == "fluct":
            st["est"] = diff.BatchFluctuationEstimator(st["batch"], 4, 4, 0)
            torch.cuda.synchronize()
        return st
    st["lat"], st["store"] = _lattice(case, seed, gen, st["stream"])
    if do == "qsro":
        W = np.random.default_rng(int(seed)).integers(-300, 301, (case["K"], case["M"])).astype(np.int32)
        st["lat"].set_qsro(W)
    if do == "clusters":
        # a configuration with short-range order, and the threshold below
        # which a site counts as part of a precipitate
        lat = st["lat"]
        lat.sweep(900.0, 3, st["seed"])
        st["labels"] = torch.empty(lat.N, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        lat.local_energy(st["labels"].data_ptr())
        torch.cuda.synchronize()
        step = max(1, lat.N // 1_000_000)
        sample = st["labels"][::step].to(torch.float32)
        st["thr2"] = int(sample.kthvalue(max(1, int(case["quantile"] * sample.numel())))[0])
    return st


def run(st):
    case, do = st["case"], st["case"]["do"]
    if do == "fit":
        V = st["V"].detach().requires_grad_(True)
        C = diff.pair_counts(st["configs"], _kind(case), (case["n"],) * 3, case["M"], case["K"])
        E = diff.epi_energy(V, C)
        loss = ((E / st["configs"].shape[1] - st["target"]) ** 2).mean()
        loss.backward()
        return C, E.detach(), V.grad
    if do == "replicas":
        st["batch"].sweep(st["T"], case["sweeps"], st["seed"])
        return st["store"]
    if do == "fluct":
        st["est"].add()
        st["batch"].sweep(st["T"], case["sweeps"], st["seed"])
        return st["est"].acc, st["store"]
    lat = st["lat"]
    if do == "sweep":
        lat.sweep(case["T"], case["sweeps"], st["seed"])
        return (st["store"], lat.energy()) if case["energy"] else st["store"]
    if do == "observe":
        E, alpha = lat.energy(), lat.sro()
        lat.sweep(case["T"], case["sweeps"], st["seed"])
        return E, alpha, st["store"]
    if do == "anneal":
        trace, mean, var, cv = lat.sweep_cv(case["T"], case["sweeps"], st["seed"])
        return trace, mean, var, cv, st["store"]
    if do == "qsro":
        lat.sweep(case["T"], case["sweeps"], st["seed"])
        return st["store"], lat.energy()
    n = lat.clusters(st["thr2"], st["labels"].data_ptr())
    roots, sizes, counts = lat.cluster_summary(st["labels"].data_ptr(), 8, 64)
    return n, st["labels"], roots, sizes, counts


# ---- what a pass cannot do without ---------------------------------------
_VECS = {BCC: [8, 14, 26, 50], FCC: [12, 18, 42]}


def _sites(case):
    if case["do"] in ("replicas", "fluct"):
        return sum(2 * n ** 3 for n in _edges(case))
    return case["nx"] * case["ny"] * case["nz"] * _per_cell(_kind(case))


def work(case):
    """bytes: the inputs once and the outputs once.  flops: one addition per
    neighbour of the two sites of a trial, per neighbour of a site measured
    (every pair once)."""
    do, kind = case["do"], _kind(case)
    K = case.get("K", 4)
    nv = _VECS[kind][K - 1]
    if do == "fit":
        N = case["n"] ** 3 * _per_cell(kind)
        KMM = K * case["M"] ** 2
        return dict(bytes=case["B"] * (N + 8 * KMM + 8) + 8 * KMM, flops=case["B"] * (N * nv / 2 + 4 * KMM))
    N = _sites(case)
    store = N / 2 if case.get("storage") == "packed4" else N
    if do == "clusters":
        return dict(bytes=store + 4 * N, flops=N * nv)
    flops = case["sweeps"] * N * 2.0 * nv
    if do == "qsro":
        flops += N * nv
    elif do in ("observe", "anneal", "fluct") or case.get("energy"):
        flops += N * nv / 2
    return dict(bytes=2 * store, flops=flops)


def tolerance(case):
    """Configurations, energies, counts and labels are whole numbers and exact.
    Floating results: SRO, moments and fluctuation sums in 64 bits (the SRO of a
    random configuration is near zero, a difference of two numbers near one);
    the fit's energies and gradient are 64-bit sums rounded to 32 bits, the
    gradient through 32-bit residuals."""
    return {"observe": {"rel": 4e-12}, "anneal": {"rel": 1e-12}, "fluct": {"rel": 1e-12},
            "fit": {"rel": 4e-7}}.get(case["do"], "exact")


# ---- the same in plain torch, 64 bits --------------------------------------
_BASIS = {BCC: [(0, 0, 0), (1, 1, 1)], FCC: [(0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1)]}
_SHELL = {BCC: {3: 0, 4: 1, 8: 2, 11: 3}, FCC: {2: 0, 4: 1, 6: 2}}


def _pair_counts(cfg, kind, M, K):
    """Ordered pair counts [B][K][M][M] of configurations [B][z][y][x][b]."""
    B = cfg.shape[0]
    C = torch.zeros(K, B * M * M, dtype=torch.int64, device=cfg.device)
    row = torch.arange(B, device=cfg.device, dtype=torch.int32).view(B, 1, 1, 1) * (M * M)
    for b, o in enumerate(_BASIS[kind]):
        p = row + cfg[..., b].to(torch.int32) * M
        for x in range(-3, 4):
            for y in range(-3, 4):
                for z in range(-3, 4):
                    k = _SHELL[kind].get(x * x + y * y + z * z, K)
                    par = tuple((v + w) & 1 for v, w in zip((x, y, z), o))
                    if k >= K or par not in _BASIS[kind]:
                        continue
                    d = [(v + w) // 2 for v, w in zip((x, y, z), o)]
                    q = cfg[..., _BASIS[kind].index(par)].roll((-d[2], -d[1], -d[0]), (1, 2, 3))
                    C[k] += torch.bincount((p + q).view(-1), minlength=B * M * M)
    return C.view(K, B, M, M).transpose(0, 1)


def _alpha(C, k, z1, zk, N):
    """Warren-Cowley parameters of shell k, [B][M][M] in 64 bits."""
    Np = C[:, 0].sum(-1).double() / z1
    den = zk * Np[:, :, None] * Np[:, None, :] / N
    return torch.where(den > 0, 1.0 - C[:, k].double() / den, torch.zeros_like(den))


def _unpacked(case, store):
    if case["storage"] == "int8":
        return store
    return torch.stack((store & 15, store >> 4), 1).view(-1)


def exact(case, seed):
    do, kind, gen = case["do"], _kind(case), _gen(seed)
    if do == "fit":
        st = prepare(case, seed)
        B, n = case["B"], case["n"]
        cfg = st["configs"].view(B, n, n, n, _per_cell(kind))
        C = _pair_counts(cfg, kind, case["M"], case["K"])
        V = st["V"].double().requires_grad_(True)
        E = 0.5 * (C.double() * V).sum((1, 2, 3))
        (((E / st["configs"].shape[1] - st["target"].double()) ** 2).mean()).backward()
        return C, E.detach(), V.grad
    if do == "observe":
        cfg = _unpacked(case, _store(gen, _sites(case), case["M"], case["storage"]))
        cfg = cfg.view(1, case["nz"], case["ny"], case["nx"], _per_cell(kind))
        C = _pair_counts(cfg, kind, case["M"], case["K"])
        V = torch.tensor(_epi(kind, case["K"], case["M"], seed), dtype=torch.int64, device="cuda")
        z = [b - a for a, b in zip([0] + _VECS[kind], _VECS[kind])]
        alpha = torch.stack([_alpha(C, k, z[0], z[k], _sites(case))[0] for k in range(case["K"])])
        return int((V * C[0]).sum()) // 2, alpha.cpu().numpy(), None
    if do == "fluct":
        R, n = case["R"], case["n"]
        total = R * (-(-2 * n ** 3 // 256) * 256)
        cfg = _store(gen, total, 4, "int8").view(R, -1)[:, :2 * n ** 3].reshape(R, n, n, n, 2)
        C = _pair_counts(cfg, BCC, 4, 4)
        A = _alpha(C, 0, 8, 8, 2 * n ** 3).reshape(R, 16)
        c = C.reshape(R, 64).double()
        return torch.cat((torch.ones_like(A[:, :1]), A, c, (A[:, :, None] * c[:, None, :]).reshape(R, -1)), 1), None
    return None
