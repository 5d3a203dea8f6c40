"""Tiled reductions, tiled clusters and batched pair counts against the oracle at
the sizes where they can go wrong: tile edges and remainders, tiles that wrap
onto themselves, the most species, counters emptied between sites."""
import numpy as np
import pytest

import oracle as O
from paper_2503_12591_gb300 import diff, smcx
from paper_2503_12591_gb300.inputs import epi_gaussian

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lattice(kind, dims, M, K, storage, seed, W=None):
    N = O.n_sites(kind, dims)
    cfg = np.random.default_rng(seed).integers(0, M, N).astype(np.int8)
    lat = smcx.Lattice(kind, dims, M, [1.0 / M] * M, storage=storage, stream=torch.cuda.current_stream())
    V = epi_gaussian(K, M, 20.0, seed)
    lat.set_epi(V)
    lat.set_config(cfg)
    if W is not None:
        lat.set_qsro(W)
    return lat, cfg, V


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 4, 5), (15, 2, 16), (17, 31, 9), (61, 24, 46)])
@pytest.mark.parametrize("M,K,storage", [(1, 3, smcx.INT8), (4, 2, smcx.PACKED4), (5, 3, smcx.PACKED4),
                                         (5, 1, smcx.INT8), (8, 3, smcx.INT8), (6, 2, smcx.PACKED4)])
def test_fcc_counts_and_energies(dims, M, K, storage):
    lat, cfg, V = _lattice(smcx.FCC, dims, M, K, storage, 3)
    assert (lat.pair_counts() == O.pair_counts(O.FCC, dims, M, K, cfg)).all()
    assert lat.energy() == O.energy(O.FCC, dims, M, K, V, cfg)
    if M > 1:
        W = np.random.default_rng(8).integers(-300, 301, (K, M)).astype(np.int32)
        lat.set_qsro(W)
        assert lat.energy() == O.energy_qsro(O.FCC, dims, M, K, V, W, cfg)
    lat.close()


@pytest.mark.parametrize("kind,dims,M,K,storage", [
    (smcx.FCC, (2, 3, 2), 4, 3, smcx.INT8), (smcx.FCC, (25, 13, 26), 5, 3, smcx.PACKED4),
    (smcx.FCC, (13, 12, 37), 8, 2, smcx.INT8), (smcx.FCC, (50, 49, 4), 3, 1, smcx.PACKED4),
    (smcx.BCC, (4, 3, 5), 4, 2, smcx.INT8), (smcx.BCC, (33, 17, 20), 4, 4, smcx.PACKED4),
    (smcx.BCC, (16, 49, 9), 3, 3, smcx.INT8), (smcx.BCC, (21, 10, 8), 6, 4, smcx.INT8)])
@pytest.mark.parametrize("qsro", [False, True])
def test_clusters_in_tiles(kind, dims, M, K, storage, qsro):
    lat, cfg, V = _lattice(kind, dims, M, K, storage, 5)
    W = np.random.default_rng(8).integers(-60, 61, (K, M)).astype(np.int32)
    if qsro:
        lat.set_qsro(W)
    N = cfg.size
    e2 = torch.empty(N, dtype=torch.int32, device="cuda")
    lat.local_energy(e2.data_ptr())
    lat.synchronize()
    want = (O.local_energy2_qsro(kind, dims, M, K, V, W, cfg) if qsro else O.local_energy2(kind, dims, M, K, V, cfg))
    assert (e2.cpu().numpy() == want).all()
    lab = torch.empty(N, dtype=torch.int32, device="cuda")
    for q in (0.0, 0.2, 0.5, 0.85, 1.0):
        thr = int(np.quantile(want, q))
        n = lat.clusters(thr, lab.data_ptr())
        ref, rn = (O.clusters_qsro(kind, dims, M, K, V, W, cfg, thr) if qsro
                   else O.clusters(kind, dims, M, K, V, cfg, thr))
        assert n == rn and (lab.cpu().numpy() == ref).all()
        for min_size, most in ((1, 3000), (3, 7)):
            roots, sizes, counts = lat.cluster_summary(lab.data_ptr(), min_size, most)
            oroots, osizes, ocounts = O.cluster_summary(ref, cfg, M, min_size)
            k = min(most, oroots.size)
            assert roots.tolist() == oroots[:k].tolist() and sizes.tolist() == osizes[:k].tolist()
            assert counts.tolist() == ocounts[:k].tolist()
    lat.close()


@pytest.mark.parametrize("kind,dims,M,K,B", [
    (smcx.BCC, (2, 2, 2), 4, 4, 3), (smcx.BCC, (3, 5, 7), 8, 4, 5), (smcx.BCC, (14, 15, 16), 4, 3, 3),
    (smcx.BCC, (5, 4, 3), 5, 1, 9), (smcx.BCC, (9, 9, 9), 1, 2, 2), (smcx.FCC, (2, 2, 3), 7, 3, 4),
    (smcx.FCC, (12, 13, 11), 5, 3, 3), (smcx.FCC, (3, 3, 3), 4, 2, 11), (smcx.FCC, (1, 2, 2), 3, 1, 4),
    (smcx.BCC, (8, 8, 8), 9, 4, 3)])
def test_pair_counts_batch_sizes(kind, dims, M, K, B):
    N = O.n_sites(kind, dims)
    cfg = np.random.default_rng(11).integers(0, M, (B, N)).astype(np.int8)
    pad = torch.zeros(B * N + 3, dtype=torch.int8, device="cuda")
    for off in (0, 2):  # whole words of a configuration, and not
        view = pad[off:off + B * N]
        view.copy_(torch.from_numpy(cfg.reshape(-1)))
        C = diff.pair_counts(view.view(B, N), kind, dims, M, K).cpu().numpy()
        for b in range(B):
            assert (C[b] == O.pair_counts(kind, dims, M, K, cfg[b])).all()


@pytest.mark.parametrize("dims,B", [((3, 4, 5), 3), ((3, 3, 5), 600), ((3, 3, 5), 620), ((5, 5, 5), 620), ((6, 5, 5), 310),
                                    ((6, 7, 7), 310), ((7, 7, 7), 310), ((8, 8, 7), 310), ((8, 8, 8), 160), ((9, 8, 8), 5)])
@pytest.mark.parametrize("M,K", [(5, 1), (8, 1), (8, 2), (5, 3), (8, 3), (6, 4)])
def test_pair_counts_batch_many_species(dims, B, M, K):
    # five to eight species: both sides of the sizes at which whole shells take over
    # from half shells, aligned and not, one configuration with an id out of range
    N = O.n_sites(smcx.BCC, dims)
    cfg = np.random.default_rng(12).integers(0, M, (B, N)).astype(np.int8)
    cfg[B - 1, N // 2] = M
    pad = torch.zeros(B * N + 3, dtype=torch.int8, device="cuda")
    for off in (0, 2):
        view = pad[off:off + B * N]
        view.copy_(torch.from_numpy(cfg.reshape(-1)))
        C = diff.pair_counts(view.view(B, N), smcx.BCC, dims, M, K).cpu().numpy()
        for b in [*range(0, B - 1, max(1, B // 8))]:
            assert (C[b] == O.pair_counts(smcx.BCC, dims, M, K, cfg[b])).all()
        assert (C[B - 1] == -1).all()


@pytest.mark.parametrize("dims,nt", [((40, 38, 42), (12, 12, 12)), ((18, 21, 40), (2, 2, 2)), ((34, 33, 32), (2, 2, 2))])
@pytest.mark.parametrize("M,K,storage", [(5, 3, smcx.PACKED4), (4, 2, smcx.INT8), (8, 3, smcx.INT8)])
def test_qsro_sweeps_few_and_many_tiles(dims, nt, M, K, storage):
    # 216 tiles a colour: a thread per trial; one tile a colour: four threads per
    # trial, in the boxes of 20-cell and of 17-cell tiles
    W = np.random.default_rng(8).integers(-300, 301, (K, M)).astype(np.int32)
    lat, cfg, V = _lattice(smcx.FCC, dims, M, K, storage, 9)
    lat.set_qsro(W)
    lat.set_schedule((4, nt))
    lat.sweep(900.0, 2, 31)
    st = O.sweep_qsro(O.FCC, dims, M, K, V, W, cfg, 900.0, 2, 31, L=4, nt=nt)
    assert (lat.get_config() == cfg).all()
    assert lat.state()[1].tolist() == st.tolist()
    assert lat.energy() == O.energy_qsro(O.FCC, dims, M, K, V, W, cfg)
    lat.close()


@pytest.mark.parametrize("proposal,R,lo,hi,tile", [(0, 40, 24, 66, 12), (1, 40, 24, 66, 12), (2, 33, 12, 72, 14), (1, 1, 16, 16, 8),
                                                   (0, 600, 12, 12, 6)])
def test_batch_list_longer_than_the_grid(proposal, R, lo, hi, tile):
    # tile passes drawn from the list by CTAs that run ahead of other replicas
    stream = torch.cuda.current_stream()
    V = epi_gaussian(4, 4, 20.0, 2)
    edges = np.linspace(lo, hi, R).astype(int)

    def lattice(r):
        n = int(edges[r])
        nt = 2 * -(-n // (2 * tile))
        lat = smcx.Lattice(smcx.BCC, (n, n, n), 4, [0.25] * 4, init_seed=50 + r, storage=smcx.PACKED4,
                           sched=(3, (nt, nt, nt)), stream=stream)
        lat.set_replica(r)
        lat.set_epi(V)
        lat.set_proposal(proposal)
        return lat

    T = np.linspace(400.0, 2400.0, R)
    lats = [lattice(r) for r in range(R)]
    b = smcx.Batch(lats, stream)
    b.sweep(T, 1, 9)
    b.sweep(T, 3, 9)
    for r in range(0, R, max(1, R // 20)):
        one = lattice(r)
        one.sweep(T[r], 4, 9)
        assert (lats[r].get_config() == one.get_config()).all()
        assert lats[r].state()[1].tolist() == one.state()[1].tolist()
        one.close()
    b.close()


@pytest.mark.parametrize("M,R,block", [(6, 56, 0), (6, 57, 0), (8, 57, 256), (5, 19, 128), (6, 48, 0), (4, 57, 0)])
def test_batch_tiles_in_place(M, R, block):
    # 8 tiles a replica and colour: two counter words on evenly filled SMs (448, 456 and
    # 152 tiles) keep their tiles, 384 tiles and one word draw them
    stream = torch.cuda.current_stream()
    V = epi_gaussian(4, M, 20.0, 7)

    def lattice(r):
        lat = smcx.Lattice(smcx.BCC, (24, 25 + r % 3, 26), M, [1.0 / M] * M, init_seed=70 + r, storage=smcx.INT8,
                           sched=(3, (4, 4, 4)), stream=stream)
        lat.set_replica(r)
        lat.set_epi(V)
        return lat

    T = np.linspace(500.0, 2400.0, R)
    lats = [lattice(r) for r in range(R)]
    b = smcx.Batch(lats, stream)
    b.set_block(block)
    b.sweep(T, 1, 9)
    b.sweep(T, 3, 9)
    assert b.info()["grid"] == 8 * R
    for r in range(0, R, 3):
        one = lattice(r)
        one.sweep(T[r], 4, 9)
        assert (lats[r].get_config() == one.get_config()).all()
        assert lats[r].state()[1].tolist() == one.state()[1].tolist()
        one.close()
    cfg = O.init_config(O.BCC, (24, 25, 26), M, [1.0 / M] * M, 70)
    O.sweep(O.BCC, (24, 25, 26), M, 4, V, cfg, T[0], 4, 9, L=3, nt=(4, 4, 4))
    assert (lats[0].get_config() == cfg).all()
    b.close()
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("L,nt,dims", [(3, 2, (24, 23, 22)), (3, 2, (30, 27, 25)), (3, 2, (36, 33, 31)), (3, 2, (32, 31, 30)),
                                       (4, 2, (32, 27, 29)),
                                       (4, 2, (40, 33, 36)), (4, 4, (44, 43, 42)), (5, 2, (40, 34, 31)), (6, 2, (40, 38, 36))])
@pytest.mark.parametrize("M,proposal,storage", [(4, 0, smcx.PACKED4), (4, 1, smcx.PACKED4), (4, 2, smcx.INT8), (6, 0, smcx.INT8)])
def test_bcc_lane_orders(L, nt, dims, M, proposal, storage):
    # 4^3 to 6^3 link-cell slots, full and ragged tiles; L = 6 has no order of its own
    lat, cfg, V = _lattice(smcx.BCC, dims, M, 4, storage, 17)
    lat.set_schedule((L, (nt, nt, nt)))
    lat.set_proposal(proposal)
    lat.sweep(1100.0, 2, 23)
    st = O.sweep(O.BCC, dims, M, 4, V, cfg, 1100.0, 2, 23, L=L, nt=(nt, nt, nt), proposal=proposal)
    assert (lat.get_config() == cfg).all()
    assert lat.state()[1].tolist() == st.tolist()
    lat.close()


@pytest.mark.parametrize("L,nt,dims", [(3, 2, (6, 7, 9)), (4, 2, (12, 17, 24)), (6, 2, (36, 25, 31)), (3, 4, (24, 36, 33)),
                                       (3, 2, (24, 23, 19)), (4, 2, (32, 29, 26)), (5, 2, (40, 31, 33)), (7, 2, (40, 39, 37)),
                                       (3, 14, (84, 85, 86))])
@pytest.mark.parametrize("M,K,proposal,storage", [(4, 4, 0, smcx.PACKED4), (4, 4, 1, smcx.INT8), (4, 3, 0, smcx.INT8),
                                                  (6, 4, 0, smcx.PACKED4), (3, 2, 0, smcx.PACKED4), (5, 1, 0, smcx.INT8)])
def test_bcc_lanes_per_trial(L, nt, dims, M, K, proposal, storage):
    # two and four lanes per trial, 2^3 to 4^3 slots, and one: 84 cells in 14 tiles, and
    # shared directions of link cells above 6 (2 L^3 of them)
    lat, cfg, V = _lattice(smcx.BCC, dims, M, K, storage, 21)
    lat.set_schedule((L, (nt, nt, nt)))
    lat.set_proposal(proposal)
    lat.sweep(1300.0, 2, 29)
    st = O.sweep(O.BCC, dims, M, K, V, cfg, 1300.0, 2, 29, L=L, nt=(nt, nt, nt), proposal=proposal)
    assert (lat.get_config() == cfg).all()
    assert lat.state()[1].tolist() == st.tolist()
    lat.close()


@pytest.mark.parametrize("M,scale,proposal", [(4, 20.0, 0), (4, 20.0, 2), (6, 20.0, 0), (4, 9000.0, 0), (7, 9000.0, 0)])
def test_batch_lanes_per_trial(M, scale, proposal):
    # both counter widths and both numbers of byte planes
    stream = torch.cuda.current_stream()
    V = epi_gaussian(4, M, scale, 5)
    dims = [(12, 14, 16), (24, 18, 21), (8, 9, 24)]
    T = [700.0, 1100.0, 1900.0]
    lats = []
    for r, d in enumerate(dims):
        lat = smcx.Lattice(smcx.BCC, d, M, [1.0 / M] * M, init_seed=30 + r, storage=smcx.INT8, sched=(4, (2, 2, 2)),
                           stream=stream)
        lat.set_replica(r)
        lat.set_epi(V)
        lat.set_proposal(proposal)
        lats.append(lat)
    cfg = [lat.get_config().copy() for lat in lats]
    b = smcx.Batch(lats, stream)
    b.sweep(T, 3, 13)
    for r, d in enumerate(dims):
        st = O.sweep(O.BCC, d, M, 4, V, cfg[r], T[r], 3, 13, replica=r, L=4, nt=(2, 2, 2), proposal=proposal)
        assert (lats[r].get_config() == cfg[r]).all()
        assert lats[r].state()[1].tolist() == st.tolist()
    b.close()


@pytest.mark.parametrize("kind,L,nt,dims", [(smcx.BCC, 6, 2, (36, 25, 31)), (smcx.BCC, 7, 2, (40, 39, 37)),
                                            (smcx.BCC, 9, 2, (40, 38, 36)), (smcx.BCC, 18, 2, (40, 39, 37)),
                                            (smcx.FCC, 5, 2, (30, 27, 23)), (smcx.FCC, 6, 2, (30, 27, 25)),
                                            (smcx.FCC, 14, 2, (30, 29, 28)), (smcx.FCC, 7, 4, (56, 29, 30))])
@pytest.mark.parametrize("proposal", [1, 2])
def test_shared_directions_of_long_link_cells(kind, L, nt, dims, proposal):
    # 2 L^3 (BCC) or 4 L^3 (FCC) phases a pass, 432 to 11,664 of them
    M, K = (4, 4) if kind == smcx.BCC else (5, 3)
    lat, cfg, V = _lattice(kind, dims, M, K, smcx.PACKED4, 33)
    nts = tuple(nt if n // nt >= L else 2 for n in dims)
    lat.set_schedule((L, nts))
    lat.set_proposal(proposal)
    start = cfg.copy()
    lat.sweep(1000.0, 2, 37)
    st = O.sweep(kind, dims, M, K, V, cfg, 1000.0, 2, 37, L=L, nt=nts, proposal=proposal)
    assert (lat.get_config() == cfg).all()
    assert lat.state()[1].tolist() == st.tolist()
    if kind == smcx.BCC:
        lat2 = smcx.Lattice(kind, dims, M, [0.25] * 4, storage=smcx.PACKED4, sched=(L, nts),
                            stream=torch.cuda.current_stream())
        lat2.set_epi(V)
        lat2.set_config(start)
        lat2.set_proposal(proposal)
        b = smcx.Batch([lat2], torch.cuda.current_stream())
        b.sweep([1000.0], 2, 37)
        assert (lat2.get_config() == cfg).all()
        b.close()
        lat2.close()
    lat.close()


@pytest.mark.parametrize("dims", [(25, 24, 27), (28, 29, 27), (32, 31, 33), (40, 39, 36), (48, 50, 41), (60, 49, 55), (7, 150, 31)])
@pytest.mark.parametrize("kind,M,K,storage", [(smcx.FCC, 5, 3, smcx.PACKED4), (smcx.FCC, 8, 2, smcx.INT8),
                                              (smcx.BCC, 4, 4, smcx.PACKED4), (smcx.BCC, 3, 2, smcx.INT8)])
def test_reduction_tile_edges(dims, kind, M, K, storage):
    # lattices of fewer than two 12-cell tiles per SM: tiles of 4, 6, 7, 8, 10 and 12 cells;
    # two-shell BCC int8 lattices on both sides of the 2^16 sites up to which they gather
    lat, cfg, V = _lattice(kind, dims, M, K, storage, 43)
    assert (lat.pair_counts() == O.pair_counts(kind, dims, M, K, cfg)).all()
    assert lat.energy() == O.energy(kind, dims, M, K, V, cfg)
    e2 = torch.empty(cfg.size, dtype=torch.int32, device="cuda")
    lat.local_energy(e2.data_ptr())
    lat.synchronize()
    assert (e2.cpu().numpy() == O.local_energy2(kind, dims, M, K, V, cfg)).all()
    lat.close()
