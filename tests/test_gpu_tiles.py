"""Tiled reductions against the oracle at
the sizes where they can go wrong: tile edges and remainders, tiles that wrap
onto themselves, the most species, counters emptied between sites."""
import numpy as np
import pytest

import oracle as O
from paper_2503_12591_gb300 import smcx
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
        try:
            lat.set_qsro(W)
        except smcx.SmcxError:
            return  # no schedule for the longer reach: the model is refused
        assert lat.energy() == O.energy_qsro(O.FCC, dims, M, K, V, W, cfg)
    lat.close()
