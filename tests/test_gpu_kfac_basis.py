"""K-FAC eigenbases of factor covariances with crowded spectra (eigenvalues within 1e-4 of each other, geometric
sequences, low rank), written into the state directly: orthonormal to fp64 rounding and diagonalising.

Tolerances: a sweep turns every column n - 1 times, each time within an ulp or so, so (sweeps + 2) n 2^-52 on the
entries of U^T U - I; the fp64 sweeps stop at an off-diagonal norm of 1e-14 |C|, and rounding adds about as much."""
import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


@pytest.mark.parametrize("k,spectrum,seed", [(64, "geometric", 2), (64, "crowded", 1), (64, "crowded", 2),
                                             (48, "crowded", 2), (48, "low rank", 1), (32, "crowded", 2),
                                             (33, "linear", 1), (7, "crowded", 1), (4, "crowded", 1),
                                             (3, "crowded", 1), (3, "low rank", 1), (2, "linear", 1), (1, "linear", 1)])
def test_eigenbases_are_orthonormal(dev, k, spectrum, seed):
    rng = np.random.default_rng(seed)
    U = np.linalg.qr(rng.standard_normal((k, k)))[0]
    i = np.arange(k)
    w = {"geometric": lambda: 0.7 ** i, "crowded": lambda: 1 + 1e-4 * rng.standard_normal(k),
         "low rank": lambda: np.where(i < k // 4, 1.0 + i, 0), "linear": lambda: 1.0 + i}[spectrum]()
    C = (U * w) @ U.T
    C = (C + C.T) / 2
    state = torch.zeros(tda.tda_kfac_state_bytes(k, k), dtype=torch.uint8, device=dev)
    d = state.view(torch.float64)
    d[0] = 1.0
    d[8:8 + k * k] = torch.from_numpy(C.ravel()).to(dev)
    d[8 + k * k:8 + 2 * k * k] = d[8:8 + k * k]
    tda.tda_kfac_eigen(k, k, state)
    o = d.cpu().numpy()
    for side in (0, 1):
        sweeps = o[2 + side]
        assert sweeps >= 0
        at = 8 + 2 * k * k + side * (k * k + k)  # a side's basis, then its eigenvalues
        u = o[at:at + k * k].reshape(k, k)
        assert np.abs(u.T @ u - np.eye(k)).max() <= (sweeps + 2) * k * 2.0 ** -52
        r = u.T @ C @ u
        assert np.linalg.norm(r - np.diag(np.diag(r))) <= 2e-14 * np.linalg.norm(C)
