"""Accuracy of the tensor-core projection of wide layers whose features differ widely in size (cubed normal values),
where a long truncating sum of the tensor pipe drifts towards zero.

Tolerance: a sum of at most 256 features takes 16 additions that truncate, each by at most one ulp (2^-23) of the
running sum; every later addition rounds to nearest, 64 to 128 of them per entry here (a random walk of half ulps:
at most 5e-7). Both sides of the projection: 2 * 16 * 2^-23 + 2 * 5e-7 = 4.8e-6 of an example's features."""
import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild

pytestmark = pytest.mark.gpu
TOL = 4.8e-6


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


def check(dev, orc, dtype, N, T, di, do, ki, ko):
    rng = np.random.default_rng(di + ko)
    td, code = (torch.bfloat16, tda.TDA_BF16) if dtype == "bf16" else (torch.float32, tda.TDA_F32)
    A, B = (torch.from_numpy((rng.standard_normal((N, T, d)) ** 3).astype(np.float32)).to(td) for d in (di, do))
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    phi = torch.empty((N, ki * ko), device=dev)
    Ad, Bd = A.to(dev), B.to(dev)
    assert tda.tda_project_engine(L, code, Ad, Bd) == 1
    tda.tda_project(L, code, Ad, Bd, N, phi, ki * ko, tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()
    ref = orc.project(A.double().numpy(), B.double().numpy(), ki, ko, 7, 2).reshape(N, -1)
    got = phi.cpu().numpy().astype(np.float64)
    assert max(np.linalg.norm(got[n] - ref[n]) / np.linalg.norm(ref[n]) for n in range(N)) <= TOL


@pytest.mark.parametrize("dtype,N,T,di,do,ki,ko", [
    ("f32", 2, 40, 16384, 64, 32, 32), ("f32", 3, 33, 64, 16388, 64, 64), ("f32", 1, 150, 16384, 300, 16, 12),
    ("bf16", 2, 40, 16384, 64, 32, 48), ("bf16", 1, 130, 72, 16392, 8, 24)])
def test_wide_layers_of_uneven_features(dev, orc, dtype, N, T, di, do, ki, ko):
    check(dev, orc, dtype, N, T, di, do, ki, ko)


@pytest.mark.parametrize("N,T,di,do,ki,ko", [(2, 40, 16384, 64, 100, 72), (3, 200, 64, 16392, 72, 128),
                                             (160, 130, 1000, 72, 65, 3), (1, 520, 72, 64, 128, 96)])
def test_wide_layers_of_uneven_features_k_above_64(dev, orc, N, T, di, do, ki, ko):
    # groups that end with a side, several tiles an example, clusters and whole examples a CTA
    check(dev, orc, "bf16", N, T, di, do, ki, ko)


@pytest.mark.parametrize("N,T,di,do,ki,ko", [(4000, 5, 64, 72, 8, 5), (64, 32, 576, 256, 16, 16), (8, 32, 576, 256, 16, 16),
                                             (1, 1, 516, 4, 1, 1), (300, 64, 64, 64, 12, 16)])
def test_fp32_packed_tiles_of_few_columns(dev, orc, N, T, di, do, ki, ko):
    # fp32 factors at k up to 16 past the limits of the CUDA-core kernel for short jobs (16384 tokens, 512 features)
    rng = np.random.default_rng(N)
    A, B = (rng.standard_normal((N, T, d)).astype(np.float32) for d in (di, do))
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    phi = torch.full((N, ki * ko + 1), 7.0, device=dev)
    tda.tda_project(L, tda.TDA_F32, torch.from_numpy(A).to(dev), torch.from_numpy(B).to(dev), N, phi, ki * ko + 1,
                    tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()
    ref = orc.project(A.astype(np.float64), B.astype(np.float64), ki, ko, 7, 2).reshape(N, -1)
    got = phi.cpu().numpy().astype(np.float64)
    assert (got[:, ki * ko] == 7.0).all()
    assert max(np.linalg.norm(got[n, :ki * ko] - ref[n]) / np.linalg.norm(ref[n]) for n in range(N)) <= TOL


@pytest.mark.parametrize("N,T,di,do,ki,ko", [(1, 1, 64, 64, 100, 100), (2, 8, 128, 128, 100, 90), (200, 8, 128, 136, 128, 72),
                                             (16, 17, 256, 256, 96, 100), (16, 16, 256, 256, 96, 100), (300, 64, 64, 72, 65, 1),
                                             (3, 128, 8, 8, 127, 128), (5, 33, 520, 8, 70, 128)])
def test_short_jobs_of_k_above_64(dev, orc, N, T, di, do, ki, ko):
    # either side of the line between the general and the tensor-core kernel: one result, padding columns untouched
    rng = np.random.default_rng(N + T)
    A, B = (torch.from_numpy(rng.standard_normal((N, T, d)).astype(np.float32)).bfloat16() for d in (di, do))
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    phi = torch.full((N, ki * ko + 1), 7.0, device=dev)
    tda.tda_project(L, tda.TDA_BF16, A.to(dev), B.to(dev), N, phi, ki * ko + 1, tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()
    ref = orc.project(A.double().numpy(), B.double().numpy(), ki, ko, 7, 2).reshape(N, -1)
    got = phi.cpu().numpy().astype(np.float64)
    assert (got[:, ki * ko] == 7.0).all()
    assert max(np.linalg.norm(got[n, :ki * ko] - ref[n]) / np.linalg.norm(ref[n]) for n in range(N)) <= TOL
