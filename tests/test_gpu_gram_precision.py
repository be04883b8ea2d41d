"""Accuracy of the tensor-core Gram kernel (Eq. 4, bf16 factors) at short sequences, where its blocks weigh most:
against fp32 sums taken in order with round-to-nearest (emulated here), and against a bound from its longest blocks.

Bound: a block has at most 256 features, 16 additions of the tensor pipe that truncate by at most one ulp (2^-23) of
the running sum: 1.9e-6 on X and on Y. Everything after that rounds to nearest, less than 3e-7 more. A running sum is
at most the sum of its terms' absolute values, so every output is within 4.2e-6 of sum_ts X_ts Y_ts with X and Y the
token Grams of the factors' absolute values."""
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


def chain(q, i):
    """Token Grams of fp32 factors, the features added in order (products of bf16 values are exact)."""
    g = np.zeros((len(q), len(i), q.shape[1], i.shape[1]), np.float32)
    for c in range(q.shape[2]):
        g += q[:, None, :, None, c] * i[None, :, None, :, c]
    return g


@pytest.mark.parametrize("T,di,do", [(3, 256, 256), (5, 2048, 2048), (13, 2048, 2048), (7, 512, 4096)])
def test_gram_of_short_sequences(dev, T, di, do):
    nq, nt = 4, 60
    rng = np.random.default_rng(T)
    f = [torch.from_numpy(rng.standard_normal(s).astype(np.float32)).bfloat16()
         for s in ((nq, T, di), (nq, T, do), (nt, T, di), (nt, T, do))]
    d = [x.to(dev) for x in f]
    L = tda.LayerDesc(di, do, T, 1, 1)
    assert tda.tda_similarity_gram_engine(L, tda.TDA_BF16, *d) == 1
    S = torch.empty((nq, nt), device=dev)
    tda.tda_similarity_exact(L, tda.TDA_BF16, d[0], d[1], nq, d[2], d[3], nt, S, nt, 0.0, tda.TDA_ROUTE_GRAM)
    tda.tda_device_status()
    got = S.cpu().numpy().astype(np.float64)
    f32 = [x.float().numpy() for x in f]
    f64 = [x.astype(np.float64) for x in f32]
    gram = lambda q, i: np.einsum("qtd,isd->qits", q, i, optimize=True)  # noqa: E731
    ref = (gram(f64[0], f64[2]) * gram(f64[1], f64[3])).sum((2, 3))
    bound = (gram(abs(f64[0]), abs(f64[2])) * gram(abs(f64[1]), abs(f64[3]))).sum((2, 3))
    assert (np.abs(got - ref) <= 4.2e-6 * bound).all()
    X, Y, s = chain(f32[0], f32[2]), chain(f32[1], f32[3]), np.zeros((nq, nt), np.float32)
    for t in range(T):
        for u in range(T):
            s = (X[:, :, t, u].astype(np.float64) * Y[:, :, t, u] + s).astype(np.float32)
    assert np.linalg.norm(got - ref) <= np.linalg.norm(s - ref)


@pytest.mark.parametrize("nq,nt,T,di,do", [(1, 1, 1, 64, 64), (1, 8, 3, 64, 72), (4, 16, 5, 128, 128), (4, 16, 5, 256, 256),
                                           (17, 18, 2, 64, 40), (19, 17, 2, 64, 40), (1, 100, 7, 128, 136), (2, 3, 15, 64, 64),
                                           (2, 3, 16, 64, 64), (1, 304, 4, 8, 8), (1, 305, 4, 8, 8)])
def test_few_short_pairs(dev, nq, nt, T, di, do):
    # either side of the line between the CUDA-core and the tensor-core kernel; an accumulated score, a padded row
    rng = np.random.default_rng(nq + T)
    f = [torch.from_numpy(rng.standard_normal(s).astype(np.float32)).bfloat16()
         for s in ((nq, T, di), (nq, T, do), (nt, T, di), (nt, T, do))]
    d = [x.to(dev) for x in f]
    L = tda.LayerDesc(di, do, T, 1, 1)
    S, n = torch.full((nq, nt + 1), 0.5, device=dev), torch.empty(nt, device=dev)
    tda.tda_similarity_exact(L, tda.TDA_BF16, d[0], d[1], nq, d[2], d[3], nt, S, nt + 1, 2.0, tda.TDA_ROUTE_GRAM)
    tda.tda_norms(tda.TDA_OP_NORM_EXACT, L, tda.TDA_BF16, d[2], d[3], nt, n, tda.TDA_ROUTE_GRAM)
    tda.tda_device_status()
    f = [x.double().numpy() for x in f]
    gram = lambda q, i: np.einsum("qtd,isd->qits", q, i, optimize=True)  # noqa: E731
    ref = (gram(f[0], f[2]) * gram(f[1], f[3])).sum((2, 3))
    bound = (gram(abs(f[0]), abs(f[2])) * gram(abs(f[1]), abs(f[3]))).sum((2, 3))
    got = S.cpu().numpy().astype(np.float64)
    assert (np.abs(got[:, :nt] - 1.0 - ref) <= 4.2e-6 * (bound + 1.0)).all() and (got[:, nt] == 0.5).all()
    for i in range(nt):
        X, Y = f[2][i] @ f[2][i].T, f[3][i] @ f[3][i].T
        assert abs(float(n[i]) - (X * Y).sum()) <= 4.2e-6 * ((abs(f[2][i]) @ abs(f[2][i]).T) * (abs(f[3][i]) @ abs(f[3][i]).T)).sum()
