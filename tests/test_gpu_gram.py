"""The tensor-core Gram kernel (Eq. 4, bf16 factors) at the token counts where its tiles can go wrong: examples
packed into 128-row and 256-column tiles whose edges no T divides, examples straddling the two column halves of a
tile, tile pairs with rows past T, one to three tokens, units that wrap the persistent grid; similarities and norms.

Tolerance: bf16 products are exact in fp32; a 128-feature block takes at most 8 truncating additions of the tensor
pipe (at most one ulp of the running sum, 2^-23, each: 9.6e-7), on X and on Y; everything after that rounds to
nearest, a few ulps more. A running sum is at most the sum of its terms' absolute values, so every output is within
2.5e-6 of sum_ts X_ts Y_ts with X and Y the token Grams of the factors' absolute values."""
import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild
from paper_2609_38767_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 2.5e-6


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


def factors(n, T, di, do, stream):
    A = synth.factors(synth.SEED_A, stream, n, T, di, 1.0, 0, 0, "bf16", 0.02)
    B = synth.factors(synth.SEED_B, stream, n, T, do, 0.1, 0, 0, "bf16", 0.02)
    return A, B


def up(x, dev):
    return torch.from_numpy(x.view(np.int16)).view(torch.bfloat16).to(dev)


def scale(Aq, Bq, At, Bt):
    """sum_ts X_ts Y_ts of every (query, train) pair, for the factors' absolute values and for the factors."""
    gram = lambda q, i: np.tensordot(q, i, (2, 2)).transpose(0, 2, 1, 3)  # noqa: E731
    return [(gram(f(Aq), f(At)) * gram(f(Bq), f(Bt))).sum((2, 3)) for f in (np.abs, np.asarray)]


@pytest.mark.parametrize("nq,nt,T,di,do", [
    (5, 300, 1, 64, 40), (7, 140, 2, 136, 64), (9, 100, 3, 72, 64), (30, 61, 5, 200, 136), (5, 12, 21, 520, 1032),
    (70, 131, 50, 64, 72), (5, 9, 63, 64, 64), (6, 9, 65, 128, 136), (20, 31, 100, 64, 64), (3, 5, 127, 64, 200),
    (3, 5, 129, 72, 64), (2, 3, 200, 264, 128), (2, 3, 257, 64, 72), (13, 14, 300, 64, 64),
    # pairs of CTAs: odd and even query tiles, one example a tile, ragged last train tile
    (5, 9, 50, 1544, 1608), (3, 7, 128, 2048, 1032), (140, 70, 1, 1600, 1536), (17, 33, 13, 3072, 64),
    (4, 11, 64, 64, 3080)])
def test_gram_any_token_count(dev, orc, nq, nt, T, di, do):
    Aq, Bq = factors(nq, T, di, do, 51)
    At, Bt = factors(nt, T, di, do, 52)
    L = tda.LayerDesc(di, do, T, 1, 1)
    d = [up(x, dev) for x in (Aq, Bq, At, Bt)]
    assert tda.tda_similarity_gram_engine(L, tda.TDA_BF16, *d) == 1
    S = torch.full((nq, nt + 1), 0.5, device=dev)
    tda.tda_similarity_exact(L, tda.TDA_BF16, d[0], d[1], nq, d[2], d[3], nt, S, nt + 1, 0.0, tda.TDA_ROUTE_GRAM)
    nrm = torch.empty(nt, device=dev)
    tda.tda_norms(tda.TDA_OP_NORM_EXACT, L, tda.TDA_BF16, d[2], d[3], nt, nrm, tda.TDA_ROUTE_GRAM)
    tda.tda_device_status()
    f = [synth.to_f64(x, "bf16") for x in (Aq, Bq, At, Bt)]
    sc, ref = scale(*f)
    np.testing.assert_allclose(ref, orc.similarity(*f), rtol=1e-9, atol=1e-9 * np.abs(ref).max())
    got = S.cpu().numpy().astype(np.float64)
    assert (np.abs(got[:, :nt] - ref) <= TOL * sc + 1e-30).all()
    assert (got[:, nt] == 0.5).all()
    for i in range(nt):
        sn, rn = scale(f[2][i:i + 1], f[3][i:i + 1], f[2][i:i + 1], f[3][i:i + 1])
        assert abs(float(nrm[i]) - rn[0, 0]) <= TOL * sn[0, 0]


@pytest.mark.parametrize("T", [21, 50, 130])
def test_gram_infinity_stays_in_its_example(dev, T):
    nq, nt, d = 4, 7, 64
    Aq, Bq = (up(x, dev) for x in factors(nq, T, d, d, 53))
    At, Bt = (up(x, dev) for x in factors(nt, T, d, d, 54))
    L = tda.LayerDesc(d, d, T, 1, 1)
    out = []
    for bad in (False, True):
        if bad:
            At[3, T - 1, 5] = float("inf")
            Aq[1, 0, 7] = float("nan")
        S, n = torch.empty((nq, nt), device=dev), torch.empty(nt, device=dev)
        tda.tda_similarity_exact(L, tda.TDA_BF16, Aq, Bq, nq, At, Bt, nt, S, nt, 0.0, tda.TDA_ROUTE_GRAM)
        tda.tda_norms(tda.TDA_OP_NORM_EXACT, L, tda.TDA_BF16, At, Bt, nt, n, tda.TDA_ROUTE_GRAM)
        tda.tda_device_status()
        out.append((S.cpu().numpy(), n.cpu().numpy()))
    (S0, n0), (S1, n1) = out
    clean = np.ones((nq, nt), bool)
    clean[:, 3] = clean[1] = False
    np.testing.assert_array_equal(S1[clean], S0[clean])
    assert not np.isfinite(S1[~clean]).any()
    np.testing.assert_array_equal(np.delete(n1, 3), np.delete(n0, 3))
    assert not np.isfinite(n1[3])
