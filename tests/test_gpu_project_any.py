"""The tensor-core projection at projection sizes that no tile edge matches (k_in != k_out, k below the padded block)
and the shapes where its loops can go wrong: packed short sequences, tokens past a tile, widths past a K chunk, one
example over a cluster, more units than SMs; and the factor output's work split (token scores) at few long examples.
Tolerance: bf16 factors are exact in fp32 and both contractions accumulate in fp32, so the repository's fp32
tolerance (1e-5 relative, per example) holds."""
import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild
from paper_2609_38767_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5
TD = {"f32": tda.TDA_F32, "bf16": tda.TDA_BF16}


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


def factors(n, T, di, do, dtype, stream):
    A = synth.factors(synth.SEED_A, stream, n, T, di, 1.0, 0, 0, dtype, 0.02)
    B = synth.factors(synth.SEED_B, stream, n, T, do, 0.1, 0, 0, dtype, 0.02)
    return A, B


def up(x, dtype, dev):
    if dtype == "bf16":
        return torch.from_numpy(x.view(np.int16)).view(torch.bfloat16).to(dev)
    return torch.from_numpy(x).to(dev)


def rel(x, ref):
    x = np.asarray(x, dtype=np.float64)
    return float(np.linalg.norm(x - ref) / max(np.linalg.norm(ref), 1e-300))


@pytest.mark.parametrize("N,T,di,do,ki,ko", [
    (3, 7, 72, 64, 8, 8), (700, 5, 64, 72, 1, 5), (5, 45, 200, 136, 24, 24), (9, 130, 1000, 2056, 32, 48),
    (2, 300, 64, 128, 16, 64), (3, 64, 136, 64, 100, 72), (160, 200, 72, 64, 48, 33), (1, 520, 64, 64, 64, 8),
    (4, 129, 64, 200, 128, 96)])
def test_tc_projection_any_k(dev, orc, N, T, di, do, ki, ko):
    A, B = factors(N, T, di, do, "bf16", 61)
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    Ad, Bd = up(A, "bf16", dev), up(B, "bf16", dev)
    assert tda.tda_project_engine(L, tda.TDA_BF16, Ad, Bd) == 1
    ld = ki * ko + 3
    phi = torch.full((N, ld), 7.0, device=dev)
    ws = torch.empty(64 << 20, dtype=torch.uint8, device=dev)  # offered, not needed
    tda.tda_project(L, tda.TDA_BF16, Ad, Bd, N, phi, ld, tda.TDA_ROUTE_FACTORED, ws, 64 << 20)
    tda.tda_device_status()
    got = phi.cpu().numpy()
    assert (got[:, ki * ko:] == 7.0).all()
    ref = orc.project(synth.to_f64(A, "bf16"), synth.to_f64(B, "bf16"), ki, ko, 7, 2).reshape(N, -1)
    assert max(rel(got[n, :ki * ko], ref[n]) for n in range(N)) <= TOL


@pytest.mark.parametrize("N,T,di,do,ki,ko", [
    (64, 32, 256, 256, 16, 16), (8, 32, 256, 256, 16, 16),  # packed, one and several examples a tile
    (700, 5, 64, 72, 8, 5), (5, 45, 200, 136, 32, 48), (3, 33, 36, 100, 20, 12), (1, 1, 4, 4, 1, 1),
    (2, 1024, 64, 72, 64, 64), (1, 300, 128, 64, 64, 16),   # clusters sharing an example, uneven tiles
    (160, 200, 72, 64, 64, 64), (9, 130, 1000, 2056, 24, 24), (310, 70, 64, 68, 32, 32), (20, 257, 512, 136, 16, 16),
    (40, 64, 132, 64, 64, 64), (153, 129, 64, 64, 48, 64)])
def test_tc_projection_fp32(dev, orc, N, T, di, do, ki, ko):
    # fp32 factors as three exact bf16 pieces: fp32 rounding of the sums only
    A, B = factors(N, T, di, do, "f32", 63)
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    Ad, Bd = up(A, "f32", dev), up(B, "f32", dev)
    assert tda.tda_project_engine(L, tda.TDA_F32, Ad, Bd) == 1
    ld = ki * ko + 3
    outs = []
    for _ in range(2):
        phi = torch.full((N, ld), 7.0, device=dev)
        tda.tda_project(L, tda.TDA_F32, Ad, Bd, N, phi, ld, tda.TDA_ROUTE_FACTORED)
        tda.tda_device_status()
        outs.append(phi.cpu().numpy())
    np.testing.assert_array_equal(outs[0], outs[1])
    got = outs[0]
    assert (got[:, ki * ko:] == 7.0).all()
    ref = orc.project(A.astype(np.float64), B.astype(np.float64), ki, ko, 7, 2).reshape(N, -1)
    assert max(rel(got[n, :ki * ko], ref[n]) for n in range(N)) <= TOL


def test_tc_projection_fp32_extremes(dev, orc):
    # values whose pieces are subnormal, of the largest exponent, infinite or NaN stay in their example
    N, T, d, k = 4, 3, 64, 16
    A, B = factors(N, T, d, d, "f32", 64)
    A[0] *= np.float32(1e-30)
    B[0] *= np.float32(1e-3)
    A[1] *= np.float32(1e36)
    B[1] *= np.float32(1e-30)
    A[2, 1, 5] = np.inf
    B[3, 0, 7] = np.nan
    L = tda.LayerDesc(d, d, T, k, k, seed=7, layer=2)
    phi = torch.empty((N, k * k), device=dev)
    tda.tda_project(L, tda.TDA_F32, up(A, "f32", dev), up(B, "f32", dev), N, phi, k * k, tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()
    got = phi.cpu().numpy()
    ref = orc.project(A[:2].astype(np.float64), B[:2].astype(np.float64), k, k, 7, 2).reshape(2, -1)
    assert max(rel(got[n], ref[n]) for n in range(2)) <= TOL
    assert np.isinf(got[2]).all() and np.isnan(got[3]).all()


@pytest.mark.parametrize("N,T,di,do,ki,ko", [(3, 64, 256, 512, 16, 16), (5, 33, 64, 100, 12, 7), (4, 32, 256, 256, 16, 16),
                                             (9, 17, 36, 512, 1, 16), (7, 16, 128, 64, 8, 8), (300, 1, 4, 4, 3, 2)])
def test_small_projection_is_the_serial_sum(dev, orc, N, T, di, do, ki, ko):
    # short fp32 jobs of narrow layers: the sums of the definition taken in order in fp32 (features ascending, then
    # fused multiply-adds over the tokens), reproduced bit for bit
    A, B = factors(N, T, di, do, "f32", 65)
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=2)
    phi = torch.empty((N, ki * ko), device=dev)
    tda.tda_project(L, tda.TDA_F32, up(A, "f32", dev), up(B, "f32", dev), N, phi, ki * ko, tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()

    def chain(X, S):
        o = np.zeros(X.shape[:2] + (S.shape[1],), np.float32)
        for c in range(X.shape[2]):
            o += X[:, :, c, None] * S[c].astype(np.float32)
        return o

    a, b = chain(A, orc.proj_entries(7, 2, 0, di, ki)), chain(B, orc.proj_entries(7, 2, 1, do, ko))
    acc = np.zeros((N, ko, ki), np.float32)
    for t in range(T):
        acc = (b[:, t, :, None].astype(np.longdouble) * a[:, t, None, :] + acc).astype(np.float32)
    ref = acc * np.float32(1.0 / (np.sqrt(float(ki)) * np.sqrt(float(ko))))
    np.testing.assert_array_equal(phi.cpu().numpy(), ref.reshape(N, -1))


@pytest.mark.parametrize("N,T,di,do,ki,ko,nq,beta", [
    (1, 1024, 64, 72, 64, 64, 3, 0.0), (16, 300, 136, 64, 32, 32, 2, 0.0), (200, 9, 64, 64, 16, 16, 5, 0.0),
    (3, 130, 64, 64, 64, 64, 1, 0.0), (160, 130, 64, 64, 64, 64, 37, 0.5),  # more token tiles than SMs, ragged stage
    (2, 77, 64, 64, 20, 32, 9, 0.0), (3, 129, 72, 64, 48, 16, 17, 1.0), (2, 64, 64, 64, 4, 64, 5, 0.0)])
def test_token_scores_work_split(dev, orc, N, T, di, do, ki, ko, nq, beta):
    A, B = factors(N, T, di, do, "bf16", 62)
    L = tda.LayerDesc(di, do, T, ki, ko, seed=7, layer=1)
    R = np.random.default_rng(N).standard_normal((nq, ki * ko)).astype(np.float32)
    wsb = tda.tda_token_scores_workspace_size(L) * N + (4 << 20)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    out = torch.full((nq, N * T), 0.25, device=dev)
    tda.tda_token_scores(L, tda.TDA_BF16, up(A, "bf16", dev), up(B, "bf16", dev), N, torch.from_numpy(R).to(dev), nq,
                         ki * ko, out, N * T, beta, ws, wsb)
    tda.tda_device_status()
    Si = orc.proj_entries(7, 1, 0, di, ki).astype(np.float64) / np.sqrt(ki)
    So = orc.proj_entries(7, 1, 1, do, ko).astype(np.float64) / np.sqrt(ko)
    a, b = synth.to_f64(A, "bf16") @ Si, synth.to_f64(B, "bf16") @ So
    ref = np.stack([((a @ R[j].reshape(ko, ki).T.astype(np.float64)) * b).sum(2).ravel() for j in range(nq)])
    assert rel(out.cpu().numpy() - 0.25 * beta, ref) <= TOL
