"""The latency-bound small kernels at the sizes where they can go wrong: the fp64 preconditioner (ragged last blocks,
one to several CTAs of panel rows, tile sizes, pivots far from one), fp64 scores of few rows, and the top-k selection
(row lengths around every kernel's limit, ties that need the index digits, non-finite scores)."""
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


# fp64 state: backward error of a Cholesky solve is a few D eps of the condition number; with damping of a tenth of
# the mean eigenvalue and more rows than features it is below 100, so 1e-11 (D = 600: 600 * 2.2e-16 * 100) holds.
@pytest.mark.parametrize("D,nl,nq,scale", [(1, 1, 1, 1.0), (31, 2, 3, 1.0), (32, 1, 9, 1.0), (33, 1, 160, 1.0),
                                           (144, 2, 5, 1.0), (256, 1, 8, 1e-17), (256, 1, 40, 3e17), (600, 1, 2, 1.0)])
def test_fp64_preconditioner(dev, D, nl, nq, scale):
    rng = np.random.default_rng(D + nq)
    n = 2 * D + 5
    phi = (rng.standard_normal((n, nl * D)) * scale).astype(np.float32)
    q = rng.standard_normal((nq, nl * D)).astype(np.float32)
    per = tda.tda_precondition_state_bytes(D, tda.TDA_F64)
    state = torch.empty(nl * per, dtype=torch.uint8, device=dev)
    ph, qd = torch.from_numpy(phi).to(dev), torch.from_numpy(q).to(dev)
    out = torch.empty((nq, nl * D), dtype=torch.float64, device=dev)
    args = (nl, D, tda.TDA_F64, state)
    tda.tda_precondition(tda.TDA_PC_RESET, *args)
    for a, b in ((0, n // 3), (n // 3, n)):
        tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph[a:], n=b - a, ld_phi=nl * D)
    tda.tda_precondition(tda.TDA_PC_FACTOR, *args, n_total=n, lambda_rel_mean_eig=0.1)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=qd, n_q=nq, ld_q=nl * D, qhat=out, ld_qhat=nl * D)
    info = tda.tda_precondition_info(nl, D, tda.TDA_F64, state)
    for l in range(nl):
        x = phi[:, l * D:(l + 1) * D].astype(np.float64)
        F = x.T @ x / n
        lam = 0.1 * np.trace(F) / D
        assert abs(info[4 * l] / lam - 1) < 1e-12 and info[4 * l + 2] == 0
        ref = np.linalg.solve(F + lam * np.eye(D), q[:, l * D:(l + 1) * D].T.astype(np.float64)).T
        got = out[:, l * D:(l + 1) * D].cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-11 * np.linalg.norm(ref)


@pytest.mark.parametrize("D,bad", [(5, 0), (40, 31), (40, 33), (100, 70)])
def test_fp64_failed_pivot_is_reported(dev, D, bad):
    state = torch.empty(tda.tda_precondition_state_bytes(D, tda.TDA_F64), dtype=torch.uint8, device=dev)
    tda.tda_precondition(tda.TDA_PC_RESET, 1, D, tda.TDA_F64, state)
    m = state[64:64 + 8 * D * D].view(torch.float64).view(D, D)
    m.copy_(torch.eye(D, dtype=torch.float64, device=dev))
    m[bad, bad] = -50.0
    out = torch.zeros((2, D), dtype=torch.float64, device=dev)
    tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, 1, D, tda.TDA_F64, state, n_total=1, lambda_abs=1e-3,
                         q=torch.ones((2, D), device=dev), n_q=2, ld_q=D, qhat=out, ld_qhat=D)
    with pytest.raises(tda.TdaError) as e:
        tda.tda_precondition_info(1, D, tda.TDA_F64, state)
    assert e.value.status == tda.TDA_ERR_NOT_SPD and f"pivot {bad + 1}" in str(e.value)
    assert torch.isnan(out).all()


@pytest.mark.parametrize("nq,nt,D,beta", [(1, 1, 1, 0.0), (8, 64, 256, 0.0), (3, 77, 45, 1.0), (33, 1100, 40, 0.5),
                                          (64, 1300, 31, 0.0)])
def test_fp64_scores(dev, nq, nt, D, beta):
    rng = np.random.default_rng(nt)
    Q, P = rng.standard_normal((nq, D)), rng.standard_normal((nt, D)).astype(np.float32)
    S = torch.full((nq, nt + 2), 2.0, device=dev)
    tda.tda_score(torch.from_numpy(Q).to(dev), tda.TDA_F64, nq, D, torch.from_numpy(P).to(dev), nt, D, D, S, nt + 2,
                  beta)
    got = S.cpu().numpy()
    ref = Q @ P.T.astype(np.float64) + 2.0 * beta
    # one rounding to fp32 (half an ulp) of a sum that fp64 holds to far below it
    assert (np.abs(got[:, :nt] - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-12).all()
    assert (got[:, nt:] == 2.0).all()


@pytest.mark.parametrize("nt", [1, 31, 512, 513, 2048, 2049, 8192, 8193, 16384, 16385, 40000])
@pytest.mark.parametrize("values", ["normal", "ties", "equal", "odd"])
def test_topk_selection(dev, orc, nt, values):
    rng = np.random.default_rng(nt)
    nq = 3
    if values == "normal":
        S = rng.standard_normal((nq, nt))
    elif values == "ties":
        S = rng.integers(-3, 4, (nq, nt)) / 2.0
    elif values == "equal":
        S = np.full((nq, nt), -1.5)
    else:
        S = rng.choice([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-40, -1e-40, 3.4e38, 1.0], (nq, nt))
    S = S.astype(np.float32)
    Sd = torch.zeros((nq, nt + 5), device=dev)
    Sd[:, :nt] = torch.from_numpy(S).to(dev)
    for k in sorted({1, min(nt, 100), min(nt, 257), min(nt, 1024)}):
        idx = torch.full((nq, k), -7, dtype=torch.int32, device=dev)
        val = torch.empty((nq, k), device=dev)
        tda.tda_topk(Sd, nq, nt, nt + 5, k, idx, val)
        oi, _ = orc.topk(S.astype(np.float64), k)
        np.testing.assert_array_equal(idx.cpu().numpy(), oi)
        np.testing.assert_array_equal(val.cpu().numpy().view(np.uint32),
                                      np.take_along_axis(S, oi.astype(np.int64), 1).view(np.uint32))


# fp32 blocked path: rounding of a 3xTF32 / fp32 Cholesky solve, a few D eps of the condition number (below 50 with
# damping of a tenth of the mean eigenvalue and four rows a feature): 2e-5 holds with room at D = 2432.
@pytest.mark.parametrize("D,nl,nq,ld", [(2048, 1, 1, 0), (2176, 2, 17, 4), (2304, 1, 130, 0), (2432, 3, 300, 8)])
def test_blocked_panels(dev, D, nl, nq, ld):
    # panels of 256 columns, a last one of 128 or 256; few and many rows per solve launch; padded rows
    rng = np.random.default_rng(D)
    n, w = 4 * D, nl * D
    ph = torch.from_numpy(rng.standard_normal((n, w)).astype(np.float32)).to(dev)
    q = torch.from_numpy(rng.standard_normal((nq, w + ld)).astype(np.float32)).to(dev)
    state = torch.empty(nl * tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
    out = torch.full((nq, w + ld), 3.0, device=dev)
    args = (nl, D, tda.TDA_F32, state)
    tda.tda_precondition(tda.TDA_PC_RESET, *args)
    tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph, n=n, ld_phi=w)
    tda.tda_precondition(tda.TDA_PC_FACTOR, *args, n_total=n, lambda_rel_mean_eig=0.1)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=w + ld, qhat=out, ld_qhat=w + ld)
    # the other substitution path, from the same state: rows that are not 16-byte aligned
    out2 = torch.empty(nq * (w + 1) + 1, device=dev)[1:].view(nq, w + 1)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=w + ld, qhat=out2, ld_qhat=w + 1)
    tda.tda_device_status()
    tda.tda_precondition_info(nl, D, tda.TDA_F32, state)
    for l in range(nl):
        x = ph[:, l * D:(l + 1) * D].double()
        F = x.T @ x / n
        F.diagonal().add_(0.1 * F.diagonal().mean())
        ref = torch.linalg.solve(F, q[:, l * D:(l + 1) * D].double().T).T
        for o in (out, out2):
            got = o[:, l * D:(l + 1) * D].double()
            assert float((got - ref).norm() / ref.norm()) <= 2e-5
    assert (out[:, w:] == 3.0).all()


@pytest.mark.parametrize("bad", [0, 130, 255, 256, 2047])
def test_blocked_failed_pivot(dev, bad):
    D = 2048
    state = torch.empty(tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
    tda.tda_precondition(tda.TDA_PC_RESET, 1, D, tda.TDA_F32, state)
    m = state[64:64 + 4 * D * D].view(torch.float32).view(D, D)
    m.copy_(torch.eye(D, device=dev))
    m[bad, bad] = -50.0
    out = torch.zeros((2, D), device=dev)
    tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, 1, D, tda.TDA_F32, state, n_total=1, lambda_abs=1e-3,
                         q=torch.ones((2, D), device=dev), n_q=2, ld_q=D, qhat=out, ld_qhat=D)
    with pytest.raises(tda.TdaError) as e:
        tda.tda_precondition_info(1, D, tda.TDA_F32, state)
    assert e.value.status == tda.TDA_ERR_NOT_SPD and f"pivot {bad + 1}" in str(e.value)
    assert torch.isnan(out).all()


# as test_blocked_panels (condition number, rows a feature); D below 2048: FACTOR_APPLY runs the panels, APPLY by
# itself the row-by-row substitution on the state that they leave
@pytest.mark.parametrize("D,nl,nq,ld", [(256, 3, 5, 0), (320, 2, 40, 0), (384, 1, 33, 4), (448, 1, 9, 0), (576, 3, 65, 4),
                                         (1600, 1, 70, 0), (2112, 1, 20, 0), (1024, 2, 1, 0), (1152, 1, 130, 4), (1536, 3, 300, 0), (2176, 1, 40, 8)])
def test_blocked_factor_apply(dev, D, nl, nq, ld):
    rng = np.random.default_rng(D + 1)
    n, w = 4 * D, nl * D
    ph = torch.from_numpy(rng.standard_normal((n, w)).astype(np.float32)).to(dev)
    q = torch.from_numpy(rng.standard_normal((nq, w + ld)).astype(np.float32)).to(dev)
    state = torch.empty(nl * tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
    out, alone, inplace = torch.full((nq, w + ld), 3.0, device=dev), torch.empty((nq, w), device=dev), q.clone()
    args = (nl, D, tda.TDA_F32, state)
    for o in (out, inplace):
        tda.tda_precondition(tda.TDA_PC_RESET, *args)
        tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph, n=n, ld_phi=w)
        tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, *args, n_total=n, lambda_rel_mean_eig=0.1,
                             q=o if o is inplace else q, n_q=nq, ld_q=w + ld, qhat=o, ld_qhat=w + ld)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=w + ld, qhat=alone, ld_qhat=w)
    tda.tda_device_status()
    tda.tda_precondition_info(nl, D, tda.TDA_F32, state)
    for l in range(nl):
        x = ph[:, l * D:(l + 1) * D].double()
        F = x.T @ x / n
        F.diagonal().add_(0.1 * F.diagonal().mean())
        ref = torch.linalg.solve(F, q[:, l * D:(l + 1) * D].double().T).T
        for o in (out, inplace, alone):
            got = o[:, l * D:(l + 1) * D].double()
            assert float((got - ref).norm() / ref.norm()) <= 2e-5
    assert (out[:, w:] == 3.0).all() and torch.equal(inplace[:, :w], out[:, :w])


def test_blocked_state_without_64_column_inverses(dev):
    # a factored state from before the 64 x 64 inverses were kept: no mark in the header, nothing of use right of
    # the diagonal inside the 64-column blocks
    D, nq = 2048, 20
    rng = np.random.default_rng(9)
    ph = torch.from_numpy(rng.standard_normal((4 * D, D)).astype(np.float32)).to(dev)
    q = torch.from_numpy(rng.standard_normal((nq, D)).astype(np.float32)).to(dev)
    state = torch.empty(tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
    args = (1, D, tda.TDA_F32, state)
    tda.tda_precondition(tda.TDA_PC_RESET, *args)
    tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph, n=4 * D, ld_phi=D)
    tda.tda_precondition(tda.TDA_PC_FACTOR, *args, n_total=4 * D, lambda_rel_mean_eig=0.1)
    new, old = torch.empty((nq, D), device=dev), torch.empty((nq, D), device=dev)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=D, qhat=new, ld_qhat=D)
    state[32:40] = 0
    m = state[64:64 + 4 * D * D].view(torch.float32).view(D // 64, 64, D // 64, 64)
    up = torch.triu(torch.ones(64, 64, dtype=torch.bool, device=dev), 1)
    for b in range(D // 64):
        m[b, :, b, :][up] = float("nan")
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=D, qhat=old, ld_qhat=D)
    tda.tda_device_status()
    assert float((new - old).norm() / new.norm()) <= 2e-5


def test_factor_apply_row_strides_past_the_copies(dev):
    # one row whose stride no 2-D copy takes: solved by the cluster kernel, as every row of this width once was
    D = 256
    rng = np.random.default_rng(4)
    ph = torch.from_numpy(rng.standard_normal((4 * D, D)).astype(np.float32)).to(dev)
    q = torch.from_numpy(rng.standard_normal((1, D)).astype(np.float32)).to(dev)
    outs = []
    for ld in (D, 1 << 29):
        state = torch.empty(tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
        args = (1, D, tda.TDA_F32, state)
        out = torch.empty((1, D), device=dev)
        tda.tda_precondition(tda.TDA_PC_RESET, *args)
        tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph, n=4 * D, ld_phi=D)
        tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, *args, n_total=4 * D, lambda_rel_mean_eig=0.1, q=q, n_q=1, ld_q=ld,
                             qhat=out, ld_qhat=ld)
        outs.append(out)
    tda.tda_device_status()
    assert float((outs[0] - outs[1]).norm() / outs[0].norm()) <= 4e-5
