"""The preconditioner far from well-conditioned features of order one: the fp64 pivots over the whole range of exponents,
from states written directly (a diagonal block matrix of small blocks, one scale each), against exact rational
arithmetic; the fp32 blocked path with rank-deficient fits and little damping, and with tiny features."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild

pytestmark = pytest.mark.gpu
TINY = 5e-324  # the damping: the least there is


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


def solve(dev, M, q):
    D = M.shape[0]
    state = torch.zeros(tda.tda_precondition_state_bytes(D, tda.TDA_F64), dtype=torch.uint8, device=dev)
    state[64:64 + 8 * D * D].view(torch.float64).view(D, D).copy_(torch.from_numpy(M).to(dev))
    out = torch.empty((1, D), dtype=torch.float64, device=dev)
    qd = torch.from_numpy(q).to(dev).view(1, D)
    tda.tda_precondition(tda.TDA_PC_FACTOR, 1, D, tda.TDA_F64, state, n_total=1, lambda_abs=TINY)
    tda.tda_precondition(tda.TDA_PC_APPLY, 1, D, tda.TDA_F64, state, q=qd, n_q=1, ld_q=D, qhat=out, ld_qhat=D)
    info = tda.tda_precondition_info(1, D, tda.TDA_F64, state)
    assert info[2] == 0
    return out.cpu().numpy()[0]


# exponents of the scales: all normal ones, around the limits of the fast reciprocal (2^-1000, 2^1000), both ends
SCALES = [np.linspace(-990, 990, 16), np.linspace(-1003, -996, 16), np.linspace(992, 999, 16), np.linspace(999, 1013, 16),
          np.linspace(-1022, -1000, 16)]


@pytest.mark.parametrize("exps", SCALES[:4], ids=str)
def test_fp64_pivot_reciprocal(dev, exps):
    # blocks [p p; p p(1 + d)]: the second pivot is p d, so an error of the first one's reciprocal shows 1 / d times
    # larger. One ulp (2^-52) of the reciprocal and half an ulp of its product with p: 1.5 * 2^-52 / d; outside
    # 2^-1000 .. 2^1000 an ulp of rsqrt and half an ulp of its product, both squared: 3 * 2^-52 / d
    rng = np.random.default_rng(3)
    D, d = 32, 2.0 ** -20
    M, q, ref, tol = np.zeros((D, D)), np.zeros(D, np.float32), np.zeros(D), np.zeros(D)
    for i, e in enumerate(exps):
        p = float(np.ldexp(1.0 + rng.random(), int(e)))
        c = p * (1.0 + d)
        M[2 * i, 2 * i] = M[2 * i + 1, 2 * i] = p
        M[2 * i + 1, 2 * i + 1] = c
        q[2 * i + 1] = 2.0 ** (-100 if e < -850 else 0)
        x = Fraction(float(q[2 * i + 1])) / (Fraction(c) - Fraction(p))
        ref[2 * i], ref[2 * i + 1] = float(-x), float(x)
        tol[2 * i:2 * i + 2] = ((1.5 if 2.0 ** -1000 < p < 2.0 ** 1000 else 3.0) * 2.0 ** -52 / d + 1e-14) * abs(float(x))
    got = solve(dev, M, q)
    assert (np.abs(got - ref) <= tol).all(), (np.abs(got - ref) / tol).max()


@pytest.mark.parametrize("exps", SCALES + [np.linspace(-1065, -1020, 16)], ids=str)
def test_fp64_blocks_of_any_scale(dev, exps):
    # p [1 1/2 1/4; 1/2 1 1/2; 1/4 1/2 1] in rows 2i, 2i + 1 (one diagonal block) and 32 + i (a panel row): condition
    # number 4, so a dozen ulps; of a scale below 2^-1022 the products are rounded to 2^-1074
    D = 48
    B = np.array([[1, .5, .25], [.5, 1, .5], [.25, .5, 1]])
    M, q, ref, tol = np.zeros((D, D)), np.zeros(D, np.float32), np.zeros(D), np.zeros(D)
    for i, e in enumerate(exps):
        r = [2 * i, 2 * i + 1, 32 + i]
        p = float(np.ldexp(1.0, int(e)))
        M[np.ix_(r, r)] = B * p
        qs = 2.0 ** (-100 if e < -850 else 0)
        q[r] = np.array([1, -2, 3], np.float32) * np.float32(qs)
        A = [[Fraction(float(B[a, b] * p)) + (Fraction(TINY) if a == b else 0) for b in range(3)] for a in range(3)]
        y = [Fraction(float(v)) for v in q[r]]
        for a in range(3):  # elimination in exact arithmetic
            for b in range(a + 1, 3):
                f = A[b][a] / A[a][a]
                A[b] = [u - f * v for u, v in zip(A[b], A[a])]
                y[b] -= f * y[a]
        for a in (2, 1, 0):
            y[a] = (y[a] - sum(A[a][b] * y[b] for b in range(a + 1, 3))) / A[a][a]
        ref[r] = [float(v) for v in y]
        tol[r] = (12 * 2.0 ** -52 + 64 * 2.0 ** (-1074 - int(e))) * np.abs(ref[r]).max()
    got = solve(dev, np.tril(M), q)
    assert (np.abs(got - ref) <= tol).all(), (np.abs(got - ref) / tol).max()


# Random-walk rounding of a 256-feature fp32 sum, 16 * 2^-24 of a pivot's scale, is a backward error that the solve
# magnifies by the condition number (largest eigenvalue of the fit over the damping).
@pytest.mark.parametrize("D,n,lam,scale", [(256, 64, 1e-2, 1.0), (256, 64, 1e-4, 1.0), (576, 144, 1e-3, 1.0),
                                           (1024, 256, 1e-3, 1.0), (2048, 512, 1e-3, 1.0), (512, 128, 1e-2, 1e-17)])
def test_fp32_weak_damping(dev, D, n, lam, scale):
    rng = np.random.default_rng(D)
    nl, nq = 2, 20
    w = nl * D
    ph = torch.from_numpy((rng.standard_normal((n, w)) * scale).astype(np.float32)).to(dev)
    q = torch.from_numpy(rng.standard_normal((nq, w)).astype(np.float32)).to(dev)
    state = torch.empty(nl * tda.tda_precondition_state_bytes(D, tda.TDA_F32), dtype=torch.uint8, device=dev)
    out, alone = torch.empty((nq, w), device=dev), torch.empty((nq, w), device=dev)
    args = (nl, D, tda.TDA_F32, state)
    tda.tda_precondition(tda.TDA_PC_RESET, *args)
    tda.tda_precondition(tda.TDA_PC_FIT_ACCUM, *args, phi=ph, n=n, ld_phi=w)
    tda.tda_precondition(tda.TDA_PC_FACTOR_APPLY, *args, n_total=n, lambda_rel_mean_eig=lam, q=q, n_q=nq, ld_q=w,
                         qhat=out, ld_qhat=w)
    tda.tda_precondition(tda.TDA_PC_APPLY, *args, q=q, n_q=nq, ld_q=w, qhat=alone, ld_qhat=w)
    tda.tda_device_status()
    tda.tda_precondition_info(nl, D, tda.TDA_F32, state)
    for l in range(nl):
        x = ph[:, l * D:(l + 1) * D].double()
        F = x.T @ x / n
        damping = lam * F.diagonal().mean()
        cond = float((torch.linalg.eigvalsh(F)[-1] + damping) / damping)
        F.diagonal().add_(damping)
        ref = torch.linalg.solve(F, q[:, l * D:(l + 1) * D].double().T).T
        for o in (out, alone):
            got = o[:, l * D:(l + 1) * D].double()
            assert float((got - ref).norm() / ref.norm()) <= 16 * 2.0 ** -24 * cond
