"""Values that are not finite stay visible, and stay in their token, query or example, in the kernels that cut fp32
values into pieces for the tensor cores."""
import numpy as np
import pytest
import torch

import paper_2609_38767_gb300 as tda
from paper_2609_38767_gb300 import build as tbuild
from paper_2609_38767_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    tbuild.build()
    tda.load()
    return torch.device("cuda:0")


def up(x, dev):
    return torch.from_numpy(x.view(np.int16)).view(torch.bfloat16).to(dev)


@pytest.mark.parametrize("ki,ko", [(20, 32), (32, 16), (32, 64), (64, 64), (48, 32)])
def test_token_scores_keep_nan(dev, ki, ko):
    N, T, d, nq = 2, 150, 64, 5
    A = up(synth.factors(synth.SEED_A, 71, N, T, d, 1.0, 0, 0, "bf16", 0.02), dev)
    B = up(synth.factors(synth.SEED_B, 71, N, T, d, 0.1, 0, 0, "bf16", 0.02), dev)
    L = tda.LayerDesc(d, d, T, ki, ko, seed=7, layer=1)
    R = torch.from_numpy(np.random.default_rng(ki).standard_normal((nq, ki * ko)).astype(np.float32)).to(dev)
    zero = torch.zeros(1, device=dev)
    computed = (zero / zero)[0]  # the NaN that arithmetic on the device produces: every mantissa bit set
    assert int(computed.view(1).view(torch.int32)) & 0x7FFFFFFF == 0x7FFFFFFF
    wsb = tda.tda_token_scores_workspace_size(L) * N + (4 << 20)
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    outs = []
    for bad in (False, True):
        if bad:
            A[1, 7, 3] = float("nan")  # its projection is computed
            R[2, ki + 1] = computed
        out = torch.empty((nq, N, T), device=dev)
        tda.tda_token_scores(L, tda.TDA_BF16, A, B, N, R, nq, ki * ko, out, N * T, 0.0, ws, wsb)
        tda.tda_device_status()
        outs.append(out.cpu().numpy())
    lost = np.zeros((nq, N, T), bool)
    lost[:, 1, 7] = lost[2] = True
    assert np.isnan(outs[1][lost]).all()
    np.testing.assert_array_equal(outs[1][~lost], outs[0][~lost])


@pytest.mark.parametrize("T,k", [(3, 32), (40, 64), (130, 24)])
def test_fp32_pieces_extremes(dev, orc, T, k):
    # k above 16: the kernel that cuts fp32 factors into three bf16 pieces, packed and whole tiles. Tiny values, values
    # of the largest exponent, an infinity and both NaN patterns stay in their example
    N, d = 5, 64
    A, B = (synth.factors(seed, 64, N, T, d, sc, 0, 0, "f32", 0.02) for seed, sc in ((synth.SEED_A, 1.0), (synth.SEED_B, 0.1)))
    A[0] *= np.float32(1e-30)
    B[0] *= np.float32(1e-3)
    A[1] *= np.float32(1e36)
    B[1] *= np.float32(1e-30)
    A[2, 1, 5] = np.inf
    B[3, 0, 7] = np.nan
    A[4, 2, 9] = np.array(0x7FFFFFFF, np.uint32).view(np.float32)
    L = tda.LayerDesc(d, d, T, k, k, seed=7, layer=2)
    phi = torch.empty((N, k * k), device=dev)
    tda.tda_project(L, tda.TDA_F32, torch.from_numpy(A).to(dev), torch.from_numpy(B).to(dev), N, phi, k * k,
                    tda.TDA_ROUTE_FACTORED)
    tda.tda_device_status()
    got = phi.cpu().numpy().astype(np.float64)
    ref = orc.project(A[:2].astype(np.float64), B[:2].astype(np.float64), k, k, 7, 2).reshape(2, -1)
    assert max(np.linalg.norm(got[n] - ref[n]) / np.linalg.norm(ref[n]) for n in range(2)) <= 1e-5
    assert not np.isfinite(got[2]).any() and np.isnan(got[3:]).all()
