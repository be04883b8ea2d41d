"""Accuracy of tensor-core scores of few features. A chunk of 32 features takes 12 additions of the tensor pipe, each of
which loses half an ulp of the running sum (2^-24) or less on average: 7.2e-7; what the two halves of the operands leave
out (2^-22 of single products, random) and the later additions, which round to nearest, add less than 1e-7."""
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


@pytest.mark.parametrize("nq,nt", [(11, 211), (64, 1500), (130, 20000)])
@pytest.mark.parametrize("D,beta", [(64, 0.0), (100, 1.0), (192, 0.0), (256, 1.0), (384, 0.0)])
def test_scores_of_few_features(dev, nq, nt, D, beta):
    g = torch.Generator(device="cuda")
    g.manual_seed(D + nq)
    Q, P = torch.randn((nq, D), generator=g, device=dev), torch.randn((nt, D), generator=g, device=dev)
    assert tda.tda_score_engine(Q, tda.TDA_F32, nq, D, P, nt, D, D) == 1
    S = torch.full((nq, nt + 4), 0.5, device=dev)
    tda.tda_score(Q, tda.TDA_F32, nq, D, P, nt, D, D, S, nt + 4, beta)
    tda.tda_device_status()
    ref = Q.double() @ P.double().T
    assert float((S[:, :nt].double() - 0.5 * beta - ref).norm() / ref.norm()) <= 8.2e-7
    assert (S[:, nt:] == 0.5).all()
