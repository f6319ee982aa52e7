"""Backward kernels at d = 128 and under 3xTF32 (separate rings of 64-row tiles, one or two slots
of the second operand) and the dK/dV stage plans, at sizes with odd tile counts, ragged ends and
several items per CTA, against the oracle."""
import pytest
import torch

from paper_2609_33591_gb300 import kint
from paper_2609_33591_gb300.inputs import make_qkvdo
from tests import parity

pytestmark = pytest.mark.gpu

MM, FW, SM = kint.CALIB_MINMAX, kint.CALIB_FWM, kint.CALIB_SOFTMAX
LE, NE, WE, PR = kint.RECON_LERP, kint.RECON_NEAREST, kint.STE_WEIGHT, kint.STE_PROB
FU, DP = kint.GRAD_FULL, kint.GRAD_DETACH_PROJ
X3, TF = kint.PREC_3XTF32, kint.PREC_TF32


@pytest.mark.parametrize("BH,T,d,c,K,r,s,g,prec", [
    (160, 130, 128, FW, 4, NE, WE, FU, TF),  # d = 128: several items per CTA, odd tile counts
    (420, 130, 128, FW, 4, NE, WE, FU, TF),  # tiles of all heads past the L2 share: groups of heads
    (90, 193, 128, MM, 16, LE, WE, FU, TF),  # two slots of the second operand beside pair tables
    (80, 257, 128, MM, 32, NE, PR, FU, TF),  # one slot beside the largest tables
    (170, 65, 128, SM, 1, LE, WE, FU, TF),   # a one-row last tile
    (160, 129, 64, FW, 4, NE, PR, FU, X3),   # 3xTF32: hi / lo operands, cross-term accumulator
    (80, 191, 64, MM, 32, LE, WE, FU, X3),   # 3xTF32 beside the largest tables
    (160, 100, 64, MM, 8, NE, WE, DP, X3),   # 3xTF32, projected rows
    (170, 190, 64, MM, 8, NE, PR, FU, TF),   # d = 64, two passes: V and K staged, both products
])
def test_backward_plans(BH, T, d, c, K, r, s, g, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Q, K_, V, dO = make_qkvdo(1, BH, T, d, seed=T + d)
    cfg = kint.Config(Kint=K, calib=c, tau=8.0, recon=r, ste=s, grad=g)
    parity.check(Q, K_, V, dO, cfg, prec, want_bwd=True)
