"""Pass 2 under each launch plan (one or two CTAs per SM, ring depths, staging beside or over the
V^T ring, one or two output tiles) at sizes with odd tile counts, ragged ends and several items
per CTA, against the oracle."""
import pytest
import torch

from paper_2609_33591_gb300 import kint
from paper_2609_33591_gb300.inputs import make_qkvdo
from tests import parity

pytestmark = pytest.mark.gpu

MM, FW, SM = kint.CALIB_MINMAX, kint.CALIB_FWM, kint.CALIB_SOFTMAX
LE, NE, WE, PR = kint.RECON_LERP, kint.RECON_NEAREST, kint.STE_WEIGHT, kint.STE_PROB
X3, TF = kint.PREC_3XTF32, kint.PREC_TF32


@pytest.mark.parametrize("BH,T,d,c,K,r,s,prec", [
    (160, 65, 64, FW, 64, NE, WE, TF),   # two CTAs per SM, the largest line table, a one-key second tile
    (170, 130, 64, MM, 16, NE, WE, TF),  # two CTAs per SM, endpoint tables, one K slot
    (170, 129, 64, MM, 32, LE, WE, TF),  # tables too large for two CTAs per SM
    (320, 64, 64, SM, 1, LE, WE, TF),    # one tile per item, several items per CTA
    (170, 190, 64, FW, 4, NE, PR, TF),   # O and O_lerp side by side, three score buffers
    (170, 129, 64, MM, 64, NE, PR, TF),  # the same beside the largest pair tables
    (160, 129, 64, FW, 4, NE, PR, X3),   # 3xTF32, one launch each for O and O_lerp
    (160, 70, 64, MM, 32, LE, WE, X3),   # 3xTF32 beside 32 KB of tables: one K slot
    (90, 193, 128, FW, 8, NE, WE, TF),   # d = 128, staging over the V^T ring
    (90, 193, 128, FW, 8, NE, PR, TF),   # O and O_lerp one after the other
    (90, 130, 128, MM, 32, LE, WE, TF),  # d = 128 beside 32 KB of tables: one K slot
])
def test_forward_plans(BH, T, d, c, K, r, s, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Q, K_, V, dO = make_qkvdo(1, BH, T, d, seed=T + d)
    cfg = kint.Config(Kint=K, calib=c, tau=8.0, recon=r, ste=s, grad=kint.GRAD_FULL)
    parity.check(Q, K_, V, dO, cfg, prec, want_bwd=False)
