"""Pass 2 when the bounded wait for the first Q tile runs out in some warps of a CTA and not in
others: the warps agree before the item loop (one that skips it would leave the others waiting at the
item's barriers for good), the launch flags the status word and leaves, and the next call is correct.
One and two CTAs per SM, with and without the per-row tables' barrier, d = 128.  Nothing faults, traps or hangs: the wait that runs out is
on a barrier that nothing arrives at, the copies and products issued meanwhile complete."""
import pytest
import torch

from paper_2609_33591_gb300 import kint
from paper_2609_33591_gb300.inputs import make_qkvdo
from tests import parity

pytestmark = pytest.mark.gpu

DEFAULT_WAIT_NS = 2_000_000_000
MM, FW = kint.CALIB_MINMAX, kint.CALIB_FWM
LE, NE = kint.RECON_LERP, kint.RECON_NEAREST


@pytest.fixture(autouse=True)
def _restore():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kint.load()
    yield
    kint.kint_test_expire_next_q_wait(0)
    kint.kint_set_wait_timeout_ns(DEFAULT_WAIT_NS)


@pytest.mark.parametrize("BH,T,d,c,K,r", [
    (2, 200, 64, FW, 4, NE),    # one CTA per SM
    (2, 200, 64, MM, 8, LE),    # per-row tables: a barrier at the item's start
    (160, 130, 64, FW, 4, NE),  # two CTAs per SM, several items per CTA
    (160, 130, 64, MM, 8, LE),
    (2, 200, 128, FW, 4, NE),
    (2, 200, 128, MM, 8, LE),
])
def test_warps_agree_on_an_expired_q_wait(BH, T, d, c, K, r):
    prec = kint.PREC_TF32
    cfg = kint.Config(Kint=K, calib=c, tau=8.0, recon=r, ste=kint.STE_WEIGHT, grad=kint.GRAD_FULL)
    Q, K_, V, dO = make_qkvdo(1, BH, T, d, seed=41)
    q, k, v = (torch.from_numpy(x).to("cuda:0") for x in (Q, K_, V))
    assert kint.kint_get_status() == (0, 0)
    kint.kint_set_wait_timeout_ns(2_000_000)  # 2 ms
    kint.kint_test_expire_next_q_wait(1)
    kint.forward(q, k, v, cfg, prec)
    rc, detail = kint.kint_get_status()
    assert rc == -6 and detail & 1, (rc, detail)  # KINT_ERR_DEVICE, "TMA wait timed out"
    assert kint.kint_get_status() == (0, 0)  # the word was cleared
    kint.kint_set_wait_timeout_ns(DEFAULT_WAIT_NS)
    # the hook was consumed: the same call now runs normally and is correct
    parity.check(Q, K_, V, dO, cfg, prec, want_bwd=False)
    assert kint.kint_get_status() == (0, 0)
