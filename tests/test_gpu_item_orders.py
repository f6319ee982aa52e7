"""The launch plans and item orders that only many heads reach, against the oracle: pass 2 with two
CTAs per SM for the resolved grid and the rounded exponentials, its groups of compute warps taking
one-tile items in turn, output tiles staged over a V^T ring that holds both.  More items than a host
schedule holds (snake order), against the same heads in calls that have one.  And schedules asked
for by several threads at once."""
import threading

import pytest
import torch

from paper_2609_33591_gb300 import kint
from paper_2609_33591_gb300.inputs import make_qkvdo
from tests import parity

pytestmark = pytest.mark.gpu

MM, FW, SM, FR = kint.CALIB_MINMAX, kint.CALIB_FWM, kint.CALIB_SOFTMAX, kint.CALIB_FWM_RESOLVED
E8, EB = kint.CALIB_EXP_FP8, kint.CALIB_EXP_BF16
LE, NE, WE, PR = kint.RECON_LERP, kint.RECON_NEAREST, kint.STE_WEIGHT, kint.STE_PROB
X3, TF = kint.PREC_3XTF32, kint.PREC_TF32


@pytest.fixture(autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("BH,T,d,c,K,r,s,prec", [
    (170, 129, 64, FR, 8, LE, WE, TF),   # two CTAs per SM
    (170, 129, 64, FR, 8, NE, WE, TF),
    (170, 190, 64, E8, 1, LE, WE, TF),
    (170, 190, 64, EB, 1, LE, WE, TF),
    (320, 64, 128, FW, 4, NE, WE, TF),   # one tile per item, the two groups in turn
    (320, 40, 128, MM, 8, LE, WE, TF),
    (320, 64, 128, FW, 4, NE, PR, TF),
    (320, 40, 64, FW, 4, NE, PR, X3),
    (400, 130, 64, MM, 8, NE, PR, TF),   # one and three tiles
    (170, 129, 64, MM, 47, NE, PR, TF),  # O and O_lerp together over four V^T slots
    (170, 129, 64, MM, 48, NE, PR, TF),  # one after the other over three
])
def test_plans_of_many_heads(BH, T, d, c, K, r, s, prec):
    Q, K_, V, dO = make_qkvdo(1, BH, T, d, seed=T + d + K)
    cfg = kint.Config(Kint=K, calib=c, tau=8.0, recon=r, ste=s, grad=kint.GRAD_FULL)
    parity.check(Q, K_, V, dO, cfg, prec, want_bwd=False)


@pytest.mark.parametrize("BH,T,d,c,K,r,s,prec", [
    (2100, 65, 128, FW, 4, NE, WE, TF),  # passes 1 and 2, dQ, dV and dK at d = 128
    (1100, 130, 64, MM, 4, LE, WE, X3),  # and under 3xTF32
    (1100, 130, 64, MM, 8, NE, PR, TF),  # the two-pass kernels at d = 64
    (1100, 130, 64, SM, 1, LE, WE, TF),  # the single pass
])
def test_more_items_than_a_schedule_holds(BH, T, d, c, K, r, s, prec):
    """A head's results do not depend on the order of the items: bit for bit those of calls of few heads
    (also dQ of the single pass, where at most two key blocks' parts meet in a row here: a sum of two
    is the same in either order)."""
    cfg = kint.Config(Kint=K, calib=c, tau=8.0, recon=r, ste=s, grad=kint.GRAD_FULL)
    q, k, v, do = (torch.from_numpy(x).to("cuda:0") for x in make_qkvdo(1, BH, T, d, seed=T + d + K))

    def run(h0, h1):
        x = [t[:, h0:h1].contiguous() for t in (q, k, v, do)]
        O, st = kint.forward(*x[:3], cfg, prec)
        return (O, *kint.backward(*x[:3], O, x[3], st, cfg, prec))

    whole = run(0, BH)
    n = BH // 10
    parts = [torch.cat(p, 1) for p in zip(*(run(h, h + n) for h in range(0, BH, n)))]
    for name, a, b in zip(("O", "dQ", "dK", "dV"), whole, parts):
        assert torch.equal(a, b), name
    kint.check_status()


def test_calls_from_several_threads():
    """Four threads, each on its own stream, run forwards and two-pass backwards of the same new shapes
    at once; every result is bit for bit the one that a single thread gets."""
    cfg = kint.Config(Kint=4, calib=FW, tau=8.0, recon=NE, ste=WE, grad=kint.GRAD_FULL)
    shapes = [(1, 90, T, 128) for T in (257, 300, 391, 450)]
    inputs = [tuple(torch.from_numpy(x).to("cuda:0") for x in make_qkvdo(*sh, seed=5 + k)) for k, sh in enumerate(shapes)]

    def run(q, k, v, do):
        O, st = kint.forward(q, k, v, cfg, TF)
        return (O, *kint.backward(q, k, v, O, do, st, cfg, TF))

    got, errors = {}, []
    start = threading.Barrier(4)

    def work(t):
        try:
            start.wait()
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for j in range(len(shapes)):
                    i = (j + t // 2) % len(shapes)
                    got[t, i] = run(*inputs[i])
            s.synchronize()
        except Exception as e:  # noqa: BLE001 (reported below, in the main thread)
            errors.append(e)

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for i, x in enumerate(inputs):
        want = run(*x)
        for t in range(4):
            for a, b in zip(got[t, i], want):
                assert torch.equal(a, b), (t, i)
    kint.check_status()
