"""The size rules that pick a min-sum kernel, at corners where every frame runs all its
iterations (no early stop, or 1 to 2 dB): the kernel a call gets by default takes no longer
than the one-thread-per-frame kernel (BCHDEC_JIT_RC=0; plain decoder: the precompiled one).
The bound allows 15% for the scatter of two best-of-six times; past the lines the row/column
kernels took 1.2 to 2.8 times as long on these calls."""
import pytest

from helpers import autos_dev
from paper_2412_20828_gb300 import bchdec as B

pytestmark = pytest.mark.gpu

I8F = dict(msg=B.MSG_INT8, rescale=True, qfrac=8)


def _time(call):
    import torch
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(3):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _inputs(code, frames_per_sm, hi):
    import torch
    F = frames_per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    llr = torch.zeros((F, code.n + 1), device="cuda")
    B.gen_frames(code, 1.0, hi, 81, 0, llr)
    return llr, torch.zeros((F, (code.n + 63) // 64), dtype=torch.int64, device="cuda")


@pytest.mark.parametrize("nk,rows,P,iters,kw,per_sm", [
    ((127, 99), 0, 9, 4, I8F, 112), ((127, 64), 0, 5, 12, {}, 112), ((63, 45), 0, 3, 12, dict(msg=B.MSG_FP16), 224),
    ((63, 36), 122, 1, 12, {}, 300), ((63, 36), 122, 2, 2, I8F, 1500), ((15, 7), 0, 9, 12, {}, 63),
    ((63, 30), 0, 1, 12, {}, 64), ((127, 99), 0, 1, 12, {}, 100)])
@pytest.mark.parametrize("stop", [True, False])
def test_no_call_slower_than_one_thread_per_frame(nk, rows, P, iters, kw, per_sm, stop, monkeypatch):
    code = B.Code(*nk, m_rows=rows)
    llr, hard = _inputs(code, per_sm, 2.0)
    autos = autos_dev(B.draw_automorphisms_host(code.n, P, 82, 0, llr.shape[0]))
    p = B.params(iters, 0.78, n_autos=P, early_stop=stop, **kw)
    ws = B.workspace(code, p, llr.shape[0])
    t = []
    for rc in (None, "0"):
        monkeypatch.setenv("BCHDEC_JIT_RC", rc) if rc else monkeypatch.delenv("BCHDEC_JIT_RC", raising=False)
        t.append(_time(lambda: B.nms_decode(code, p, llr, autos, hard, ws=ws)))
    assert t[0] <= 1.15 * t[1], t


def test_plain_decoder_of_the_shortest_code_not_slower_than_precompiled(monkeypatch):
    code = B.Code(15, 7, kind=B.PCM_STANDARD)
    llr, hard = _inputs(code, 2000, 2.0)
    p = B.params(8, 0.78, n_autos=0)
    ws = B.workspace(code, p, llr.shape[0])
    t = []
    for mode in ("auto", "generic"):
        monkeypatch.setenv("BCHDEC_NMS_KERNEL", mode)
        t.append(_time(lambda: B.nms_decode(code, p, llr, None, hard, ws=ws)))
    assert t[0] <= 1.15 * t[1], t


@pytest.mark.parametrize("P", [1, 3])
def test_backward_of_the_shortest_code_not_slower_than_precompiled(P, monkeypatch):
    import torch
    code, iters = B.Code(15, 7), 12
    llr, _ = _inputs(code, 2000, 5.0)
    F, ld = llr.shape
    autos = autos_dev(B.draw_automorphisms_host(15, P, 83, 0, F))
    p = B.params(iters, 0.7, n_autos=P)
    ckpt = torch.zeros((iters + 1, F, ld), device="cuda")
    B.nms_forward_train(code, p, llr, autos, ckpt)
    go, gl, ga = torch.ones_like(llr), torch.zeros_like(llr), torch.zeros(iters, device="cuda")
    ws = B.workspace(code, p, F)
    t = []
    for mode in ("auto", "generic"):
        monkeypatch.setenv("BCHDEC_NMS_KERNEL", mode)
        t.append(_time(lambda: B.nms_backward(code, p, autos, ckpt, go, gl, ga, ws)))
    assert t[0] <= 1.15 * t[1], t
