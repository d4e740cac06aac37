"""The row/column kernels (one frame or 32 frames per block) against the one-thread-per-frame
kernel: the same additions in the same order, so every output is bit-identical -- hard
decisions, iterations, flags and the final LLRs -- for each message format, at batch sizes
around the blocks' edges, for any number of copies, and on frames with ties, zeros, tiny
and huge values, infinities and NaN.  (The other decode tests hold both to the oracle.)
The plain decoder's kernel against the precompiled one likewise.
The row-by-row backward kernel against the precompiled one: the same terms in another
order, on the same kinds of frames."""
import numpy as np
import pytest

from helpers import autos_dev, frames, to_dev
from paper_2412_20828_gb300 import bchdec as B

pytestmark = pytest.mark.gpu

I8F = dict(msg=B.MSG_INT8, rescale=True, qfrac=8)


def _llr(n, k, F, ld, seed):
    _, llr = frames(n, k, F, 2.5, seed, ld=ld)
    odd = [lambda r: r.__setitem__(slice(0, 8), 1.5), lambda r: r.fill(0.0), lambda r: r.fill(-1.0),
           lambda r: r.__setitem__(3, np.nan), lambda r: r.__setitem__(slice(2, 9), np.inf),
           lambda r: r.__setitem__(1, -np.inf), lambda r: r.__setitem__(slice(0, 5), 1e-40),
           lambda r: r.__imul__(1e30), lambda r: r.__imul__(1e-20), lambda r: r.__setitem__(2, -0.0),
           lambda r: np.rint(r, out=r), lambda r: r.__setitem__(slice(5, n - 5), np.nan)]
    for f, change in enumerate(odd):
        if f + 1 < F:
            change(llr[f + 1, :n])
    return llr


def _decode(monkeypatch, rc, code, llr, autos, iters, kw):
    import torch
    monkeypatch.setenv("BCHDEC_JIT_RC", str(rc))
    F, ld = llr.shape
    out = [torch.full((F, (code.n + 63) // 64), -1, dtype=torch.int64, device="cuda"),
           torch.zeros(F, dtype=torch.uint8, device="cuda"),
           torch.full((F,), 9, dtype=torch.uint8, device="cuda"), torch.zeros((F, ld), device="cuda")]
    B.nms_decode(code, B.params(iters, 0.78, n_autos=autos.shape[1], **kw), to_dev(llr), autos_dev(autos), *out)
    torch.cuda.synchronize()
    return [o.cpu().numpy().view(np.uint8) for o in out]


@pytest.mark.parametrize("nk", [(15, 7), (63, 36), (63, 45), (127, 64), (127, 99)])
@pytest.mark.parametrize("kw", [{}, dict(msg=B.MSG_FP16), dict(msg=B.MSG_FP16, rescale=True),
                                dict(msg=B.MSG_INT8), I8F], ids=["fp32", "fp16", "fp16r", "int8", "int8f"])
def test_bit_identical_to_one_thread_per_frame(nk, kw, monkeypatch):
    n, k = nk
    code = B.Code(n, k)
    shapes = [(1, 3, 12, True, n), (33, 3, 12, True, n + 1), (500, 3, 12, True, n + 1)]
    if not kw:  # any number of copies; long decodes pass 2^100; refilled slots
        shapes += [(203, 1, 32, False, n), (300, 4, 6, True, n + 1), (200, 9, 4, True, n), (12000, 3, 12, True, n)]
    for F, P, iters, stop, ld in shapes:
        llr = _llr(n, k, F, ld, 600 + F)
        autos = B.draw_automorphisms_host(n, P, 31, 0, F)
        kk = dict(kw, early_stop=stop)
        ref = _decode(monkeypatch, 0, code, llr, autos, iters, kk)
        for rc in (1, 32):
            got = _decode(monkeypatch, rc, code, llr, autos, iters, kk)
            for name, x, y in zip(("hard", "iters", "flags", "llr"), ref, got):
                assert np.array_equal(x, y), (name, F, P, iters, rc)


@pytest.mark.parametrize("nk", [(15, 7), (63, 36), (127, 64), (127, 99)])
def test_plain_bit_identical_to_precompiled(nk, monkeypatch):
    import torch
    n, k = nk
    code = B.Code(n, k, kind=B.PCM_STANDARD)
    for F, iters, stop, ld in ((1, 8, True, n), (33, 8, True, n + 1), (700, 10, False, n + 1), (9000, 8, True, n)):
        llr, got = to_dev(_llr(n, k, F, ld, 700 + F)), []
        for rc in ("generic", "1", "16", "32"):
            monkeypatch.setenv("BCHDEC_NMS_KERNEL", "generic" if rc == "generic" else "auto")
            monkeypatch.setenv("BCHDEC_JIT_RC", rc)
            out = [torch.full((F, (n + 63) // 64), -1, dtype=torch.int64, device="cuda"),
                   torch.zeros(F, dtype=torch.uint8, device="cuda"),
                   torch.full((F,), 9, dtype=torch.uint8, device="cuda"), torch.zeros((F, ld), device="cuda")]
            B.nms_decode(code, B.params(iters, 0.78, n_autos=0, early_stop=stop), llr, None, *out)
            got.append([o.cpu().numpy().view(np.uint8) for o in out])
        for rc in (1, 2, 3):
            for name, x, y in zip(("hard", "iters", "flags", "llr"), got[0], got[rc]):
                assert np.array_equal(x, y), (name, F, rc)


@pytest.mark.parametrize("nk", [(63, 45), (127, 64)])
def test_checkpoints_bit_identical(nk, monkeypatch):
    import torch
    n, k = nk
    code, F, iters = B.Code(n, k), 301, 7
    _, llr = frames(n, k, F, 2.5, 77, ld=n)
    autos = B.draw_automorphisms_host(n, 3, 32, 0, F)
    got = []
    for rc in (0, 1, 32):
        monkeypatch.setenv("BCHDEC_JIT_RC", str(rc))
        ck = torch.zeros((iters + 1, F, n), device="cuda")
        B.nms_forward_train(code, B.params(iters, 0.7), to_dev(llr), autos_dev(autos), ck)
        got.append(ck)
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


@pytest.mark.parametrize("nk", [(15, 7), (63, 45), (127, 64), (127, 99)])
@pytest.mark.parametrize("F,P,iters,pad", [(1, 3, 4, 0), (33, 3, 6, 1), (500, 3, 12, 1), (65, 9, 3, 0)])
def test_backward_against_precompiled(nk, F, P, iters, pad, monkeypatch):
    """Both kernels add the same FP32 terms; each iteration's gradient is a chain of at most
    (row weight + copies x column degree) additions, so their results differ by at most
    iterations x that x 2^-24 of the gradient's norm (dL/dalpha: the oracle tests' 2e-3)."""
    import torch
    n, k = nk
    code, ld = B.Code(n, k), n + pad
    H = code.dense()
    llr = _llr(n, k, F, ld, 800 + F)
    autos = autos_dev(B.draw_automorphisms_host(n, P, 33, 0, F))
    p = B.params(iters, 0.7, n_autos=P)
    ck = torch.zeros((iters + 1, F, ld), device="cuda")
    B.nms_forward_train(code, p, to_dev(llr), autos, ck)
    go = torch.from_numpy(np.random.default_rng(F).standard_normal((F, ld)).astype(np.float32)).cuda()
    got = []
    for mode in ("generic", "auto"):
        monkeypatch.setenv("BCHDEC_NMS_KERNEL", mode)
        gl, ga = torch.zeros((F, ld), device="cuda"), torch.zeros(iters, device="cuda")
        B.nms_backward(code, p, autos, ck, go, gl, ga)
        got.append((gl[:, :n].double(), ga.double()))
    (g0, a0), (g1, a1) = got
    fine = torch.isfinite(g0)
    assert torch.equal(fine, torch.isfinite(g1))
    chain = int(H.sum(1).max()) + P * int(H.sum(0).max())
    assert (g0 - g1)[fine].norm() <= iters * chain * 2.0 ** -24 * g0[fine].norm()
    usable = torch.isfinite(a0) & torch.isfinite(a1)
    assert torch.equal(usable, torch.isfinite(a0))
    # against the largest factor's gradient: the terms of opposite sign cancel in the others
    if usable.any():  # a frame of infinities makes every factor's gradient NaN
        assert ((a0 - a1)[usable].abs() <= 2e-3 * a0[usable].abs().max()).all()
