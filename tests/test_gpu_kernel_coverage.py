"""Every min-sum and backward kernel at the sizes that make it do its work, whatever kernel the
size rules would pick: the older parity tests on the one-thread-per-frame kernel and on 32
frames per block (their few hundred frames otherwise run one frame per block), slots that take
several frames one after the other, and blocks of the backward pass that take several groups."""
import numpy as np
import pytest

import test_gpu_decode as decode_tests
import test_gpu_precision as precision_tests
from helpers import autos_dev, to_dev
from paper_2412_20828_gb300 import bchdec as B
from test_gpu_special_values import _batch

pytestmark = pytest.mark.gpu

I8F = dict(msg=B.MSG_INT8, rescale=True, qfrac=8)
both = pytest.mark.parametrize("rc", ["0", "32"])


@both
@pytest.mark.parametrize("nk", [(63, 45), (127, 64)])
def test_fp32_against_oracle(nk, rc, monkeypatch):
    import torch
    monkeypatch.setenv("BCHDEC_JIT_RC", rc)
    decode_tests.test_enhanced_one_iteration(torch, nk)
    decode_tests.test_enhanced_full_decode(torch, nk, 1.5)


@both
@pytest.mark.parametrize("nk", [(63, 36), (127, 64)])
@pytest.mark.parametrize("msg", [B.MSG_FP32, B.MSG_INT8])
def test_jit_and_generic_agree(nk, msg, rc, monkeypatch):
    import torch
    monkeypatch.setenv("BCHDEC_JIT_RC", rc)
    decode_tests.test_jit_and_generic_kernels_agree(torch, msg, nk, monkeypatch)


@both
@pytest.mark.parametrize("nk", [(63, 36), (63, 45), (127, 99)])
@pytest.mark.parametrize("rescale", [False, True])
def test_reduced_formats_against_oracle(nk, rescale, rc, monkeypatch):
    import torch
    monkeypatch.setenv("BCHDEC_JIT_RC", rc)
    precision_tests.test_int8_bit_exact(torch, nk, rescale)
    precision_tests.test_int8_fractional_bit_exact(torch, nk, rescale, "jit", monkeypatch)
    if nk != (63, 36):
        precision_tests.test_fp16_close_to_oracle(torch, nk, 2.5 if nk[0] == 63 else 3.5, rescale)


@pytest.mark.parametrize("kw", [{}, dict(msg=B.MSG_FP16)], ids=["fp32", "fp16"])
def test_straight_line_row_forms_bit_identical(kw, monkeypatch):
    """The one-thread-per-frame kernel's forms of a row: min1/min2 from a grid or in edge order,
    the min2 correction by a compare or on the FMA pipe."""
    import torch
    code, F = B.Code(63, 45), 60_001
    llr = torch.zeros((F, 64), device="cuda")
    B.gen_frames(code, 1.0, 6.0, 61, 0, llr)
    llr[: F // 4, :8] = 1.5  # ties
    llr[F // 4: F // 2, :8] = 1e-40  # differences below the normal range
    autos = autos_dev(B.draw_automorphisms_host(63, 3, 62, 0, F))
    monkeypatch.setenv("BCHDEC_JIT_RC", "0")
    got = []
    for grid, pct in (("0", "0"), ("0", "50"), ("1", "0"), ("1", "50"), ("1", "100")):
        monkeypatch.setenv("BCHDEC_JIT_GRID", grid)
        monkeypatch.setenv("BCHDEC_JIT_FMA_PCT", pct)
        got.append(_decode(code, llr, autos, 12, kw))
    for other in got[1:]:
        assert all(torch.equal(x, y) for x, y in zip(got[0], other))


def _decode(code, llr, autos, iters, kw):
    import torch
    F, ld = llr.shape
    out = [torch.full((F, (code.n + 63) // 64), -1, dtype=torch.int64, device="cuda"),
           torch.zeros(F, dtype=torch.uint8, device="cuda"),
           torch.full((F,), 9, dtype=torch.uint8, device="cuda"), torch.zeros((F, ld), device="cuda")]
    B.nms_decode(code, B.params(iters, 0.78, n_autos=autos.shape[1], **kw), llr, autos, *out)
    return [o.view(torch.uint8) for o in out]


@pytest.mark.parametrize("nk", [(15, 7), (63, 36), (127, 99)])
@pytest.mark.parametrize("kw", [dict(msg=B.MSG_FP16), dict(msg=B.MSG_FP16, rescale=True), dict(msg=B.MSG_INT8),
                                dict(msg=B.MSG_INT8, rescale=True), I8F], ids=["fp16", "fp16r", "int8", "int8r", "int8f"])
def test_reduced_formats_refill_their_slots(nk, kw, monkeypatch):
    """More frames than any kernel holds at a time (one thread per frame 38 912, 32 frames per
    block 9 728 for n = 63), infinities and NaN among them: exponents and hard decisions start
    afresh in a slot's next frame."""
    import torch
    code, F = B.Code(*nk), 60_001
    llr = _batch(code, F, nk[0] + 1, 71)
    autos = autos_dev(B.draw_automorphisms_host(nk[0], 3, 72, 0, F))
    got = []
    for rc in ("0", "1", "32"):
        monkeypatch.setenv("BCHDEC_JIT_RC", rc)
        got.append(_decode(code, llr, autos, 12, kw))
    for rc, other in zip((1, 32), got[1:]):
        for name, x, y in zip(("hard", "iters", "flags", "llr"), got[0], other):
            assert torch.equal(x, y), (name, rc)


@pytest.mark.parametrize("nk", [(15, 7), (63, 45), (127, 64)])
def test_backward_blocks_take_several_groups(nk):
    """20 001 ordinary frames, 626 groups of 32 on at most 608 blocks.  Each frame's gradient is
    the same bits as in a call of its group alone.  dL/dalpha is the sum of the groups' values
    d_g, each exact in its own call of one block: 626 additions in FP32, so within
    626 x 2^-24 x sum |d_g| of the FP64 sum."""
    import torch
    n, F, iters, P = nk[0], 20_001, 5, 3
    code, ld = B.Code(*nk), nk[0] + 1
    p = B.params(iters, [0.7, 0.75, 0.8, 0.72, 0.78], n_autos=P)
    llr = torch.zeros((F, ld), device="cuda")
    B.gen_frames(code, 2.0, 5.0, 73, 0, llr)
    autos = autos_dev(B.draw_automorphisms_host(n, P, 74, 0, F))
    ckpt = torch.zeros((iters + 1, F, ld), device="cuda")
    B.nms_forward_train(code, p, llr, autos, ckpt)
    go = torch.randn((F, ld), generator=torch.Generator("cuda").manual_seed(75), device="cuda")

    def backward(sl):
        gl, ga = torch.zeros_like(go[sl]), torch.zeros(iters, device="cuda")
        B.nms_backward(code, p, autos[sl].contiguous(), ckpt[:, sl].contiguous(), go[sl].contiguous(), gl, ga)
        return gl[:, :n], ga

    gl, ga = backward(slice(0, F))
    d = []
    for f in range(0, F, 32):
        one, da = backward(slice(f, min(F, f + 32)))
        assert torch.equal(one.view(torch.int32), gl[f:f + 32].view(torch.int32)), f
        d.append(da.double())
    d = torch.stack(d)
    assert ((ga.double() - d.sum(0)).abs() <= len(d) * 2.0 ** -24 * d.abs().sum(0)).all()


@pytest.mark.parametrize("nk", [(15, 7), (63, 45), (127, 64)])
def test_backward_alpha_gradient_of_ordinary_frames_against_precompiled(nk, monkeypatch):
    """dL/dalpha of ordinary frames over one iteration, both kernels against FP64.  It is a sum of
    terms g m (a row's gradients times its minimum without them).  A value passes through at
    most N = edges x copies additions in its lane, which holds one frame here, and 1024 on the way
    through lanes, warps and blocks, so the result is within N 2^-24 of the terms' magnitudes."""
    import torch
    n, F, P, alpha = nk[0], 3000, 3, 0.7
    code, ld = B.Code(*nk), nk[0]
    H = torch.from_numpy(code.dense()).cuda().bool()
    p = B.params(1, alpha, n_autos=P)
    llr = torch.zeros((F, ld), device="cuda")
    B.gen_frames(code, 2.0, 5.0, 76, 0, llr)
    host = B.draw_automorphisms_host(n, P, 77, 0, F)
    autos = autos_dev(host)
    ckpt = torch.zeros((2, F, ld), device="cuda")
    B.nms_forward_train(code, p, llr, autos, ckpt)
    go = torch.randn((F, ld), generator=torch.Generator("cuda").manual_seed(78), device="cuda")
    ga = []
    for mode in ("generic", "auto"):
        monkeypatch.setenv("BCHDEC_NMS_KERNEL", mode)
        ga.append(torch.zeros(1, device="cuda"))
        B.nms_backward(code, p, autos, ckpt, go, torch.zeros_like(go), ga[-1])
    # the terms in FP64: z[pi(i)] = y[i], pi(i) = 2^j i + s mod n
    shift, power = to_dev((host & 0xff).astype(np.int64)), to_dev((host >> 8).astype(np.int64))
    pos = torch.arange(n, device="cuda")
    total = torch.zeros(1, dtype=torch.float64, device="cuda")
    mags = torch.zeros_like(total)
    for c in range(P):
        pi = (pos[None] * (1 << power[:, c:c + 1]) + shift[:, c:c + 1]) % n
        z = torch.zeros((F, n), dtype=torch.float64, device="cuda").scatter_(1, pi, llr.double())
        g = torch.zeros_like(z).scatter_(1, pi, go.double() / P)
        for row in H:
            v, gr = z[:, row], g[:, row]
            two, at = v.abs().topk(2, dim=1, largest=False)
            m = two[:, :1].expand_as(v).scatter(1, at[:, :1], two[:, 1:])
            s = torch.where(v < 0, -1.0, 1.0)
            terms = gr * s * s.prod(1, keepdim=True) * m
            total += terms.sum()
            mags += terms.abs().sum()
    n_terms = int(H.sum()) * P + 1024
    for x in ga:
        err = (x.double() - total).abs()
        assert (err <= n_terms * 2.0 ** -24 * mags).all(), (err, mags)
