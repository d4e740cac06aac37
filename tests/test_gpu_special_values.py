"""FP32 decoding of frames with infinite, NaN and overflowing LLRs among ordinary ones, in
batches large enough that every kernel refills its slots with new frames.

The reference is the one-thread-per-frame kernel whose rows run in edge order
(BCHDEC_JIT_GRID=0, BCHDEC_JIT_RC=0): it takes every value as it comes and leaves no frame to
another kernel.  All kernels add the same terms in the same order, so every output is the
same bits."""
import numpy as np
import pytest

from helpers import autos_dev
from paper_2412_20828_gb300 import bchdec as B

pytestmark = pytest.mark.gpu

FMAX = np.float32(3.402823466e38)


def _batch(code, F, ld, seed):
    """F frames at 1 to 6 dB; every third one with special values, spread over the batch."""
    import torch
    n = code.n
    llr = torch.zeros((F, ld), device="cuda")
    B.gen_frames(code, 1.0, 6.0, seed, 0, llr)
    rng = np.random.default_rng(seed)
    x = llr.cpu().numpy()
    for f in range(0, F, 3):
        r = x[f, :n]
        at = rng.permutation(n)[:rng.integers(1, n + 1)]
        what = rng.integers(0, 8)
        if what == 0:
            r[at[:9]] = np.inf
        elif what == 1:  # rows with all or all but one infinite
            r[at] = rng.choice([-np.inf, np.inf], at.size)
        elif what == 2:
            r[:] = np.inf
            r[at[0]] = 1.5
        elif what == 3:
            r[at[:2]] = np.nan
        elif what == 4:
            r[at] = np.nan
        elif what == 5:  # passes 2^100 and the range after a merge: infinities, then NaN
            with np.errstate(over="ignore"):
                r *= np.float32(1e37)
        elif what == 6:
            r[:] = np.where(r < 0, -FMAX, FMAX)
        else:
            r[at[:2]] = [np.inf, np.nan][:at[:2].size]
    return torch.from_numpy(x).cuda()


def _decode(code, llr, autos, iters, stop):
    import torch
    F, ld = llr.shape
    out = [torch.full((F, (code.n + 63) // 64), -1, dtype=torch.int64, device="cuda"),
           torch.zeros(F, dtype=torch.uint8, device="cuda"),
           torch.full((F,), 9, dtype=torch.uint8, device="cuda"), torch.zeros((F, ld), device="cuda")]
    B.nms_decode(code, B.params(iters, 0.78, n_autos=autos.shape[1], early_stop=stop), llr, autos, *out)
    return [o.view(torch.uint8) for o in out]


# 100 003 frames: 256 x 152 in flight on the one-thread-per-frame kernel, so its lanes go from a
# deferred or finished frame to a new one; the row/column kernels hold fewer
@pytest.mark.parametrize("nk,F", [((15, 7), 100_003), ((63, 36), 100_003), ((63, 45), 100_003), ((127, 99), 30_001)])
@pytest.mark.parametrize("P,iters,stop", [(3, 12, True), (3, 7, False), (4, 5, True)])
def test_special_values_bit_identical(nk, F, P, iters, stop, monkeypatch):
    import torch
    code = B.Code(*nk)
    llr = _batch(code, F, nk[0] + 1, F + P)
    autos = autos_dev(B.draw_automorphisms_host(nk[0], P, 51, 0, F))
    monkeypatch.setenv("BCHDEC_JIT_GRID", "0")
    monkeypatch.setenv("BCHDEC_JIT_RC", "0")
    ref = _decode(code, llr, autos, iters, stop)
    monkeypatch.delenv("BCHDEC_JIT_GRID")
    for rc in ("0", "1", "32", None):
        monkeypatch.setenv("BCHDEC_JIT_RC", rc) if rc else monkeypatch.delenv("BCHDEC_JIT_RC")
        for name, x, y in zip(("hard", "iters", "flags", "llr"), ref, _decode(code, llr, autos, iters, stop)):
            assert torch.equal(x, y), (name, rc)


@pytest.mark.parametrize("nk", [(63, 36), (63, 45)])
def test_infinite_bits_keep_the_batch_kernel_s_speed(nk):
    """Known bits arrive as infinite LLRs, in every frame.  They scale a frame down at each
    merge and change how many iterations it runs, 1.1 to 1.5 times the time of finite frames
    on the edge-order kernel; on a kernel of one frame per block it is 7 to 10 times."""
    import torch
    code, F = B.Code(*nk), 400_000
    autos = autos_dev(B.draw_automorphisms_host(63, 3, 52, 0, F))
    times = []
    for infinite in (False, True):
        llr = torch.zeros((F, 64), device="cuda")
        B.gen_frames(code, 1.0, 6.0, 53, 0, llr)
        if infinite:
            llr[:, 5:14] = float("inf")
        hard = torch.zeros((F, 1), dtype=torch.int64, device="cuda")
        p, best = B.params(12, 0.78), float("inf")
        ws = B.workspace(code, p, F)
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            B.nms_decode(code, p, llr, autos, hard, ws=ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] <= 3.0 * times[0], times


def test_checkpoints_of_deferred_frames(monkeypatch):
    """The training forward pass on a batch large enough to defer its NaN frames: every
    checkpoint is the same bits as in edge order."""
    import torch
    code, F, iters = B.Code(63, 45), 70_001, 6
    llr = _batch(code, F, 64, 9)
    autos = autos_dev(B.draw_automorphisms_host(63, 3, 54, 0, F))
    p = B.params(iters, 0.7)
    assert code.kernel_name(B.params(iters, 0.7, early_stop=False), F) == "bch_nms_jit + bch_nms_rc"
    got = []
    for grid in ("0", "1"):
        monkeypatch.setenv("BCHDEC_JIT_GRID", grid)
        ck = torch.zeros((iters + 1, F, 64), device="cuda")
        B.nms_forward_train(code, p, llr, autos, ck)
        got.append(ck.view(torch.int32))
    assert torch.equal(got[0], got[1])
