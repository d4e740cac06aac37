"""bch_nms_kernel_info loads every kernel that later decodes run (none compiles then), and
bch_nms_kernel_name names the kernels a call of a given size runs."""
import os

import pytest

from helpers import autos_dev
from paper_2412_20828_gb300 import bchdec as B

pytestmark = pytest.mark.gpu


def _decode(code, F, P=3, **kw):
    import torch
    llr = torch.zeros((F, code.n + 1), device="cuda")
    B.gen_frames(code, 1.0, 6.0, 91, 0, llr)
    autos = autos_dev(B.draw_automorphisms_host(code.n, P, 92, 0, F)) if P else None
    hard = torch.zeros((F, (code.n + 63) // 64), dtype=torch.int64, device="cuda")
    B.nms_decode(code, B.params(12, 0.78, n_autos=P, **kw), llr, autos, hard)
    torch.cuda.synchronize()


@pytest.mark.parametrize("nk,msg,kernels", [((63, 51), B.MSG_FP32, 3), ((63, 51), B.MSG_INT8, 3),
                                            ((127, 99), B.MSG_FP32, 2)])
def test_kernel_info_compiles_what_decodes_run(nk, msg, kernels, tmp_path, monkeypatch):
    """A matrix of this test's own seed, so that nothing of it is in the process yet; every
    compile leaves a file in the cache folder.  n = 127 with three copies never runs the
    straight-line kernel, so its compile, the longest, is not among them."""
    monkeypatch.setenv("BCHDEC_JIT_CACHE_DIR", str(tmp_path))
    code = B.Code(*nk, seed=20_000 + msg)
    assert code.kernel_info(msg) == "jit"
    assert len(os.listdir(tmp_path)) == kernels
    for F in (1, 700, 9000, 25_000, 60_000):
        _decode(code, F, msg=msg)
        assert len(os.listdir(tmp_path)) == kernels, F


def test_kernel_names_by_size(monkeypatch):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    short, long_, plain = B.Code(63, 45), B.Code(127, 99), B.Code(63, 45, kind=B.PCM_STANDARD)
    p, p0 = B.params(12, 0.78), B.params(12, 0.78, n_autos=0)
    assert short.kernel_name(p, 1) == "bch_nms_rc" == short.kernel_name(p, 64 * sms)
    assert short.kernel_name(p, 1_000_000) == "bch_nms_jit + bch_nms_rc"
    assert short.kernel_name(B.params(12, 0.78, msg=B.MSG_FP16), 1_000_000) == "bch_nms_jit"
    assert long_.kernel_name(p, 1_000_000) == "bch_nms_rc"
    assert plain.kernel_name(p0, 10_000) == "bch_plain_rc" and plain.kernel_info(n_autos=0) == "jit"
    # the launches of a decode are those of the named kernels
    for code, par, F, P in ((short, p, 50, 3), (short, p, 60_000, 3), (long_, p, 20_000, 3), (plain, p0, 50, 0)):
        name, n0 = code.kernel_name(par, F), B.kernel_launches()
        _decode(code, F, P)
        drawn = 1  # gen_frames
        assert B.kernel_launches() - n0 == drawn + len(name.split(" + ")), name
    monkeypatch.setenv("BCHDEC_NMS_KERNEL", "generic")
    assert short.kernel_name(p, 1) == "nms_enhanced_kernel" and plain.kernel_name(p0, 1) == "nms_plain_kernel"
    with pytest.raises(B.BchError):
        short.kernel_name(p, 0)
