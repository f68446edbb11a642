"""Flooding slot decoder with rows end to end in a warp: thread slots packed (large and middling batches
of narrow codes) and row groups spread (small ones).  Every codeword's arithmetic is its own, so all
batch sizes agree bit for bit, and a small one agrees with the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, assert_binary16_close, binary16_band, rel_err
from tests.test_gpu_flood_shapes import base_of, decode

pytestmark = pytest.mark.gpu

# widths that leave warps idle, all row degree classes and their neighbours in one warp
CODES = {
    "z3": (base_of([3, 3, 4, 5, 6, 7, 8, 8, 2, 2, 5, 5], 24, 3, 21), 3),
    "z5_wide": (base_of([9, 12, 13, 16, 17, 24, 25, 32, 8, 3], 40, 5, 22), 5),
    "z9_many_rows": (base_of([20, 21, 22] * 10 + [4] * 10, 80, 9, 23), 9),
    "z20": (base_of([20, 20, 21, 19], 24, 20, 24), 20),
    "z36": (base_of([6, 7, 7, 8, 8, 7, 6, 7, 7, 8, 8, 7], 24, 36, 25), 36),
    "z66_large": (base_of([15, 16] * 24, 96, 66, 26), 66),
}


@pytest.mark.parametrize("X", [80.0, 6.0])
@pytest.mark.parametrize("form", ["flood_f32", "flood_f16"])
@pytest.mark.parametrize("name", list(CODES))
def test_batches_agree(cuda_dev, name, form, X):
    B, Z = CODES[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    sms = torch.cuda.get_device_properties(cuda_dev).multi_processor_count
    rng = np.random.default_rng(13)
    n = 40
    L = (2.5 + 2.2 * rng.standard_normal((4 * sms if Z > 40 else 40 * sms + 5, code.N))).astype(np.float32)
    L[::7, ::5] = 0.0
    for T in (1, 2):
        app, bits, iters = decode(code, form, L[:n].copy(), cuda_dev, max_iter=T, early_exit=0, phi_clamp=X)
        if form == "flood_f32" and (T == 1 or X == 80.0):
            # (an erased value in a column of one check has Q = APP - R = 0 exactly from the second
            # iteration on, whose sign, and with X = 6 a message of phi(6), is rounding's to choose)
            ref, _, _ = oc.spa_flood(L[:n], T, early_exit=False, X=X)
            assert rel_err(app, ref).max() <= FP32_TOL, T
        elif form == "flood_f16" and T == 1:
            ref, band = binary16_band(oc, False, L[:n], 1, 4, X=X)
            assert_binary16_close(app, ref, band, strict=True)
        assert np.array_equal(bits, app < 0) and (iters == T).all()
    big = decode(code, form, L, cuda_dev, max_iter=9, phi_clamp=X)
    if name == "z3":
        assert len(set(big[2].tolist())) > 1  # codewords end in different rounds
    for m in (1, n, sms + 1, 2 * sms, 4 * sms, 10 * sms):
        if m < len(L):
            for a, b in zip(decode(code, form, L[:m].copy(), cuda_dev, max_iter=9, phi_clamp=X), big):
                assert np.array_equal(a, b[:m]), m


def test_mixed_widths(cuda_dev):
    """Narrow codes beside one of whole warps in one launch, each as alone."""
    p = ldpc.params_for("flood_f16", max_iter=7)
    codes = [ldpc.Code(*CODES[k]) for k in ("z3", "z36", "z20")] + [ldpc.Code(base_of([5, 6, 7, 8], 12, 64, 27), 64)]
    rng = np.random.default_rng(14)
    reqs, outs, alone = [], [], []
    for code, n in zip(codes, (3000, 700, 1, 300)):
        L = torch.from_numpy((2.5 + 2.2 * rng.standard_normal((n, code.N))).astype(np.float32)).to(cuda_dev)
        alone.append(ldpc.decode(code, p, L, app=True))
        outs.append([torch.empty_like(x) for x in alone[-1]])
        reqs.append((code.handle, L, n, *outs[-1]))
    ldpc.ldpc_decode_multi(reqs, p, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    for a, b in zip(alone, outs):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
