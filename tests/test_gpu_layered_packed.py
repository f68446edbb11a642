"""Layered sum-product with thread slots end to end in a warp (narrow codes, several codewords to an SM):
every codeword's arithmetic is its own, so all batch sizes agree bit for bit, and a small one with
the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, rel_err
from tests.test_gpu_flood_packed import CODES
from tests.test_gpu_flood_shapes import decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("X", [80.0, 6.0])
@pytest.mark.parametrize("form", ["layered_f32", "layered_f16"])
@pytest.mark.parametrize("name", ["z3", "z5_wide", "z9_many_rows", "z20", "z36"])
def test_batches_agree(cuda_dev, name, form, X):
    B, Z = CODES[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    sms = torch.cuda.get_device_properties(cuda_dev).multi_processor_count
    rng = np.random.default_rng(15)
    n = 2 * sms + 40  # two and three codewords to an SM
    L = (2.5 + 2.2 * rng.standard_normal((40 * sms + 5, code.N))).astype(np.float32)
    for T in (1, 2):
        app, bits, iters = decode(code, form, L[:n].copy(), cuda_dev, max_iter=T, early_exit=0, phi_clamp=X)
        if form == "layered_f32" and X == 80.0:
            ref, _, _ = oc.spa_layered(L[:n], T, early_exit=False, X=X)
            assert rel_err(app, ref).max() <= FP32_TOL, T
        assert np.array_equal(bits, app < 0) and (iters == T).all()
    big = decode(code, form, L, cuda_dev, max_iter=9, phi_clamp=X)
    if name == "z3":
        assert len(set(big[2].tolist())) > 1  # codewords end in different iterations
    for m in (1, sms, sms + 1, n, 4 * sms, 10 * sms):
        for a, b in zip(decode(code, form, L[:m].copy(), cuda_dev, max_iter=9, phi_clamp=X), big):
            assert np.array_equal(a, b[:m]), m
