"""Two-SM cluster decoder with rows and columns end to end over its threads (widths that leave many lanes
of whole warps idle): every row and column degree class, pairs with and without a partner, quads."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, assert_binary16_close, binary16_band, rel_err
from tests.test_gpu_flood_shapes import base_of, decode

pytestmark = pytest.mark.gpu

CODES = {
    "narrow_z34": (base_of([2, 3, 4, 5, 6, 7, 8, 8] * 8, 72, 34, 31), 34),
    "to12_z68": (base_of([4, 9, 10, 11, 12, 12, 8, 7] * 8, 80, 68, 32), 68),
    "wide_z65": (base_of([3, 13, 16, 17, 24, 25, 32, 12] * 6, 72, 65, 33), 65),
    "wide_z36": (base_of([16] * 56, 112, 36, 34), 36),
    "one_group_z621": (base_of([13, 14, 15, 16] * 2, 17, 621, 35), 621),
}


@pytest.mark.parametrize("form", ["cluster_f32", "cluster_f16"])
@pytest.mark.parametrize("name", list(CODES))
def test_against_oracle(cuda_dev, name, form):
    B, Z = CODES[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    n = 160  # more codewords than clusters
    rng = np.random.default_rng(16)
    L = (2.5 + 2.2 * rng.standard_normal((n, code.N))).astype(np.float32)
    L[::7, ::5] = 0.0
    for T in (1, 2):
        app, bits, iters = decode(code, form, L, cuda_dev, max_iter=T, early_exit=0)
        if form == "cluster_f32":
            ref, _, _ = oc.spa_flood(L, T, early_exit=False)
            assert rel_err(app, ref).max() <= FP32_TOL, T
        elif T == 1:
            ref, band = binary16_band(oc, False, L, T, 4)
            assert_binary16_close(app, ref, band, strict=True)
        assert np.array_equal(bits, app < 0) and (iters == T).all()
    # early exit with refills, channel values on a 16-byte boundary or not: the same bits
    odd = torch.empty(L.size + 1, device=cuda_dev)[1:].view(n, code.N)
    odd.copy_(torch.from_numpy(L))
    a = ldpc.decode(code, ldpc.params_for(form, max_iter=9), odd, app=True)
    b = ldpc.decode(code, ldpc.params_for(form, max_iter=9), torch.from_numpy(L).to(cuda_dev), app=True)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
