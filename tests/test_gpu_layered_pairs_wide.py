"""Layered int8 min-sum where 1024 threads hold a thread slot more than 896 (rows of 9 to 16 edges): one and
two thread slots of Z up to 512, and the batch sizes that choose between the two forms, bit-exact."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.test_gpu_flood_shapes import base_of, decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sat", [(31, 127), (31, 40)])
@pytest.mark.parametrize("Z", [250, 449, 480, 512])
def test_bit_exact(cuda_dev, Z, sat):
    B = base_of([9, 12, 16, 3], 18, Z, 41)
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    rng = np.random.default_rng(17)
    q = np.clip(np.rint(5 + 5 * rng.standard_normal((1300, code.N))), -31, 31).astype(np.int8)
    kw = dict(max_iter=5, msg_sat=sat[0], app_sat=sat[1])
    a, b, i = oc.nms_layered(q[:60], 5, early_exit=True, msg_sat=sat[0], app_sat=sat[1])
    big = decode(code, "layered_i8", q, cuda_dev, **kw)
    for n in (60, 400, 1000, 1300):
        got = decode(code, "layered_i8", q[:n].copy(), cuda_dev, **kw)
        assert all(np.array_equal(x, y[:n]) for x, y in zip(got, big)), n
    assert np.array_equal(big[0][:60].astype(np.int32), a) and np.array_equal(big[1][:60], b)
    assert np.array_equal(big[2][:60], i)
