"""Layered decoders at the edges of their forms: every check-row degree class, slots of Z around the
warp size; sum-product with one codeword per thread and (FP16 messages, rows up to degree 8,
large batches) two; int8 min-sum with and without its offset table, bit-exact."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, assert_binary16_close, binary16_band, rel_err
from tests.test_gpu_flood_shapes import CODES, base_of, decode

pytestmark = pytest.mark.gpu

# (two codewords per thread need more codewords per SM than single slots fit: Z = 81, N = 1944)
ALL = dict(CODES, z81=(base_of([4, 4, 5, 5, 6, 6, 7, 7, 8, 8, 8, 3], 24, 81, 6), 81))


@pytest.mark.parametrize("form", ["layered_f32", "layered_f16"])
@pytest.mark.parametrize("name", list(ALL))
def test_against_oracle_and_across_forms(cuda_dev, name, form):
    B, Z = ALL[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    n_small, n_big = 40, 152 * 24 + 5
    rng = np.random.default_rng(8)
    L = (2.5 + 2.2 * rng.standard_normal((n_big, code.N))).astype(np.float32)  # noisy all-zero codewords
    L[::7, ::5] = 0.0
    for T in (1, 2):
        app, bits, iters = decode(code, form, L[:n_small].copy(), cuda_dev, max_iter=T, early_exit=0)
        if form == "layered_f32":
            ref, _, _ = oc.spa_layered(L[:n_small], T, early_exit=False)
            assert rel_err(app, ref).max() <= FP32_TOL, (name, T)
        elif T == 1:
            ref, band = binary16_band(oc, True, L[:400], 1, 8)
            app, _, _ = decode(code, form, L[:400].copy(), cuda_dev, max_iter=T, early_exit=0)
            assert_binary16_close(app, ref, band, strict=False, what=name)
        assert np.array_equal(bits, (app[:n_small] < 0)) and (iters == T).all()
    # each codeword's arithmetic is its own: the same, bit for bit, in a large batch with refills
    small = decode(code, form, L[:n_small].copy(), cuda_dev, max_iter=9)
    big = decode(code, form, L, cuda_dev, max_iter=9)
    for a, b in zip(small, big):
        assert np.array_equal(a, b[:n_small]), name


# (a code whose offset table does not fit beside a thread slot)
DENSE = dict(ALL, no_table=(base_of([16] * 16, 32, 256, 9), 256))


@pytest.mark.parametrize("sat", [(31, 127), (31, 40)])  # the posterior's saturation cannot / can bind
@pytest.mark.parametrize("name", list(DENSE))
def test_int8_bit_exact(cuda_dev, name, sat):
    B, Z = DENSE[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    n_small, n_big = 41, 152 * 24 + 5
    rng = np.random.default_rng(9)
    q = np.clip(np.rint(5 + 5 * rng.standard_normal((n_big, code.N))), -31, 31).astype(np.int8)
    q[::7, ::5] = 0
    kw = dict(max_iter=6, msg_sat=sat[0], app_sat=sat[1])
    a, b, i = oc.nms_layered(q[:n_small], 6, early_exit=True, msg_sat=sat[0], app_sat=sat[1])
    small = decode(code, "layered_i8", q[:n_small].copy(), cuda_dev, **kw)
    big = decode(code, "layered_i8", q, cuda_dev, **kw)
    for got in (small, [x[:n_small] for x in big]):
        assert np.array_equal(got[0].astype(np.int32), a) and np.array_equal(got[1], b) and np.array_equal(got[2], i)


@pytest.mark.parametrize("form", ["flood_f32", "flood_f16", "layered_f32", "layered_f16", "layered_i8"])
def test_batches_around_the_number_of_sms(cuda_dev, form):
    """Up to one codeword per SM needs no scratch, up to one per slot no work counter: at each edge
    every codeword is decoded once, as in a larger batch."""
    sms = torch.cuda.get_device_properties(cuda_dev).multi_processor_count
    code = ldpc.Code(*CODES["to12"])
    rng = np.random.default_rng(10)
    L = (2.5 + 2.2 * rng.standard_normal((40 * sms, code.N))).astype(np.float32)
    big = decode(code, form, L, cuda_dev, max_iter=7)
    for n in (1, 2, sms - 1, sms, sms + 1, 2 * sms + 1, 3 * sms):
        for a, b in zip(decode(code, form, L[:n].copy(), cuda_dev, max_iter=7), big):
            assert np.array_equal(a, b[:n]), (form, n)
