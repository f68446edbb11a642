"""Flooding slot decoder at the edges of its forms: every check-row degree class (2..8 exact,
up to 12, 16, 24, 32), column degrees 1..9, slots of Z around the warp size, one codeword per
thread (small batches, spread over row groups) and two (large batches with refills)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, assert_binary16_close, binary16_band, rel_err

pytestmark = pytest.mark.gpu


def base_of(degrees, nb, Z, seed):
    """Random base matrix with the given row degrees, no empty column; column weights uneven."""
    rng = np.random.default_rng(seed)
    while True:
        B = -np.ones((len(degrees), nb), np.int32)
        for l, d in enumerate(degrees):
            w = 1.0 / (1.0 + np.arange(nb))  # a few heavy columns
            for j in rng.choice(nb, d, replace=False, p=w / w.sum()):
                B[l, j] = rng.integers(Z)
        for j in np.flatnonzero((B >= 0).sum(0) == 0):  # move an edge of the heaviest column there
            l = rng.choice(np.flatnonzero(B[:, 0] >= 0))
            B[l, j], B[l, 0] = B[l, 0], -1
        if ((B >= 0).sum(0) > 0).all():
            return B


CODES = {
    "narrow": (base_of([2, 3, 4, 5, 6, 7, 8, 8], 11, 31, 1), 31),
    "to12": (base_of([2, 3, 5, 8, 9, 10, 11, 12, 12], 14, 33, 2), 33),
    "wide": (base_of([4, 12, 13, 16, 17, 24, 25, 32], 34, 32, 3), 32),
    "z1": (base_of([3, 3, 4, 9], 12, 1, 4), 1),
    "z96": (base_of([20, 21, 19], 24, 96, 5), 96),
}


def decode(code, form, L, dev, **kw):
    bits, iters, app = ldpc.decode(code, ldpc.params_for(form, **kw), torch.from_numpy(L).to(dev), app=True)
    torch.cuda.synchronize()
    return app.cpu().numpy(), bits.cpu().numpy(), iters.cpu().numpy()


@pytest.mark.parametrize("form", ["flood_f32", "flood_f16"])
@pytest.mark.parametrize("name", list(CODES))
def test_against_oracle_and_across_forms(cuda_dev, name, form):
    B, Z = CODES[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    n_small, n_big = 40, 152 * 24 + 5
    rng = np.random.default_rng(7)
    L = (2.5 + 2.2 * rng.standard_normal((n_big, code.N))).astype(np.float32)  # noisy all-zero codewords
    L[::7, :: 5] = 0.0
    for T in (1, 2):
        app, bits, iters = decode(code, form, L[:n_small].copy(), cuda_dev, max_iter=T, early_exit=0)
        if form == "flood_f32":
            ref, _, _ = oc.spa_flood(L[:n_small], T, early_exit=False)
            assert rel_err(app, ref).max() <= FP32_TOL, (name, T)
        elif T == 1:
            ref, band = binary16_band(oc, False, L[:n_small], 1, 4)
            assert_binary16_close(app, ref, band, strict=True, what=name)
        assert np.array_equal(bits, app < 0) and (iters == T).all()
    # each codeword's arithmetic is its own: the same, bit for bit, two to a thread with refills
    small = decode(code, form, L[:n_small].copy(), cuda_dev, max_iter=9)
    big = decode(code, form, L, cuda_dev, max_iter=9)
    for a, b in zip(small, big):
        assert np.array_equal(a, b[:n_small]), name


@pytest.mark.parametrize("form", ["cluster_f32", "cluster_f16"])
@pytest.mark.parametrize("name", list(CODES))
def test_cluster_against_oracle(cuda_dev, name, form):
    """Two rows per thread (odd Z: a last row without a partner), columns in quads where Z is a
    multiple of 4 (channel values on a 16-byte boundary or not)."""
    B, Z = CODES[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    n = 200  # more codewords than clusters
    rng = np.random.default_rng(11)
    L = (2.5 + 2.2 * rng.standard_normal((n, code.N))).astype(np.float32)
    L[::7, ::5] = 0.0
    for T in (1, 2):
        app, bits, iters = decode(code, form, L, cuda_dev, max_iter=T, early_exit=0)
        if form == "cluster_f32":
            ref, _, _ = oc.spa_flood(L, T, early_exit=False)
            assert rel_err(app, ref).max() <= FP32_TOL, (name, T)
        elif T == 1:
            ref, band = binary16_band(oc, False, L, 1, 4)
            assert_binary16_close(app, ref, band, strict=True, what=name)
        assert np.array_equal(bits, app < 0) and (iters == T).all()
    odd = torch.empty(L.size + 1, device=cuda_dev)[1:].view(n, code.N)
    odd.copy_(torch.from_numpy(L))
    a = ldpc.decode(code, ldpc.params_for(form, max_iter=9), odd, app=True)
    b = ldpc.decode(code, ldpc.params_for(form, max_iter=9), torch.from_numpy(L).to(cuda_dev), app=True)
    for x, y in zip(a, b):
        assert torch.equal(x, y), name
