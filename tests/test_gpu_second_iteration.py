"""Sum-product messages read back: the second iteration against the oracle, for binary16 messages and for small
clamps, which the one-iteration checks of the shape tests do not reach (messages start at zero), at
every row degree class of every on-chip decoder; and the instances on either side of the clamp from
which the upper clamp of |Q| is left out."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1812_06545_gb300 import ldpc
from tests.gpu_helpers import FP32_TOL, assert_binary16_close, binary16_band, rel_err
from tests.test_gpu_cluster_spread import CODES as SPREAD
from tests.test_gpu_flood_shapes import CODES, decode

pytestmark = pytest.mark.gpu

N_CW = 300
FORMS = {"flood": ["narrow", "to12", "wide", "z1", "z96"], "layered": ["narrow", "to12", "wide", "z1", "z96"],
         "cluster": ["narrow", "to12", "wide", "narrow_z34", "to12_z68", "wide_z65"]}
CASES = [(f, name) for f in FORMS for name in FORMS[f]]


def setup(kind, name):
    B, Z = (SPREAD if name in SPREAD else CODES)[name]
    code, oc = ldpc.Code(B, Z), O.QCCode(B, Z)
    L = (2.5 + 2.2 * np.random.default_rng(19).standard_normal((N_CW, code.N))).astype(np.float32)
    return code, oc, L


@pytest.mark.parametrize("X", [80.0, 6.0])
@pytest.mark.parametrize("kind,name", CASES)
def test_binary16(cuda_dev, kind, name, X):
    code, oc, L = setup(kind, name)
    app, bits, _ = decode(code, kind + "_f16", L, cuda_dev, max_iter=2, early_exit=0, phi_clamp=X)
    ref, band = binary16_band(oc, kind == "layered", L, 2, 8 if kind == "layered" else 4, X=X)
    assert_binary16_close(app, ref, band, strict=False, what=name)
    assert np.array_equal(bits, app < 0)


@pytest.mark.parametrize("kind,name", CASES)
def test_fp32_small_clamp(cuda_dev, kind, name):
    code, oc, L = setup(kind, name)
    app, _, _ = decode(code, kind + "_f32", L, cuda_dev, max_iter=2, early_exit=0, phi_clamp=6.0)
    orc = oc.spa_layered if kind == "layered" else oc.spa_flood
    ref, _, _ = orc(L, 2, early_exit=False, X=6.0)
    # (a clamped message jumps by 2 phi(X) where Q passes zero: codewords that the oracle itself moves by a
    # tenth of the tolerance when its input moves by FP32 rounding have such a Q)
    noise = 3e-7 * np.random.default_rng(20).standard_normal((4, *L.shape))
    moved = [orc((L * (1 + e)).astype(np.float32), 2, early_exit=False, X=6.0)[0] for e in noise]
    firm = np.max([rel_err(m, ref).max(axis=1) for m in moved], axis=0) < 0.1 * FP32_TOL
    assert firm.sum() >= 0.95 * N_CW
    assert rel_err(app[firm], ref[firm]).max() <= FP32_TOL


@pytest.mark.parametrize("msg", ["f32", "f16"])
@pytest.mark.parametrize("kind,name", CASES)
def test_clamp_left_out(cuda_dev, kind, name, msg):
    code, oc, L = setup(kind, name)
    L = 0.25 * L
    at = decode(code, f"{kind}_{msg}", L, cuda_dev, max_iter=2, early_exit=0, phi_clamp=40.0)
    below = decode(code, f"{kind}_{msg}", L, cuda_dev, max_iter=2, early_exit=0,
                   phi_clamp=float(np.nextafter(np.float32(40), np.float32(0))))
    small = np.abs(at[0]).max(axis=1) < 35.0  # (the lower clamp, X itself, is not reached)
    assert small.sum() > N_CW // 2
    assert np.array_equal(at[0][small], below[0][small]) and np.array_equal(at[1][small], below[1][small])
