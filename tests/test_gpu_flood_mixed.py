"""Mixed launches of the flooding slot decoder whose codes leave little shared memory: every request
decodes as it does alone, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1812_06545_gb300 import ldpc
from tests.test_flood_plan_cpu import PAIRS, base_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f16,big,small", PAIRS)
def test_pairs_as_alone(cuda_dev, f16, big, small):
    codes = [ldpc.Code(base_of(*s, seed=i), s[3]) for i, s in enumerate((big, small))]
    p = ldpc.params_for("flood_f16" if f16 else "flood_f32", max_iter=6)
    rng = np.random.default_rng(12)
    reqs, outs, alone = [], [], []
    for code, n in zip(codes, (400, 5000)):
        L = torch.from_numpy((2.5 + 2.2 * rng.standard_normal((n, code.N))).astype(np.float32)).to(cuda_dev)
        alone.append(ldpc.decode(code, p, L, app=True))
        out = [torch.empty_like(x) for x in alone[-1]]
        outs.append(out)
        reqs.append((code.handle, L, n, *out))
    ldpc.ldpc_decode_multi(reqs, p, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    for a, b in zip(alone, outs):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
