"""Launch sizing of the flooding slot decoder, on the CPU: codes that are each served alone are
served together, whatever their sizes, and no code's layout leaves the shared memory asked for."""
import os
import subprocess

import numpy as np
import pytest

from paper_1812_06545_gb300 import _build

LIMIT = 227 * 1024


def base_of(mb, nb, blocks, Z, seed):
    """Random base matrix with the given number of blocks, at least two to a row and one to a column."""
    rng = np.random.default_rng(seed)
    B = -np.ones((mb, nb), np.int64)
    for j in range(nb):
        B[j % mb, j] = rng.integers(Z)
    for l in range(mb):
        while (B[l] >= 0).sum() < 2:
            B[l, rng.integers(nb)] = rng.integers(Z)
    while (B >= 0).sum() < blocks:
        l, j = rng.integers(mb), rng.integers(nb)
        if (B[l] >= 0).sum() < 32:
            B[l, j] = rng.integers(Z)
    return B


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "flood_plan_host")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([_build.nvcc(), "-std=c++17", "-O1", *_build.ARCH, "-I", _build.CSRC, "-I", _build.INCLUDE,
                    os.path.join(here, "flood_plan_host.cu"), "-o", exe], check=True)

    def run(codes, launches):
        """codes: (base, Z); launches: (f16, [(code, codewords)]) -> one list of ints per launch."""
        lines = [f"C {B.shape[0]} {B.shape[1]} {Z} " + " ".join(map(str, B.ravel())) for B, Z in codes]
        lines += [f"L {f16} {len(r)} " + " ".join(f"{c} {n}" for c, n in r) for f16, r in launches]
        out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
        return [list(map(int, x.split())) for x in out.splitlines()]

    return run


def check(launch, row):
    served, status, smem, threads, ctas, V, form = row[:7]
    if not served:
        return False
    assert status == 0, (launch, row)
    assert smem <= LIMIT and threads <= 768 and 1 <= ctas <= 152, (launch, row)
    for g in range(7, len(row), 6):
        Z, G, W, TPG, K, end = row[g:g + 6]
        assert G >= 1 and G % K == 0 and G // K * TPG <= threads and end <= smem, (launch, row)
        # K thread slots' rows (form 2: of all row groups) end to end over whole warps, a warp's lane to
        # each of their codewords
        lanes = K * Z * (W if form == 2 else 1)
        assert TPG == (lanes + 31) // 32 * 32 * (1 if form == 2 else W), (launch, row)
        assert K * V <= 32 and (form or K == 1) and (form != 2 or V == 1), (launch, row)
    return True


# a code that nearly fills an SM beside one of many small slots, or of many blocks
PAIRS = [
    (0, (5, 20, 62, 352), (4, 16, 48, 54)),
    (0, (10, 20, 70, 320), (6, 24, 72, 27)),
    (0, (4, 24, 86, 512), (34, 68, 400, 16)),
    (1, (16, 48, 166, 27), (12, 48, 96, 8)),
    (1, (8, 48, 159, 112), (7, 20, 70, 8)),
]


@pytest.mark.parametrize("f16,big,small", PAIRS)
def test_named_pairs(plan, f16, big, small):
    codes = [(base_of(*s, seed=i), s[3]) for i, s in enumerate((big, small))]
    launches = [(f16, [(0, n), (1, m)]) for n in (1, 3000) for m in (1, 500, 20000)]
    served = [check(x, row) for x, row in zip(launches, plan(codes, launches))]
    assert all(served)


def test_random_launches(plan):
    rng = np.random.default_rng(1)
    codes = []
    while len(codes) < 160:
        mb = int(rng.integers(3, 47))
        nb = int(min(128, mb * rng.uniform(1.4, 5) + 1))
        Z = int(np.exp(rng.uniform(0, np.log(640))))
        blocks = int(min(1000, 30 * mb, max(nb, 2 * mb) * rng.uniform(1.2, 4)))
        codes.append((base_of(mb, nb, min(blocks, mb * nb // 2), Z, len(codes)), Z))
    launches = []
    for _ in range(6000):
        k = int(rng.choice([1, 2, 2, 3, 6]))
        launches.append((int(rng.integers(2)), [(int(c), int(np.exp(rng.uniform(0, 11))))
                                                for c in rng.choice(len(codes), k, replace=False)]))
    n = sum(check(x, row) for x, row in zip(launches, plan(codes, launches)))
    assert n > 2000  # launches of codes that are all served alone
