"""The decoding work a user of this library has it do, as cases that can be timed and compared.

A case is one pass through a public entry point of ``paper_1812_06545_gb300.ldpc``: a batch
decode of device LLRs, one mixed-code launch, a host-to-host decode over several streams, or
a burst of requests to a serving session.  Codes, batch sizes, Eb/N0 and iteration limits are
those of the repository's own workloads (``inputs.WORKLOADS``, the mixed-code family at its
operating points, the frame lengths of the paper's figures), with ragged sizes among them.

Fields of a case:
  api         batch | multi | host | session
  form        a form of ``ldpc.FORMS`` (schedule, rule, message type)
  code        a committed code, or "family" (the 12 mixed codes; api multi and session)
  n           codewords (api session: requests, each of 1..512 codewords)
  ebn0        Eb/N0 in dB (family: offset from each code's operating point)
  max_iter, early_exit, app   decode options; app asks for the posterior LLRs
  llr         f32 | i8 (already quantised, layered min-sum only)
"""
import math

import numpy as np
import torch

from paper_1812_06545_gb300 import inputs as I
from paper_1812_06545_gb300 import ldpc

POOL = 64  # distinct transmitted codewords per code; every received frame has its own noise


def _case(name, api, form, code, n, ebn0, max_iter=20, early_exit=True, app=False, llr="f32"):
    c = dict(api=api, form=form, code=code, n=n, ebn0=ebn0, max_iter=max_iter, early_exit=early_exit, app=app,
             llr=llr)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one received frame at a time: a control channel, a link-level debugger
        _case("one_frame_f32", "batch", "flood_f32", "qc12x24_z27_s1", 1, 2.5),
        # a short latency-bound batch with soft output (an outer receiver loop), fixed iterations
        _case("latency_n648_b128_app", "batch", "flood_f32", "qc12x24_z27_s1", 128, 2.0, 10, False, True),
        # a point in the middle of the headline Eb/N0 sweep
        _case("flood_f32_n1944_b8192", "batch", "flood_f32", "qc12x24_z81_s2", 8192, 1.75),
        # the same code with half-precision messages, in the waterfall
        _case("flood_f16_n1944_b8192", "batch", "flood_f16", "qc12x24_z81_s2", 8192, 2.25),
        # a high-rate code (rows of about 20 edges), a ragged batch, soft output
        _case("flood_f32_r56_b3001_app", "batch", "flood_f32", "qc4x24_z81_s51", 3001, 3.75, 6, False, True),
        # the layered schedule on the headline code: the best error rate per iteration
        _case("layered_f32_n1944_b8192", "batch", "layered_f32", "qc12x24_z81_s2", 8192, 2.0),
        # the paper's setting: a few fixed layered iterations, 2^24 coded bits
        _case("layered_f16_n2304_b7281", "batch", "layered_f16", "qc12x24_z96_s9", 7281, 2.0, 5, False),
        # high-throughput fixed-point decoding of a high-rate link
        _case("layered_i8_r56_b65536", "batch", "layered_i8", "qc4x24_z81_s3", 65536, 4.0, 10),
        # fixed-point front end that quantises by itself, long frames, odd batch
        _case("layered_i8_n4000_b4193", "batch", "layered_i8", "qc10x20_z200_s10", 4193, 3.0, 10, True, False, "i8"),
        # a base station's mix of 12 codes at their operating points in one launch
        _case("mixed_f16_b20000", "multi", "flood_f16", "family", 20000, 0.0),
        # long codewords (one per two SMs)
        _case("large_f16_n26112_b2048", "batch", "flood_f16", "qc34x68_z384_s5", 2048, 2.0),
        # end to end from pinned host memory over four streams
        _case("host_f32_n1944_b16384", "host", "flood_f32", "qc12x24_z81_s2", 16384, 2.25),
    ]


# ------------------------------------------------------------------ sizes

def _sizes(code):
    B, Z = I.load_code(code)
    mb, nb = B.shape
    return nb * Z, int((B >= 0).sum()) * Z, (nb - mb) / nb


def _parts(case):
    """[(code, codewords)] of a case."""
    if case["code"] != "family":
        return [(case["code"], case["n"])]
    if case["api"] == "session":  # the requests' sizes and codes follow from their number
        rng = np.random.default_rng(case["n"])
        return [(I.MIXED_FAMILY[int(rng.integers(12))], int(round(512 ** rng.random()))) for _ in range(case["n"])]
    k = len(I.MIXED_FAMILY)
    return [(c, case["n"] // k + (i < case["n"] % k)) for i, c in enumerate(I.MIXED_FAMILY)]


def _updates(case):
    """Edge updates of a pass: codewords x edges x iterations.  With early exit about half of
    the allowed iterations are run near a code's operating point."""
    it = case["max_iter"] * (0.5 if case["early_exit"] else 1.0)
    return sum(n * _sizes(code)[1] for code, n in _parts(case)) * it


def work(case):
    """Channel values in, decisions, iteration counts and posteriors out; per edge update one
    message formed from the posterior (1), the check rule (sum-product: an exponential, two
    logarithms, 4 pair maps of 2 multiply-adds, a difference; min-sum: saturation, magnitude,
    two minima, scaling) and its addition to the posterior (1)."""
    per = 22 if "i8" not in case["form"] else 10
    b = sum(n * (_sizes(code)[0] * ((4 if case["llr"] == "f32" else 1) + 1 + (4 if case["app"] else 0)) + 4)
            for code, n in _parts(case))
    return {"bytes": float(b), "flops": float(per * _updates(case))}


_SINGLE = [c for c in I.CODE_SPECS if c != "qc34x68_z384_s5"]


def draw(rng):
    """One more case: any form and code, batches from one codeword to the largest listed work."""
    largest = max(c["n"] * _sizes(c["code"])[1] * c["max_iter"] for c in listed() if c["code"] != "family")
    kind = rng.choice(["batch"] * 8 + ["multi", "host", "session"])
    if kind in ("multi", "session"):
        form = rng.choice(["flood_f16", "flood_f32", "layered_i8"])
        n = int(round(math.exp(rng.uniform(math.log(60), math.log(20000))))) if kind == "multi" else rng.randint(4, 64)
        return _case(None, kind, form, "family", n, round(rng.uniform(0.0, 1.0), 2), 10 if form == "layered_i8" else 20)
    form = rng.choice(["flood_f32"] * 3 + ["flood_f16"] * 2 + ["layered_f32", "layered_f16", "layered_i8", "layered_i8"])
    code = rng.choice(_SINGLE)
    if kind == "batch" and form in ("flood_f32", "flood_f16") and rng.random() < 0.15:
        code = "qc34x68_z384_s5"
    early = rng.random() < 0.7
    max_iter = rng.choice([5, 10, 20]) if early else rng.randint(2, 10)
    top = largest / (_sizes(code)[1] * max_iter)
    n = int(round(math.exp(rng.uniform(0.0, math.log(min(65536.0, top))))))
    n = max(1, min(n | 1 if rng.random() < 0.5 else n, int(top)))
    rate = _sizes(code)[2]
    point = I.operating_points().get(code, 2.0 if rate < 0.6 else 4.0) + (0.75 if form == "layered_i8" else 0.0)
    llr = "i8" if form == "layered_i8" and kind == "batch" and rng.random() < 0.5 else "f32"
    app = kind == "batch" and rng.random() < 0.3
    return _case(None, kind, form, code, n, round(point + rng.uniform(-0.5, 0.5), 2), max_iter, early, app, llr)


# ------------------------------------------------------------------ inputs

def _llr(code, n, ebn0, seed):
    """Channel LLRs [n, N] on the GPU: random codewords over BPSK / AWGN, L = 2 y / sigma^2."""
    B, Z = I.load_code(code)
    mb, nb = B.shape
    c = I.encode(B, Z, I.info_bits(min(n, POOL), (nb - mb) * Z, seed))
    sent = torch.from_numpy(c).cuda()[torch.arange(n, device="cuda") % len(c)]
    s2 = I.sigma2_for(ebn0, (nb - mb) / nb)
    g = torch.Generator("cuda").manual_seed(seed * 2 + 1)
    y = torch.randn((n, nb * Z), generator=g, device="cuda")
    y.mul_(math.sqrt(s2)).add_(1.0).sub_(sent, alpha=2.0)
    return y.mul_(2.0 / s2)


def _pinned(*shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


class _Session:
    """A serving session, destroyed with its last reference."""

    def __init__(self):
        self.handle = ldpc.ldpc_session_create(ldpc.ldpc_session_default_config(hbm_budget_bytes=1 << 30))

    def __del__(self):
        ldpc.ldpc_session_destroy(self.handle)


def prepare(case, seed):
    family = case["code"] == "family"
    points = I.operating_points()
    codes, reqs = {}, []
    scale = 2.0
    for i, (name, n) in enumerate(_parts(case)):
        if name not in codes:
            codes[name] = ldpc.Code(*I.load_code(name))
        ebn0 = points[name] + case["ebn0"] if family else case["ebn0"]
        llr = _llr(name, n, ebn0, seed * 1000 + i)
        code = codes[name]
        if case["form"] == "layered_i8" and not family:
            scale = I.llr_scale_for(_sizes(name)[2], ebn0)
        if case["llr"] == "i8":
            llr = torch.clamp(torch.round(llr * scale), -31, 31).to(torch.int8)
        reqs.append((code, llr, n))
    params = ldpc.params_for(case["form"], max_iter=case["max_iter"], early_exit=int(case["early_exit"]),
                             llr_scale=scale)
    state = {"case": dict(case), "params": params, "codes": codes}
    if case["api"] == "batch":
        state["llr"] = reqs[0][1]
    elif case["api"] == "multi":
        out = [(torch.empty((n, c.N), dtype=torch.uint8, device="cuda"),
                torch.empty((n,), dtype=torch.int32, device="cuda")) for c, _, n in reqs]
        state["requests"] = [(c.handle, L, n, b, it, None) for (c, L, n), (b, it) in zip(reqs, out)]
        state["out"] = out
        state["ws"] = torch.empty(ldpc.ldpc_multi_workspace_size(), dtype=torch.uint8, device="cuda")
    else:
        host = []
        for c, L, n in reqs:
            h = _pinned(n, c.N, dtype=torch.float32)
            h.copy_(L)
            host.append((c, h, n, _pinned(n, c.N, dtype=torch.uint8), _pinned(n, dtype=torch.int32)))
        state["host"] = host
        if case["api"] == "session":
            state["session"] = _Session()
    return state


def run(state):
    case, p = state["case"], state["params"]
    if case["api"] == "batch":
        (code,) = state["codes"].values()
        return ldpc.decode(code, p, state["llr"], app=case["app"])
    if case["api"] == "multi":
        ldpc.ldpc_decode_multi(state["requests"], p, workspace=state["ws"], workspace_bytes=state["ws"].numel(),
                               stream=torch.cuda.current_stream())
        return state["out"]
    if case["api"] == "host":
        ((code, L, n, bits, iters),) = state["host"]
        ldpc.ldpc_decode_host(code.handle, p, L, n, bits, iters, n_streams=4, chunk_cw=4096)
        return bits, iters
    s = state["session"].handle
    ids = [ldpc.ldpc_session_submit(s, c.handle, p, L, n, bits, iters) for c, L, n, bits, iters in state["host"]]
    for rid in ids:
        status, _ = ldpc.ldpc_session_wait(s, rid, 60.0)
        if status != ldpc.LDPC_OK:
            raise RuntimeError(f"request {rid} ended with status {status}")
    return [torch.cat([h[k].reshape(-1) for h in state["host"]]) for k in (3, 4)]


# ------------------------------------------------------------------ the same in 64 bits

def _phi(x):
    return -torch.log(torch.tanh(0.5 * x))


def _check(q, X):
    """Sum-product messages of one block row from its Q [n, degree, Z] (phi domain): the sums
    over the other edges are formed directly, without a subtraction."""
    lo = math.log1p(2.0 / math.expm1(X))
    f = _phi(q.abs().clamp(lo, X))
    neg = q < 0
    sign = 1.0 - 2.0 * ((neg.sum(1, keepdim=True) - neg.long()) % 2).double()
    ex = torch.zeros_like(f)
    ex[:, 1:] += torch.cumsum(f, 1)[:, :-1]
    ex[:, :-1] += torch.flip(torch.cumsum(torch.flip(f, [1]), 1), [1])[:, 1:]
    return sign * _phi(ex).clamp(max=X)


def _spa(code, L, max_iter, early, layered, X=80.0):
    """Posteriors of the sum-product decoder in 64 bits (messages not rounded to 16 bits)."""
    B, Z = I.load_code(code)
    n, (mb, nb) = len(L), B.shape
    rows = [[(j, int(B[l, j])) for j in range(nb) if B[l, j] >= 0] for l in range(mb)]
    L = L.double().reshape(n, nb, Z)
    app, out = L.clone(), torch.empty_like(L)
    R = [torch.zeros((n, len(r), Z), dtype=torch.float64, device=L.device) for r in rows]
    at = torch.arange(n, device=L.device)

    def read(a, r):
        return torch.stack([torch.roll(a[:, j], -s, 1) for j, s in r], 1)

    for t in range(1, max_iter + 1):
        new = L.clone()
        for l, r in enumerate(rows):
            q = read(app, r) - R[l]
            R[l] = _check(q, X)
            if layered:
                q = q + R[l]
            for k, (j, s) in enumerate(r):
                if layered:
                    app[:, j] = torch.roll(q[:, k], s, 1)
                else:
                    new[:, j] += torch.roll(R[l][:, k], s, 1)
        if not layered:
            app = new
        if early and t < max_iter:
            bad = torch.zeros(len(app), dtype=torch.bool, device=L.device)
            for r in rows:
                bad |= ((read(app, r) < 0).sum(1) % 2 == 1).any(1)
            out[at[~bad]] = app[~bad]
            at, app, L, R = at[bad], app[bad], L[bad], [x[bad] for x in R]
            if not len(at):
                break
    out[at] = app
    return out.reshape(n, nb * Z)


def exact(case, seed):
    if case["api"] != "batch" or not case["app"] or case["form"] == "layered_i8" or _updates(case) > 1.5e9:
        return None  # decisions, counts and integer posteriors have no rounding
    L = _llr(case["code"], case["n"], case["ebn0"], seed * 1000)
    step = max(1, 40_000_000 // _sizes(case["code"])[1])
    app = [_spa(case["code"], L[a:a + step], case["max_iter"], case["early_exit"], "layered" in case["form"])
           for a in range(0, case["n"], step)]
    return None, None, torch.cat(app)
