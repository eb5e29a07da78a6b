"""The work that users of this prover have it do, as measurable cases.

A case is one pass through the public Python binding (``Context`` and its
methods): a proof of one form, a proof of each form from host buffers, a
commitment with its proof and opening, or a prepared batch.  Witnesses are
satisfying ones with uniform field elements, made on the GPU from the seed.
Proofs, quotients and openings are byte strings that two correct provers make
equal, so there is nothing to round.

Work is counted in field multiplications (``costs.algorithmic_mulmods``), each
as the 136 32-bit multiply-adds of a schoolbook Montgomery product on eight
limbs, plus the SHA-256 compressions where hashing is part of the call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_16146_gb300 import costs, workloads, zc

R = 0x73EDA753299D7D483339D80809A1D80553BDA402FFFE5BFEFFFFFFFF00000001
FLOPS_PER_MULMOD = 2 * 136
OPS_PER_COMPRESSION = 64 * 24
PCS_QUERIES = 189
LARGEST_MULMODS = 2.3e9  # no drawn case does more than the largest listed one

_ctx = None


def _context():
    """One context for the process, as a proving service keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = zc.Context(0, max_n=24, max_d=32)
    return _ctx


def listed():
    P, G = zc.ZC_GATE_PLONK, zc.ZC_GATE_PRODUCT
    return [
        # the smallest standard circuit: launches, transcript and challenges count
        {"name": "sc_plonk_n12", "kind": "sumcheck", "gate": P, "n": 12, "d": 3, "roots": True},
        # a small circuit proved with the eq-factored messages, column roots inside the call
        {"name": "sc_eq_plonk_n17", "kind": "sumcheck_eq", "gate": P, "n": 17, "d": 3, "roots": False},
        # the headline circuit's SumCheck proof
        {"name": "sc_plonk_n22", "kind": "sumcheck", "gate": P, "n": 22, "d": 3, "roots": True},
        # a high-degree custom gate, as in the degree sweep and the served mix
        {"name": "sc_product_d8_n20", "kind": "sumcheck", "gate": G, "n": 20, "d": 8, "roots": True},
        # g1 g2 + g3 + g4 + g5, of the paper's polynomials, at a large odd size
        {"name": "sc_sum_d2_m3_n21", "kind": "sumcheck", "gate": zc.gate_sum(3), "n": 21, "d": 2, "roots": True},
        # the smallest standard circuit in the NTT form
        {"name": "ntt_plonk_n12", "kind": "ntt", "gate": P, "n": 12, "d": 3, "roots": True, "domain": 0},
        # a medium circuit in the NTT form, column roots inside the call
        {"name": "ntt_plonk_n20", "kind": "ntt", "gate": P, "n": 20, "d": 3, "roots": False, "domain": 0},
        # the headline circuit's NTT proof, the largest case
        {"name": "ntt_plonk_n22", "kind": "ntt", "gate": P, "n": 22, "d": 3, "roots": True, "domain": 0},
        # a degree whose quotient needs 5N points: the step-radix domain
        {"name": "ntt_product_d6_5N_n19", "kind": "ntt", "gate": G, "n": 19, "d": 6, "roots": True,
         "domain": zc.domain_word(2, 0)},
        # both forms through the C ABI from pinned host columns, proofs and quotient back on the host
        {"name": "host_step_plonk_n20", "kind": "host_step", "gate": P, "n": 20, "d": 3, "roots": True, "domain": 0},
        # commit, prove with the commitment's root, replay for the point, open
        {"name": "pcs_plonk_n18", "kind": "pcs", "gate": P, "n": 18, "d": 3},
        # many uneven instances of both forms in one prepared graph
        {"name": "batch_24_n10_17", "kind": "batch", "count": 24, "n_lo": 10, "n_hi": 17, "sampler": 3,
         "ntt_every": 4},
    ]


def _random_case(rng):
    kind = rng.choice(["sumcheck", "sumcheck", "sumcheck", "sumcheck_eq", "ntt", "ntt", "ntt", "host_step", "pcs",
                       "batch"])
    if kind == "batch":
        lo = rng.randint(8, 12)
        return {"kind": kind, "count": rng.randint(8, 32), "n_lo": lo, "n_hi": rng.randint(lo + 2, 17),
                "sampler": rng.randint(1, 1 << 20), "ntt_every": rng.randint(2, 6)}
    gate = zc.ZC_GATE_PLONK
    d, m = 3, 0
    family = rng.random()
    if kind != "pcs" and family > 0.5:
        d = rng.choice([2, 3, 4, 5, 6, 7, 8, 11, 16, 32])
        gate = zc.ZC_GATE_PRODUCT
        if family > 0.8:
            d, m = rng.randint(2, 4), rng.randint(0, 3)
            gate = zc.gate_sum(m)
    if kind == "pcs":
        return {"kind": kind, "gate": gate, "n": rng.randint(10, 20), "d": d}
    case = {"kind": kind, "gate": gate, "n": rng.randint(10, 24), "d": d, "roots": rng.random() < 0.5}
    if kind in ("ntt", "host_step"):
        k = max(0, (d - 2).bit_length())  # 2^k N is the smallest power of two that holds the quotient
        words = [0] + ([k] if k else []) + ([zc.domain_word(k - 1, 0)] if k > 1 and (1 << (k - 1)) + 1 >= d - 1 else [])
        case["domain"] = rng.choice(words)
        case["roots"] = case["roots"] or kind == "host_step"
    return case


def draw(rng):
    """A case of any kind and size above whose work and memory stay within the listed ones'."""
    while True:
        case = _random_case(rng)
        if case["kind"] == "batch":
            return case
        if case["kind"] == "host_step" and case["n"] > 20:
            continue
        if costs.ncols(case["gate"], case["d"]) << case["n"] > 8 << 22:
            continue
        if _mulmods(case) <= LARGEST_MULMODS:
            return case


# ------------------------------------------------------------------- work --

def _batch_shapes(case):
    out = []
    for i, (s, _) in enumerate(workloads.batched_instances(case["count"], case["sampler"], 0, case["n_lo"],
                                                           case["n_hi"])):
        out.append((s, zc.ZC_FORM_NTT if i % case["ntt_every"] == case["ntt_every"] - 1 else zc.ZC_FORM_SUMCHECK))
    return out


def _form_work(form, n, d, gate, domain, roots):
    """(mulmods, compressions, bytes) of one proof: columns read, proof and quotient written."""
    c, N = costs.ncols(gate, d), 1 << n
    M = zc.domain_size(n, d, domain) if form == "ntt" else 0
    comp = M / 2 + (0 if roots else c * N / 2)
    return costs.algorithmic_mulmods(form, n, d, gate, domain), comp, 32.0 * (c * N + M)


def _work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_form_work("ntt" if f == zc.ZC_FORM_NTT else "sumcheck", s.n, s.d, s.gate, 0, False)
                 for s, f in _batch_shapes(case)]
        return tuple(sum(x) for x in zip(*parts))
    n, d, gate = case["n"], case["d"], case["gate"]
    c, N = costs.ncols(gate, d), 1 << n
    if kind == "pcs":
        nc = min(n, 12)
        mul, comp, byts = _form_work("sumcheck", n, d, gate, 0, True)
        mul += 4 * c * (N / 2 * nc + N) + 2 * c * N
        return mul, comp + 2 * c * N, byts + zc.pcs_proof_size(n, c, PCS_QUERIES)
    if kind == "host_step":
        a = _form_work("sumcheck", n, d, gate, 0, True)
        b = _form_work("ntt", n, d, gate, case["domain"], True)
        return tuple(x + y for x, y in zip(a, b))
    return _form_work("ntt" if kind == "ntt" else "sumcheck", n, d, gate, case.get("domain", 0), case["roots"])


def _mulmods(case):
    return _work(case)[0]


def work(case):
    mul, comp, byts = _work(case)
    return {"bytes": byts, "flops": FLOPS_PER_MULMOD * mul + OPS_PER_COMPRESSION * comp}


# -------------------------------------------------------------- witnesses --
# Field elements as 16 rows of 16-bit limbs in int64; multiplication in
# Montgomery form, R = 2^256.

_P16 = [(R >> (16 * i)) & 0xFFFF for i in range(16)]
_PINV = (-pow(R, -1, 1 << 16)) & 0xFFFF
_R2 = [(pow(2, 512, R) >> (16 * i)) & 0xFFFF for i in range(16)]


def _carry(t):
    for i in range(t.shape[0] - 1):
        t[i + 1] += t[i] >> 16
        t[i] &= 0xFFFF
    return t


def _reduce(t):
    """t - r where t >= r (t below 2r, normalised limbs)."""
    p = torch.tensor(_P16, dtype=torch.int64, device=t.device)[:, None]
    s = _carry(t - p)
    return torch.where((s[-1] < 0)[None], t, s)


def _montmul(x, y, p):
    t = torch.zeros((33, x.shape[1]), dtype=torch.int64, device=x.device)
    for i in range(16):
        t[i:i + 16] += x * y[i]
    for i in range(16):
        t[i + 1] += t[i] >> 16
        t[i] &= 0xFFFF
        m = (t[i] * _PINV) & 0xFFFF
        t[i:i + 16] += p * m
        t[i + 1] += t[i] >> 16
    return _reduce(_carry(t[16:32]))


def _mul(x, y):
    p = torch.tensor(_P16, dtype=torch.int64, device=x.device)[:, None]
    r2 = torch.tensor(_R2, dtype=torch.int64, device=x.device)[:, None].expand(16, x.shape[1])
    return _montmul(_montmul(x, y, p), r2, p)


def _add(x, y):
    return _reduce(_carry(x + y))


def _neg(x):
    p = torch.tensor(_P16, dtype=torch.int64, device=x.device)[:, None]
    return torch.where((x == 0).all(0)[None], x, _carry(p - x))


def _uniform(count, gen):
    t = torch.randint(0, 1 << 16, (16, count), generator=gen, device="cuda", dtype=torch.int64)
    t[15] = torch.randint(0, R >> 240, (count,), generator=gen, device="cuda", dtype=torch.int64)
    return t


def _rows(gate, d, count, gen):
    """count rows of a satisfying witness: one limb array per column."""
    if gate == zc.ZC_GATE_PLONK:  # qC solved: the same distribution as c solved with qO nonzero
        qL, qR, qM, qO, a, b, c = (_uniform(count, gen) for _ in range(7))
        u = _mul(a, _add(qL, _mul(qM, b)))
        return [qL, qR, qM, qO, _neg(_add(u, _add(_mul(qR, b), _mul(qO, c)))), a, b, c]
    cols = [_uniform(count, gen) for _ in range(d)]
    if gate != zc.ZC_GATE_PRODUCT and gate >> 8 == 0:  # a bare product: one factor zero at every point
        at = torch.randint(0, d, (count,), generator=gen, device="cuda")
        return [x.masked_fill_((at == j)[None], 0) for j, x in enumerate(cols)]
    s = cols[0]
    for x in cols[1:]:
        s = _mul(s, x)
    if gate == zc.ZC_GATE_PRODUCT:
        return cols + [s]
    for _ in range((gate >> 8) - 1):
        cols.append(_uniform(count, gen))
        s = _add(s, cols[-1])
    return cols + [_neg(s)]


def _columns(gate, n, d, seed):
    """Device columns (uint8, 32 bytes per element) of a satisfying witness."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed % (1 << 62))
    N, step = 1 << n, 1 << 19
    out = [torch.empty(N * 32, dtype=torch.uint8, device="cuda") for _ in range(costs.ncols(gate, d))]
    for k in range(0, N, step):
        count = min(step, N - k)
        for dst, x in zip(out, _rows(gate, d, count, gen)):
            dst[32 * k:32 * (k + count)] = x.to(torch.int16).t().contiguous().view(torch.uint8).reshape(-1)
    return out


# -------------------------------------------------------------------- run --

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    gate, n, d = case["gate"], case["n"], case["d"]
    ctx = _context()
    cols = _columns(gate, n, d, seed)
    state = {"kind": kind, "args": (gate, n, d), "cols": cols, "domain": case.get("domain", 0)}
    state["roots"] = ctx.roots(gate, n, d, cols) if case.get("roots") else None
    if kind == "ntt":
        state["q"] = torch.empty(zc.domain_size(n, d, state["domain"]) * 32, dtype=torch.uint8, device="cuda")
    elif kind == "host_step":
        state["cols"] = [x.cpu().pin_memory().numpy() for x in cols]
        M = zc.domain_size(n, d, state["domain"])
        state["q"] = torch.empty(M * 32, dtype=torch.uint8).pin_memory().numpy()
    return state


def _prepare_batch(case, seed):
    # a graph keeps the scratch of its context's lanes: one context per prepared batch
    ctx = zc.Context(0, max_n=24, max_d=32)
    shapes = _batch_shapes(case)
    forms = [f for _, f in shapes]
    params = [(s.gate, s.n, s.d, 0) for s, _ in shapes]
    cols = [_columns(s.gate, s.n, s.d, seed * 64 + i) for i, (s, _) in enumerate(shapes)]
    sizes = [zc.proof_size(s.gate, s.n, s.d, f) for s, f in shapes]
    qsizes = [32 * zc.domain_size(s.n, s.d) if f == zc.ZC_FORM_NTT else 0 for s, f in shapes]
    proofs = torch.zeros(sum(-(-x // 256) * 256 for x in sizes), dtype=torch.uint8, device="cuda")
    q = torch.zeros(sum(qsizes) + 256, dtype=torch.uint8, device="cuda")
    pv, qv, po, qo = [], [], 0, 0
    for x, y in zip(sizes, qsizes):
        pv.append(proofs[po:po + x])
        qv.append(q[qo:qo + y] if y else None)
        po += -(-x // 256) * 256
        qo += y
    torch.cuda.synchronize()
    graph = ctx.batch_graph(forms, params, cols, pv, qv)
    return {"kind": "batch", "ctx": ctx, "graph": graph, "cols": cols, "proofs": proofs, "q": q, "views": (pv, qv)}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["graph"].launch()
        return [state["proofs"], state["q"]]
    ctx = _context()
    gate, n, d = state["args"]
    cols = state["cols"]
    if kind in ("sumcheck", "sumcheck_eq"):
        return ctx.prove_sumcheck(gate, n, d, cols, roots=state["roots"], eq_factored=kind == "sumcheck_eq")
    if kind == "ntt":
        return list(ctx.prove_ntt(gate, n, d, cols, roots=state["roots"], q_out=state["q"],
                                  log_blowup=state["domain"]))
    if kind == "host_step":
        proof = ctx.prove_sumcheck(gate, n, d, cols, roots=state["roots"])
        return [proof, *ctx.prove_ntt(gate, n, d, cols, roots=state["roots"], q_out=state["q"],
                                      log_blowup=state["domain"])]
    com = ctx.pcs_commit(n, cols, PCS_QUERIES)
    roots = [com.root] * len(cols)
    proof = ctx.prove_sumcheck(gate, n, d, cols, roots=roots)
    alpha, values, _ = zc.sumcheck_point(gate, n, d, zc.ZC_FORM_SUMCHECK, roots, proof)
    opening = np.frombuffer(com.open(alpha, values), dtype=np.uint8)
    root = np.frombuffer(com.root, dtype=np.uint8)
    com.close()
    return [root, proof, opening]


def exact(case, seed):
    """Every output is a byte string (field elements and digests): none is rounded, so none has a 64-bit value."""
    return None
