"""The per-size NTT tables at their limit (ZC_NTT_TABLE_BYTES lowers it): a
batch graph's tables stay while the context proves other sizes, a prepared set
keeps the tables of all its sizes that fit, step-radix domains (which have no
other route) prove whatever else is held.  Every byte is the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu


def table_bytes(n, lb):
    return 64 * (2 * (1 << n) + 2 * (1 << n + lb) + 2 * (1 << lb))


def ctx_with(monkeypatch, limit, **kw):
    monkeypatch.setenv("ZC_NTT_TABLE_BYTES", str(limit))
    c = zc.Context(0, max_n=18, max_d=32, **kw)
    monkeypatch.delenv("ZC_NTT_TABLE_BYTES")
    return c


def instance(gate, n, d, lb, seed):
    import torch
    cols = witness.generate(gate, n, d, seed)
    want, q = oracle.prove_ntt(gate, n, d, cols, log_blowup=lb)
    proof = torch.zeros(zc.proof_size(gate, n, d, zc.ZC_FORM_NTT), dtype=torch.uint8, device="cuda")
    return dict(p=(gate, n, d, lb), dcols=to_device(cols), want=want, q=q.tobytes(), proof=proof)


def prove(ctx, x):
    """One proof alone; the number of kernels it launched."""
    gate, n, d, lb = x["p"]
    p, q = ctx.prove_ntt(gate, n, d, x["dcols"], log_blowup=lb)
    assert proof_bytes(p) == x["want"]
    assert np.asarray(q).tobytes() == x["q"]
    return int(ctx.stats()[9])


def batch(ctx, xs):
    return ctx.batch_graph([zc.ZC_FORM_NTT] * len(xs), [x["p"] for x in xs], [x["dcols"] for x in xs],
                           [x["proof"] for x in xs], None)


def check(xs):
    import torch
    torch.cuda.synchronize()
    for x in xs:
        assert proof_bytes(x["proof"]) == x["want"]
        x["proof"].zero_()


def test_graph_keeps_its_tables(monkeypatch):
    a, b = instance(1, 8, 3, 2, 9600), instance(1, 9, 3, 2, 9601)
    free = ctx_with(monkeypatch, 1 << 30)
    try:
        prove(free, b)
        with_tables = prove(free, b)
    finally:
        free.close()
    # room for either size, not for both
    ctx = ctx_with(monkeypatch, table_bytes(9, 2) + table_bytes(8, 2) - 1)
    try:
        g = batch(ctx, [a])
        for _ in range(2):
            g.launch()
            check([a])
            assert prove(ctx, b) > with_tables  # no tables: theirs are held by the graph
        g.close()
        prove(ctx, b)
        assert prove(ctx, b) == with_tables  # the graph is gone, and so may its tables
    finally:
        ctx.close()


# shapes in the order in which they are prepared, the step-radix one first, in
# the middle and last; each limit holds the largest alone
@pytest.mark.parametrize("shapes", [[(1, 9, 3, 0x101), (1, 8, 3, 2), (2, 9, 4, 2)],
                                    [(1, 8, 3, 2), (2, 8, 4, 0x102), (2, 9, 4, 2)],
                                    [(1, 9, 3, 2), (1, 8, 3, 2), (1, 7, 3, 0x101), (2, 7, 6, 0x102)]])
def test_prepared_sets_past_the_limit(monkeypatch, shapes):
    import torch
    xs = [instance(*s, 9610 + i) for i, s in enumerate(shapes)]
    ctx = ctx_with(monkeypatch, max(table_bytes(n, lb & 255) for _, n, _, lb in shapes))
    try:
        g = batch(ctx, xs)
        g.launch()
        check(xs)
        ctx.prove_batch([zc.ZC_FORM_NTT] * len(xs), [x["p"] for x in xs], [x["dcols"] for x in xs],
                        [x["proof"] for x in xs], None)
        check(xs)
        reqs = [dict(arrival_s=0.0, gate=x["p"][0], n=x["p"][1], d=x["p"][2], log_blowup=x["p"][3],
                     form=zc.ZC_FORM_NTT, cols=x["dcols"], proof=x["proof"]) for x in xs]
        res = ctx.serve(reqs, slots=2, hbm_budget_bytes=64 << 20, timeout_s=60.0)
        assert all(r["status"] == 0 for r in res)
        check(xs)
        g.close()
        torch.cuda.synchronize()
        for x in xs:
            prove(ctx, x)
    finally:
        ctx.close()


def test_step_tables_count(monkeypatch):
    """The step-radix part of a size makes room for itself as the size does."""
    a, b = instance(1, 7, 3, 2, 9630), instance(1, 8, 3, 0x101, 9631)
    ctx = ctx_with(monkeypatch, table_bytes(7, 2) + table_bytes(8, 1))
    try:
        first = prove(ctx, a)
        assert prove(ctx, a) < first  # its tables are there
        prove(ctx, b)
        assert prove(ctx, a) == first  # they went for b's
        prove(ctx, b)
    finally:
        ctx.close()


def test_default_limit_holds_three_large_sizes():
    """25 GiB of tables in one prepared set (12.5 GiB with 32-byte entries), none without them."""
    import torch
    shapes = [(witness.gate_sum(0), 24, 2, 1), (witness.gate_sum(0), 24, 3, 2), (witness.gate_sum(0), 23, 2, 3)]
    assert sum(table_bytes(n, lb) for _, n, _, lb in shapes) > 24 << 30
    cols = [torch.empty(32 << 24, dtype=torch.uint8, device="cuda") for _ in range(3)]  # captured, never launched
    proofs = [torch.empty(zc.proof_size(g, n, d, zc.ZC_FORM_NTT), dtype=torch.uint8, device="cuda")
              for g, n, d, _ in shapes]

    def kernels(idx):
        ctx = zc.Context(0, max_n=24, max_d=4)
        try:
            g = ctx.batch_graph([zc.ZC_FORM_NTT] * len(idx), [shapes[i] for i in idx],
                                [cols[:shapes[i][2]] for i in idx], [proofs[i] for i in idx], None)
            k = g.kernels
            g.close()
            return k
        finally:
            ctx.close()

    assert kernels([0, 1, 2]) == sum(kernels([i]) for i in range(3))
