"""A batch graph keeps the scratch of its lanes: it proves the oracle's bytes
after the context's lanes took larger scratch for another batch, after a
serving run (which gives the lanes blocks of its pool), and again after that."""
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu


def _batch(shapes, seed):
    import torch
    xs = []
    for i, (form, gate, n, d) in enumerate(shapes):
        cols = witness.generate(gate, n, d, seed + i)
        want = oracle.prove_sumcheck(gate, n, d, cols) if form == 1 else oracle.prove_ntt(gate, n, d, cols)[0]
        xs.append(dict(form=form, p=(gate, n, d, 0), dcols=to_device(cols), want=want,
                       proof=torch.zeros(zc.proof_size(gate, n, d, form), dtype=torch.uint8, device="cuda")))
    return xs


def _args(xs):
    return [x["form"] for x in xs], [x["p"] for x in xs], [x["dcols"] for x in xs], [x["proof"] for x in xs], None


def _check(xs):
    import torch
    torch.cuda.synchronize()
    for x in xs:
        assert proof_bytes(x["proof"]) == x["want"]
        x["proof"].zero_()


def test_graph_keeps_its_scratch():
    small = _batch([(1, 1, 8, 3), (2, 1, 7, 3), (1, 2, 6, 4)], 9700)
    large = _batch([(1, 1, 16, 3), (2, 1, 15, 3), (1, 2, 14, 4), (2, 2, 12, 4)], 9710)
    ctx = zc.Context(0, max_n=18, max_d=8)
    try:
        g = ctx.batch_graph(*_args(small))
        h = ctx.batch_graph(*_args(large))  # the same lanes, more scratch
        for b, xs in ((g, small), (h, large), (g, small)):
            b.launch()
            _check(xs)
        reqs = [dict(arrival_s=0.0, gate=x["p"][0], n=x["p"][1], d=x["p"][2], form=x["form"], cols=x["dcols"],
                     proof=x["proof"]) for x in large]
        ctx.serve(reqs, slots=4, hbm_budget_bytes=256 << 20, timeout_s=60.0)
        _check(large)
        for b, xs in ((h, large), (g, small)):
            b.launch()
            _check(xs)
        ctx.prove_batch(*_args(large))  # the lanes again without scratch of their own
        _check(large)
        h.close()
        g.launch()
        _check(small)
        g.close()
    finally:
        ctx.close()
