"""The product and sum gates' persistent round kernel (their rounds with at
most 2^16 pairs before the tail, in one cooperative launch): its proofs equal
the oracle's, as do those of the per-round kernels, at sizes with one and many
such rounds, both forms of a round (every point evaluated, one derived) and
degrees whose points fill the CTA or leave threads over; a hand-off whose
bounded wait runs out is reported, and the context proves correctly after."""
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gate,n,d", [(2, 8, 2), (2, 9, 8), (2, 17, 3), (2, 13, 16), (2, 10, 64),
                                      (witness.gate_sum(0), 12, 2), (witness.gate_sum(3), 18, 2),
                                      (witness.gate_sum(1), 11, 4)])
def test_product_persistent_and_per_round_kernels_agree(monkeypatch, gate, n, d):
    cols = witness.generate(gate, n, d, 9800 + 10 * n + d)
    want = oracle.prove_sumcheck(gate, n, d, cols)
    dc = to_device(cols)
    for flag in ("1", "0"):
        monkeypatch.setenv("ZC_SC_PERSISTENT", flag)
        ctx = zc.Context(0, max_n=18, max_d=64)
        try:
            assert proof_bytes(ctx.prove_sumcheck(gate, n, d, dc)) == want, flag
        finally:
            ctx.close()


def test_product_handoff_timeout_is_reported_and_recovered(monkeypatch):
    gate, n, d = 2, 14, 4
    cols = witness.generate(gate, n, d, 9900)
    dc = to_device(cols)
    ctx = zc.Context(0, max_n=16, max_d=8)
    try:
        monkeypatch.setenv("ZC_SPIN_LIMIT", "1")
        with pytest.raises(zc.ZCError) as e:
            ctx.prove_sumcheck(gate, n, d, dc)
        assert e.value.status == 4                      # ZC_ERR_TIMEOUT
        monkeypatch.delenv("ZC_SPIN_LIMIT")
        assert proof_bytes(ctx.prove_sumcheck(gate, n, d, dc)) == oracle.prove_sumcheck(gate, n, d, cols)
    finally:
        ctx.close()
