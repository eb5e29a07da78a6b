"""Several N2 slices per launch (small NTT proofs): the oracle's bytes where the
slices share a launch, where a memory budget of exactly the reported scratch
leaves room for one slice at a time, and at the first size with one slice per
launch; openings with the shortest and with growing segments."""
import numpy as np
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gate,n,d,lb", [(1, 2, 3, 0), (1, 10, 3, 0), (1, 13, 3, 1), (2, 11, 8, 0), (2, 12, 6, 0x102),
                                         (witness.gate_sum(0), 16, 2, 0), (1, 16, 3, 0), (1, 17, 3, 0)])
def test_slices_share_a_launch_or_not(gate, n, d, lb):
    cols = witness.generate(gate, n, d, 9400 + n)
    want_p, want_q = oracle.prove_ntt(gate, n, d, cols, log_blowup=lb)
    dc = to_device(cols)
    free = zc.Context(0, max_n=18, max_d=8)
    try:
        need = free.scratch_bytes(gate, n, d, zc.ZC_FORM_NTT, False, lb)
        got = [free.prove_ntt(gate, n, d, dc, log_blowup=lb)]
    finally:
        free.close()
    tight = zc.Context(0, max_n=18, max_d=8, mem_budget_bytes=need)
    try:
        got += [tight.prove_ntt(gate, n, d, dc, log_blowup=lb) for _ in range(2)]
    finally:
        tight.close()
    for p, q in got:
        assert proof_bytes(p) == want_p
        assert np.asarray(q).tobytes() == want_q.tobytes()


def test_slices_as_the_scratch_has_room():
    """A context whose scratch, sized by another shape, holds two of the four slices."""
    ctx = zc.Context(0, max_n=14, max_d=4)
    try:
        for gate, d in ((2, 4), (1, 3)):
            cols = witness.generate(gate, 13, d, 9500 + d)
            p, q = ctx.prove_ntt(gate, 13, d, to_device(cols))
            want_p, want_q = oracle.prove_ntt(gate, 13, d, cols)
            assert proof_bytes(p) == want_p
            assert np.asarray(q).tobytes() == want_q.tobytes()
    finally:
        ctx.close()
