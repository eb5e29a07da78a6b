"""The NTT form without per-size tables (ZC_NTT_TABLE_BYTES=0; sizes whose
tables pass the limit take this route): factors from the two-level power
tables, through the general pass form, prove the oracle's bytes."""
import numpy as np
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    mp = pytest.MonkeyPatch()
    mp.setenv("ZC_NTT_TABLE_BYTES", "0")
    c = zc.Context(0, max_n=18, max_d=64)
    mp.undo()
    yield c
    c.close()


def check(ctx, gate, n, d, lb, cols, arg):
    want_p, want_q = oracle.prove_ntt(gate, n, d, cols, log_blowup=lb)
    p, q = ctx.prove_ntt(gate, n, d, arg, log_blowup=lb)
    assert proof_bytes(p) == want_p
    assert np.asarray(q).tobytes() == want_q.tobytes()


# part-filled tiles, one sub-DFT per column (2^11 and 2^12 too), two digits of
# equal and of unequal length, 2 to 64 slices, columns up to 34
@pytest.mark.parametrize("gate,n,d,lb", [(1, 1, 3, 0), (1, 2, 3, 0), (1, 3, 3, 1), (1, 5, 3, 0), (2, 6, 8, 0),
                                         (1, 9, 3, 0), (2, 11, 4, 0), (1, 12, 3, 0), (1, 13, 3, 1), (2, 7, 33, 0),
                                         (2, 12, 16, 0), (witness.gate_sum(0), 10, 2, 0),
                                         (witness.gate_sum(3), 15, 2, 1), (1, 17, 3, 0), (1, 18, 3, 0)])
def test_bytes(ctx, gate, n, d, lb):
    cols = witness.generate(gate, n, d, 9900 + n)
    check(ctx, gate, n, d, lb, cols, to_device(cols))


@pytest.mark.parametrize("n,two_log", [(9, 4), (12, 13), (14, 0)])
@pytest.mark.parametrize("tile", [10, 11, 12])
def test_tiles_and_digits(ctx, n, two_log, tile):
    cols = witness.generate(1, n, 3, 9930 + n)
    keys = {zc.ZC_TUNE_NTT_TILE_LOG: tile, zc.ZC_TUNE_NTT_TWO_LOG: two_log}
    for k, v in keys.items():
        ctx.tune_set(zc.ZC_FORM_NTT, n, k, v)
    try:
        check(ctx, 1, n, 3, 0, cols, to_device(cols))
    finally:
        for k in keys:
            ctx.tune_set(zc.ZC_FORM_NTT, n, k, 0)


@pytest.mark.parametrize("n", [10, 14])
def test_host_columns(ctx, n):
    cols = witness.generate(1, n, 3, 9950 + n)
    check(ctx, 1, n, 3, 0, cols, cols)


def test_witness_that_does_not_vanish(ctx):
    cols = witness.generate(1, 13, 3, 9960, tamper=True)
    check(ctx, 1, 13, 3, 0, cols, to_device(cols))


def test_step_radix_is_refused(ctx):
    cols = to_device(witness.generate(1, 9, 3, 9970))
    with pytest.raises(zc.ZCError):
        ctx.prove_ntt(1, 9, 3, cols, log_blowup=0x101)
