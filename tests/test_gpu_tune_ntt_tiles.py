"""The NTT tile and residency keys act at every size: the kernels that a proof
launches are those the keys ask for, and the bytes are the oracle's."""
import re

import numpy as np
import pytest

import oracle
from gpu_util import proof_bytes, to_device
from paper_2606_16146_gb300 import witness, zc

pytestmark = pytest.mark.gpu

TILE, MINB = zc.ZC_TUNE_NTT_TILE_LOG, zc.ZC_TUNE_NTT_MINB


def pass_kernels(ctx, gate, n, d, dcols, tmp):
    """The pass kernels of one proof, from a stream capture of it (never launched)."""
    import torch
    proof = torch.zeros(zc.proof_size(gate, n, d, zc.ZC_FORM_NTT), dtype=torch.uint8, device="cuda")
    g = torch.cuda.CUDAGraph(keep_graph=True)
    s = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        ctx.prove_ntt(gate, n, d, dcols, stream=s, proof_out=proof, want_q=False)
    g.debug_dump(str(tmp / "g.dot"))
    names = set(re.findall(r"k_ntt_pass\w*", (tmp / "g.dot").read_text()))
    # mangled: k_ntt_passILi<threads>ELi<resident>ELb<fast>E..., k_ntt_pass_small...
    return {"small" if x.startswith("k_ntt_pass_small") else tuple(map(int, re.findall(r"Li(\d+)", x)))
            for x in names}


# n = 9: one sub-DFT of 2^9 per column and slice; 13: two digits; 17: launches past 2^19 elements
@pytest.mark.parametrize("gate,n,d", [(1, 9, 3), (2, 13, 5), (1, 17, 3)])
def test_keys_choose_the_pass_kernel(gate, n, d, tmp_path):
    cols = witness.generate(gate, n, d, 9800 + n)
    want_p, want_q = oracle.prove_ntt(gate, n, d, cols)
    dc = to_device(cols)
    ctx = zc.Context(0, max_n=18, max_d=8)
    try:
        for tile, minb, want in [(0, 0, None), (10, 0, {(128, 4)}), (11, 0, {(256, 2)}), (11, 1, {(256, 1)}),
                                 (12, 0, {(512, 1)}), (0, 2, {(128, 4)})]:
            ctx.tune_set(zc.ZC_FORM_NTT, n, TILE, tile)
            ctx.tune_set(zc.ZC_FORM_NTT, n, MINB, minb)
            p, q = ctx.prove_ntt(gate, n, d, dc)
            assert proof_bytes(p) == want_p, (tile, minb)
            assert np.asarray(q).tobytes() == want_q.tobytes(), (tile, minb)
            got = pass_kernels(ctx, gate, n, d, dc, tmp_path)
            if want is None:
                assert "small" in got and (n < 17 or (128, 4) in got), got
            else:
                assert got == want, (tile, minb, got)
    finally:
        ctx.close()
