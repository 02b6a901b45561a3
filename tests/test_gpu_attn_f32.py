"""The CUDA-core attention (fp32; bf16 with d_head 32) inside whole rounds against the oracle, at context lengths around
the edges of its 32-row query tiles and 128-key tiles, for both head widths."""
import pytest

import synth
from tests import parity, roundcheck

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol,heads", [("fp32", 1e-4, (2, 4)), ("bf16", 2e-2, (4, 4))])
@pytest.mark.parametrize("plen,gamma", [([121, 24, 2], 7), ([300, 129, 250], 33)])
def test_rounds_at_tile_edges(dtype, tol, heads, plen, gamma):
    import paper_2408_05636_b200 as sdd
    wl = synth.scaled_workload(
        synth.WORKLOADS["tiny_fp32"], dtype=dtype, batch=3, gamma=gamma, T=2,
        target=synth.ModelShape(512, 2, 128, heads[0], 512, True), drafter=synth.ModelShape(512, 2, 128, heads[1], 512, False))
    mp, mq, dp, dq = roundcheck.build_pair(wl, bias_std=0.05, perturb_ln=True)
    prompts = synth.prompt_ids(512, 3, max(plen), wl.prompt_seed)
    s = sdd.Session(dp, dq, prompts, plen, gamma, 2, 40, 1.0, 1.0, wl.philox_seed)
    log, _ = roundcheck.check_rounds(s, mp, mq, wl, 2, 1.0, 1.0, tol)
    parity.assert_few(log)
    s.close()
