"""The register-tiled fp32 kernels at the edges of their tiles, for every pair of head dimensions: sequences that end at,
before and after the 4-row, 16-row and 32-row blocks of a chunk, one chunk and several (the carries' double buffer), closed
and on a workspace fresh from the forward.

Tolerance: every output is a chain of at most six products with contractions of up to 128 terms, each summed in fp32; rounding
adds up like sqrt(6 * 128) * 2^-24 = 1.7e-6 of the summands, and the decay gradient is a difference of such sums.  3e-6 for
whole tensors, three times that for one 64-token block."""
import numpy as np
import pytest
import torch

import oracle

from paper_2608_12700_b200 import runner, synth
from helpers import block_errors, check_against_oracle, oracle_grads, rel

pytestmark = pytest.mark.gpu


def heads_beyond(lengths):
    """Fewest heads with which two CTAs per chunk-head do not fit the SMs any more (chunk-heads are counted by the host's bound on the chunks)."""
    chunks = -(-sum(lengths) // 64) + len(lengths)
    return torch.cuda.get_device_properties(0).multi_processor_count // (2 * chunks) + 1


@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (128, 64), (64, 128)])
@pytest.mark.parametrize("lengths", [[1, 3, 5, 15, 16, 17], [31, 32, 33, 63, 64, 65], [127, 0, 193, 256, 321]])
@pytest.mark.parametrize("delta_rule", [1, 0])
@pytest.mark.parametrize("heads", [3, None], ids=["several_ctas", "one_cta"])
def test_tile_edges(dk, dv, lengths, delta_rule, heads):
    """With three heads the preparation takes two CTAs per chunk-head (and at d_k = 64 the gradient stage a cluster of two), with `heads_beyond`
    both take one."""
    wl = synth.make_workload("tiles", dtype="f32", lengths=lengths, H=heads or heads_beyond(lengths), d_k=dk, d_v=dv, seed=310, states=True, scale=0.7,
                             delta_rule=delta_rule)
    ref = oracle_grads(wl)
    buf = runner.to_device(wl, want_o=True)
    runner.run_bwd(buf)
    got = runner.fetch(buf)
    check_against_oracle(wl, got, tol=3e-6, ref=ref, block_tol=9e-6)
    runner.run_fwd(buf)
    f = runner.fetch(buf)
    assert rel(f["o"], ref["o"]) < 3e-6 and rel(f["hT"], ref["hT"]) < 3e-6
    runner.run_bwd(buf, fresh=1)
    fresh = runner.fetch(buf)
    for n in ("dq", "dk", "dv", "dg", "dh0") + (("dbeta",) if delta_rule else ()):
        assert np.array_equal(fresh[n], got[n]), n


@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (128, 64), (64, 128)])
@pytest.mark.parametrize("lengths,decay", [([1, 15, 16, 17, 31], 0.1), ([32, 33, 47, 48, 49, 63, 64, 65], 0.1), ([127, 0, 193], 0.1),
                                           ([100, 64, 17], 4.0)])
def test_channelwise_tile_edges(dk, dv, lengths, decay):
    """Per-channel gates: lengths around the 16-token blocks in which the decay is split, and a decay (about -3.2 per token)
    whose factor underflows inside a chunk.  There the decay gradient is what is left of sums e^3.2 = 25 times its size:
    25 times the tolerance, for it alone."""
    wl = synth.make_channelwise("cw_tiles", member="gdn", dtype="f32", lengths=lengths, H=2, d_k=dk, d_v=dv, seed=311, states=True,
                                scale=0.7, g_scale=decay)
    ref = oracle.vec_bwd_workload(wl)
    buf = runner.to_device_channelwise(wl, want_o=True)
    runner.run_bwd_channelwise(buf)
    got = runner.fetch(buf)
    for n in ("dq", "dk", "dv", "dg", "db", "dw", "dh0"):
        tol = 3e-6 * (25 if decay > 1 and n == "dg" else 1)
        assert rel(got[n], ref[n]) < tol, (n, rel(got[n], ref[n]))
        e, _ = block_errors(wl, n, got[n], ref[n])
        assert e.max() < 3 * tol, (n, e.max())
    runner.run_fwd_channelwise(buf)
    f = runner.fetch(buf)
    assert rel(f["o"], ref["o"]) < 3e-6 and rel(f["hT"], ref["hT"]) < 3e-6
    runner.run_bwd_channelwise(buf, fresh=1)
    fresh = runner.fetch(buf)
    for n in ("dq", "dk", "dv", "dg", "db", "dw", "dh0"):
        assert np.array_equal(fresh[n], got[n]), n


@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 128), (128, 64), (64, 128)])
@pytest.mark.parametrize("heads", [1, 2, 4, 9, 12, None])
def test_columns_per_cta_of_the_carries(dk, dv, heads):
    """The carries take 4, 8 or 16 state columns per CTA, by the number of chains, and the scalar-gate preparation and gradient stage
    one or several CTAs per chunk-head (preparation two while they fit the SMs, gradient stage d_k / 32; 4, 9 and 12 heads are 24, 54 and 72 of them,
    `heads_beyond` 78 on 148 SMs): each of them, in one direction and in both, with scalar and with per-channel gates (the same code with another
    decay)."""
    lengths = [130, 65]
    heads = heads or heads_beyond(lengths)
    wl = synth.make_workload("columns", dtype="f32", lengths=lengths, H=heads, d_k=dk, d_v=dv, seed=312, states=True)
    ref = oracle_grads(wl)
    buf = runner.to_device(wl, want_o=True)
    runner.run_bwd(buf)
    got = runner.fetch(buf)
    check_against_oracle(wl, got, tol=3e-6, ref=ref, block_tol=9e-6)
    runner.run_fwd(buf)
    runner.run_bwd(buf, fresh=1)
    f = runner.fetch(buf)
    assert rel(f["o"], ref["o"]) < 3e-6 and rel(f["hT"], ref["hT"]) < 3e-6
    check_against_oracle(wl, f, tol=3e-6, ref=ref, block_tol=9e-6)
    for n in ("dq", "dk", "dv", "dg", "dbeta", "dh0"):   # the backward on the forward's workspace repeats the closed one's arithmetic
        assert np.array_equal(f[n], got[n]), n
    wl = synth.make_channelwise("columns", member="gdn", dtype="f32", lengths=lengths, H=heads, d_k=dk, d_v=dv, seed=313, states=True)
    ref = oracle.vec_bwd_workload(wl)
    buf = runner.to_device_channelwise(wl, want_o=True)
    runner.run_bwd_channelwise(buf)
    got = runner.fetch(buf)
    for n in ("dq", "dk", "dv", "dg", "db", "dw", "dh0"):
        assert rel(got[n], ref[n]) < 3e-6, (n, rel(got[n], ref[n]))
