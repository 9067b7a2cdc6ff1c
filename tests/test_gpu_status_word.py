"""The status word of a workspace: after a device-side error a call leaves its outputs unwritten, and malformed cu_seqlens are
refused before any kernel reads them, in a backward on the forward's workspace too; such a backward computes nothing after an
error of the forward (the word is written by the host here, in place of a wait that ran out).  Every kernel family."""
import numpy as np
import pytest
import torch

from paper_2608_12700_b200 import binding, runner, synth

pytestmark = pytest.mark.gpu

BAD_SEQLENS, TIMEOUT = 5, 8

FAMILIES = {   # (per-channel gates, forced family, descriptor)
    "operator_form": (False, 2, dict(dtype="bf16", d_k=128, d_v=128)),
    "low_rank_form": (False, 3, dict(dtype="bf16", d_k=128, d_v=128)),
    "narrow_values": (False, 0, dict(dtype="bf16", d_k=128, d_v=64)),
    "scalar_gate_d64": (False, 0, dict(dtype="bf16", d_k=64, d_v=64, delta_rule=0)),
    "ffma": (False, 0, dict(dtype="f32", d_k=64, d_v=128)),
    "channelwise": (True, 0, dict(dtype="bf16", d_k=128, d_v=128)),
    "channelwise_padded": (True, 0, dict(dtype="bf16", d_k=64, d_v=64)),
    "channelwise_ffma": (True, 0, dict(dtype="f32", d_k=64, d_v=64)),
}


@pytest.fixture(params=sorted(FAMILIES))
def family(request):
    channelwise, forced, kw = FAMILIES[request.param]
    binding.gdn_debug_force_family(forced)
    yield channelwise, kw
    binding.gdn_debug_force_family(0)


@pytest.mark.parametrize("bad", [[0, 180, 164, 194], [0, 100, 164, 190], [3, 100, 164, 194]], ids=["decreasing", "short", "offset"])
def test_malformed_cu_seqlens_leave_the_outputs_unwritten(family, bad):
    channelwise, fam = family
    wl = (synth.make_channelwise if channelwise else synth.make_workload)("status", lengths=[100, 64, 30], H=2, states=True, seed=190, **fam)
    buf = (runner.to_device_channelwise if channelwise else runner.to_device)(wl, want_o=True)
    buf.inputs["cu_seqlens"] = torch.tensor(bad, dtype=torch.int32, device="cuda")
    for run, outputs in ((runner.run_bwd_channelwise if channelwise else runner.run_bwd, ("dq", "dk", "dv", "dg", "dbeta", "db", "dw", "dh0")),
                         (runner.run_fwd_channelwise if channelwise else runner.run_fwd, ("o", "hT"))):
        outs = [buf.outputs[n] for n in outputs if buf.outputs.get(n) is not None]
        for v in outs:
            v.fill_(7.0)
        run(buf)
        assert binding.gdn_last_device_status(buf.workspace) == BAD_SEQLENS
        assert all(torch.all(v == 7.0) for v in outs)


def forward(family, **kw):
    """Buffers after a forward, outputs of the backward filled with 7, and the backward on that workspace."""
    channelwise, fam = family
    make = synth.make_channelwise if channelwise else synth.make_workload
    wl = make("status", H=2, states=True, seed=190, **fam, **kw)
    buf = (runner.to_device_channelwise if channelwise else runner.to_device)(wl, want_o=True)
    (runner.run_fwd_channelwise if channelwise else runner.run_fwd)(buf)
    for n, v in buf.outputs.items():
        if v is not None and n not in ("o", "hT"):
            v.fill_(7.0)
    run = runner.run_bwd_channelwise if channelwise else runner.run_bwd
    return wl, buf, lambda: run(buf, fresh=1)


def assert_unwritten(buf):
    for n, v in buf.outputs.items():
        if v is not None and n not in ("o", "hT"):
            assert torch.all(v == 7.0), n


def test_malformed_cu_seqlens_are_refused_on_a_forwards_workspace(family):
    wl, buf, bwd = forward(family, lengths=[100, 64, 30])
    good = buf.inputs["cu_seqlens"]
    for bad in ([0, 180, 164, 194], [0, 100, 164, 190], [3, 100, 164, 194]):   # decreasing; short of T; not from 0
        buf.inputs["cu_seqlens"] = torch.tensor(bad, dtype=torch.int32, device="cuda")
        bwd()
        assert binding.gdn_last_device_status(buf.workspace) == BAD_SEQLENS
        assert_unwritten(buf)
    # the forward's data is whole: with its own cu_seqlens the backward runs (twice: after a refusal, and after a good call), and as if
    # nothing had happened
    buf.inputs["cu_seqlens"] = good
    bwd()
    bwd()
    got = runner.fetch(buf)
    channelwise, _ = family
    whole = (runner.backward_channelwise if channelwise else runner.backward)(wl)
    for n in whole:
        assert np.array_equal(whole[n], got[n]), n


@pytest.mark.parametrize("seqs", [dict(lengths=[100, 64, 30]), dict(B=2, T=100)], ids=["packed", "equal"])
def test_an_error_of_the_forward_stands_in_the_backward_on_its_workspace(family, seqs):
    wl, buf, bwd = forward(family, **seqs)
    buf.workspace[:4].view(torch.int32).fill_(TIMEOUT)
    bwd()
    assert binding.gdn_last_device_status(buf.workspace) == TIMEOUT
    assert_unwritten(buf)


def test_malformed_cu_seqlens_in_the_forward_leave_nothing_for_the_backward(family):
    wl, buf, bwd = forward(family, lengths=[100, 64, 30])
    good = buf.inputs["cu_seqlens"]
    buf.inputs["cu_seqlens"] = torch.tensor([0, 100, 164, 190], dtype=torch.int32, device="cuda")
    (runner.run_fwd_channelwise if family[0] else runner.run_fwd)(buf)
    assert binding.gdn_last_device_status(buf.workspace) == BAD_SEQLENS
    buf.inputs["cu_seqlens"] = good
    bwd()
    assert binding.gdn_last_device_status(buf.workspace) == BAD_SEQLENS
    assert_unwritten(buf)
