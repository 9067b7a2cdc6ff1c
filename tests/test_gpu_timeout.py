"""Failure detection on the device: every wait in the kernels is bounded, and a wait that runs out is reported
through the workspace's status word instead of hanging or trapping.  The test makes one wait run out on the host's
terms (a debugging hook shortens the limit to a millisecond for one call and has one of the kernels leave out one of
its loads); nothing faults, and the same buffers give correct gradients on the next call."""
import numpy as np
import pytest
import torch

from paper_2608_12700_b200 import binding, runner, synth
from helpers import check_against_oracle

pytestmark = pytest.mark.gpu

GDN_ERR_DEVICE_TIMEOUT = 8


@pytest.mark.parametrize("lengths,H", [([64], 1), ([200, 64, 75], 2)])
def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_correct(lengths, H):
    wl = synth.make_workload("timeout", dtype="bf16", lengths=lengths, H=H, d_k=128, d_v=128, states=True, seed=90)
    buf = runner.to_device(wl)
    assert binding.gdn_kernel_path(buf.desc) == "tcgen05_bf16"
    for v in buf.outputs.values():
        if v is not None:
            v.fill_(7.0)
    binding.gdn_debug_inject_timeout(True)
    runner.run_bwd(buf)                                   # returns GDN_OK: the condition is only visible on the device
    assert binding.gdn_last_device_status(buf.workspace) == GDN_ERR_DEVICE_TIMEOUT
    assert "wait" in binding.status_string(GDN_ERR_DEVICE_TIMEOUT)
    # the stages after the one that gave up wrote nothing
    for n in ("dq", "dk", "dv", "dg", "dbeta"):
        assert torch.all(buf.outputs[n] == 7.0), n
    # the context is intact and the request was for one call: same buffers, same workspace, correct gradients
    runner.run_bwd(buf)
    check_against_oracle(wl, runner.fetch(buf))
    assert binding.gdn_last_device_status(buf.workspace) == binding.GDN_OK


@pytest.mark.parametrize("form", [2, 3], ids=["operator", "low_rank"])
@pytest.mark.parametrize("where", [1, 2, 3], ids=["preparation", "carries", "gradients"])
@pytest.mark.parametrize("shape", [dict(lengths=[200, 64, 75], H=2), dict(B=3, T=700, H=10)], ids=["small", "several_trips"])
def test_every_kernel_leaves_through_its_teardown(shape, where, form):
    """One wait at a time, in the preparation, the carries (one and two CTAs per chain) and the gradient stage, in both forms of the
    carries; the larger shape has 330 chunk-heads (every CTA of the persistent kernels has further trips) and 30 chains."""
    try:
        binding.gdn_debug_force_family(form)
        wl = synth.make_workload("timeout_where", dtype="bf16", d_k=128, d_v=128, states=True, seed=92, **shape)
        buf = runner.to_device(wl)
        for v in buf.outputs.values():
            if v is not None:
                v.fill_(7.0)
        binding.gdn_debug_inject_timeout(where)
        runner.run_bwd(buf)
        assert binding.gdn_last_device_status(buf.workspace) == GDN_ERR_DEVICE_TIMEOUT
        if where < 3:   # the gradient stage saw the status and wrote nothing
            for n in ("dq", "dk", "dv", "dg", "dbeta") + (("dh0",) if where == 2 else ()):
                assert torch.all(buf.outputs[n] == 7.0), n
        runner.run_bwd(buf)
        check_against_oracle(wl, runner.fetch(buf))
    finally:
        binding.gdn_debug_force_family(0)


@pytest.mark.parametrize("form", [2, 3], ids=["operator", "low_rank"])
@pytest.mark.parametrize("where", [4, 5, 6], ids=["preparation", "carries", "gradients"])
@pytest.mark.parametrize("shape", [dict(lengths=[200, 64, 75], H=2, d_v=128), dict(B=3, T=700, H=10, d_v=128), dict(lengths=[300, 64], H=2, d_v=64)],
                         ids=["small", "several_trips", "narrow_values"])
def test_warps_that_disagree_about_a_wait_leave_together(shape, form, where):
    """Each warp judges by its own clock whether a wait has run out.  Half of them say so here although nothing is missing: the call ends (the
    warps that went on are not left behind at a barrier), reports it, and the next one is correct."""
    try:
        binding.gdn_debug_force_family(form)
        wl = synth.make_workload("timeout_split", dtype="bf16", d_k=128, states=True, seed=93, **shape)
        buf = runner.to_device(wl)
        for v in buf.outputs.values():
            if v is not None:
                v.fill_(7.0)
        binding.gdn_debug_inject_timeout(where)
        runner.run_bwd(buf)
        assert binding.gdn_last_device_status(buf.workspace) == GDN_ERR_DEVICE_TIMEOUT
        for n in ("dq", "dk", "dv", "dg", "dbeta", "dh0") if where < 6 else ():   # (the kernels behind the one in question, and its final states)
            assert torch.all(buf.outputs[n] == 7.0), n
        runner.run_bwd(buf)
        check_against_oracle(wl, runner.fetch(buf))
        assert binding.gdn_last_device_status(buf.workspace) == binding.GDN_OK
    finally:
        binding.gdn_debug_force_family(0)


def test_a_cancelled_request_changes_nothing():
    wl = synth.make_workload("timeout_cancel", dtype="bf16", lengths=[100], H=1, d_k=128, d_v=128, states=True, seed=91)
    binding.gdn_debug_inject_timeout(True)
    binding.gdn_debug_inject_timeout(False)
    check_against_oracle(wl, runner.backward(wl))
