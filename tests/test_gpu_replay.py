"""GPU: plans whose calls mix direct launches, captures and graph replays (csrc/scw_replay.h)."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _plan(device, seed=5, **extra):
    import torch
    import paper_2404_07293_gb300 as scw
    W, g, a, *_ = wl.random_layer_set(seed, 7, 7, 2)
    plan = scw.Plan(U=7, V=7, L=2, lam=1.0, X=3.0, Y=3.3, z_bounds=np.array([0.0, 0.3, 0.8]), Fx=64, Fy=48,
                    z_planes=wl.cell_centred_planes(0.0, 0.8, 30), **extra)
    layers = tuple(torch.from_numpy(x).to(device) for x in (W, g, a))
    plan.set_layers(*layers)
    return plan, layers


@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
def test_two_outputs_in_any_order(precision, cuda_device):
    import torch
    plan, layers = _plan(cuda_device, precision=precision)
    ref = plan.synthesize().clone()
    outs = [torch.empty_like(ref) for _ in range(2)]
    for k in (0, 0, 1, 0, 1, 0, 1, 1, 1, 0, 0, 1):
        outs[k].zero_()
        plan.synthesize(outs[k])
        assert torch.equal(outs[k], ref), k
    other = _plan(cuda_device, seed=6, precision=precision)
    ref2 = other[0].synthesize()
    plan.set_layers(*other[1])  # another solution: no graph of the old one may run
    for k in (0, 1, 1, 0):
        outs[k].zero_()
        plan.synthesize(outs[k])
        assert torch.equal(outs[k], ref2), k
    plan.check()
    plan.close()
    other[0].close()


@pytest.mark.parametrize("calls_before", [0, 1, 2])
def test_another_thread_may_be_capturing(calls_before, cuda_device):
    """The call that captures (the second in a row) works while another thread records a graph, and leaves it whole."""
    import threading

    import torch
    plan, layers = _plan(cuda_device)
    ref = plan.synthesize().clone()
    out = torch.zeros_like(ref)
    theirs, ours = torch.cuda.Stream(), torch.cuda.Stream()
    ours.wait_stream(torch.cuda.current_stream())
    for _ in range(calls_before):
        plan.synthesize(out, stream=ours)
    x = torch.zeros(16, device=cuda_device)
    torch.cuda.synchronize()
    errors = []

    def call():
        try:
            plan.synthesize(out, stream=ours)
        except Exception as e:  # noqa: BLE001 - reported below, after the capture has ended
            errors.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(theirs):
        graph.capture_begin(capture_error_mode="global")
        x += 1
        t = threading.Thread(target=call)
        t.start()
        t.join()
        graph.capture_end()
    assert not errors, errors
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, torch.ones_like(x))
    plan.check()
    plan.close()
