"""GPU: index checks (SCW_FLAG_DEBUG_BOUNDS) cover the kernel that writes the field in normal plans. A checked plan
runs the one-kernel recomposition where the plan without the flag does, and the x-pass and the y-pass over the same
field; it gives the same bits and reports an access past a lowered extent of any buffer that they read or write."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

BOUNDS = 8  # SCW_ERR_BOUNDS
# U, V, Fx, Fy, planes: fold lengths of 8 to 48 positions, one and two columns per thread, narrow and widest rows,
# planes enough for the one-kernel form, with and without a split last round
SHAPES = [(1, 1, 8, 8, 24), (7, 5, 16, 24, 30), (9, 9, 136, 64, 40), (21, 17, 248, 16, 30), (23, 23, 256, 48, 22),
          (13, 33, 128, 32, 30), (4, 48, 104, 40, 28), (9, 7, 40, 2048, 22), (7, 7, 64, 64, 300)]


def _plan(U, V, Fx, Fy, planes, device, **extra):
    import torch
    import paper_2404_07293_gb300 as scw
    W, g, a, *_ = wl.random_layer_set(U * 100 + V, U, V, 2)
    plan = scw.Plan(U=U, V=V, L=2, lam=1.0, X=3.1, Y=2.7, z_bounds=np.array([0.0, 0.4, 0.7]), Fx=Fx, Fy=Fy,
                    z_planes=wl.cell_centred_planes(0.0, 0.7, planes), x0=0.13, y0=-0.4, k_split=2, **extra)
    plan.set_layers(*(torch.from_numpy(np.ascontiguousarray(x)).to(device) for x in (W, g, a)))
    return plan


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
def test_checked_plan_runs_every_form(shape, precision, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    plan = _plan(*shape, cuda_device, precision=precision)
    ref = plan.synthesize()
    plan.check()
    n = plan.info()["kernels_per_synthesis"]
    plan.close()
    plan = _plan(*shape, cuda_device, precision=precision, debug_bounds=True)
    out = plan.synthesize()
    plan.check()
    assert torch.equal(out, ref)
    assert n == 3  # phases, contraction, recomposition
    assert plan.info()["kernels_per_synthesis"] == n + 2  # and the x-pass and the y-pass
    for name in ("s_part", "t", "twx", "twy", "field"):
        plan.debug_set_extent(name, 1)
        plan.synthesize(out)
        with pytest.raises(scw.ScwError) as e:
            plan.check()
        assert e.value.status == BOUNDS, (name, str(e.value))
        plan.debug_set_extent(name, 0)
    plan.synthesize(out)
    plan.check()
    assert torch.equal(out, ref)
    plan.close()


def test_checked_batch_runs_every_form(cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    items, dev = [], []
    for k, (U, V, Fx, Fy, n) in enumerate([(9, 9, 64, 32, 16), (5, 25, 40, 64, 8), (21, 17, 256, 24, 12)]):
        W, g, a, *_ = wl.random_layer_set(70 + k, U, V, 2)
        items.append(dict(U=U, V=V, L=2, lam=1.0, X=3.0, Y=3.3, z_bounds=np.array([0.0, 0.3, 0.8]), Fx=Fx, Fy=Fy,
                          z_planes=wl.cell_centred_planes(0.0, 0.8, n), k_split=1))
        dev.append(tuple(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    outs, kernels = [], []
    for debug in (False, True):
        bp = scw.BatchedPlan([dict(kw, debug_bounds=debug) for kw in items])
        for i, d in enumerate(dev):
            bp.set_layers(i, *d)
        outs.append(bp.synthesize())
        bp.check()
        kernels.append(bp.info()["kernels_per_synthesis"])
        bp.close()
    assert kernels[1] == kernels[0] + 3  # the x-pass and, for 16 to 32 fold positions, both y-pass kernels
    for a, b in zip(*outs):
        assert torch.equal(a, b)


def test_rows_are_allocated_where_a_kernel_writes_them(cuda_device):
    """The x-pass rows [planes][3][V][Fx] belong to plans that run the x-pass."""
    shape = (9, 9, 136, 64, 40)
    rows = 40 * 3 * 9 * 136 * 8
    plan = _plan(*shape, cuda_device)
    fused = plan.info()["workspace_bytes"]
    ref = plan.synthesize()
    plan.set_pipeline(2)
    assert plan.info()["workspace_bytes"] == fused + rows
    out = plan.synthesize()
    plan.set_pipeline(1)
    plan.set_pipeline(2)
    assert plan.info()["workspace_bytes"] == fused + rows
    plan.check()
    assert (out == ref).all()
    plan.close()
    for extra in (dict(debug_bounds=True), dict(host_io=True)):
        with_rows = _plan(*shape, cuda_device, **extra)
        assert with_rows.info()["workspace_bytes"] >= fused + rows
        with_rows.close()


@pytest.mark.parametrize("precision", ["split_bf16", "fp16"])
@pytest.mark.parametrize("U,V,planes,k_split", [(23, 24, 16, 0), (5, 5, 16, 3), (9, 9, 24, 8), (4, 4, 30, 16)])
def test_checked_plan_with_an_empty_split(U, V, planes, k_split, precision, cuda_device):
    """K splits that leave the last one without a chunk (nk chunks in ceil(nk / k) per split) are no violation."""
    import torch
    import paper_2404_07293_gb300 as scw
    W, g, a, *_ = wl.random_layer_set(U + V, U, V, 2)
    fields = []
    for debug in (False, True):
        plan = scw.Plan(U=U, V=V, L=2, lam=1.0, X=3.1, Y=2.7, z_bounds=np.array([0.0, 0.4, 0.7]), Fx=64, Fy=32,
                        z_planes=wl.cell_centred_planes(0.0, 0.7, planes), precision=precision, k_split=k_split,
                        debug_bounds=debug)
        plan.set_layers(*(torch.from_numpy(np.ascontiguousarray(x)).to(cuda_device) for x in (W, g, a)))
        fields.append(plan.synthesize())
        plan.check()
        plan.close()
    assert torch.equal(*fields)
