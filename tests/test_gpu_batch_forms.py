"""GPU: kernels of a batch that its items choose by their plane slots, illuminations and precision give every item the
bits of its own plan with the same split; and the contraction of 128 plane slots, whose operands have rings of their own,
reports a stage that nothing fills and recovers."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _item(k, U, V, planes, illuminations, device, exterior):
    import torch
    W, g, a, pi, pr, pt = wl.random_layer_set(50 + k, U, V, 2)
    if illuminations > 1:
        a, pi, pr, pt = wl.random_illuminations(60 + k, illuminations, U, V, 2)
    zp = wl.cell_centred_planes(0.0, 0.8, planes)
    if exterior:
        zp = np.concatenate([[-0.3, -0.1], zp, [0.9]])
    kw = dict(U=U, V=V, L=2, lam=1.0, X=3.0, Y=3.3, z_bounds=np.array([0.0, 0.3, 0.8]), Fx=32, Fy=24, z_planes=zp, k_split=2,
              exterior=exterior, illuminations=illuminations)
    dev = [torch.from_numpy(np.ascontiguousarray(x)).to(device) for x in (W, g, a, pi, pr, pt)]
    return kw, dev if exterior else dev[:3]


# (orders, planes, illuminations) of each item: mixed illuminations; up to 16, 64 and 128 plane slots; all of them
@pytest.mark.parametrize("items", [
    [(5, 5, 6, 1), (7, 3, 4, 2), (4, 6, 3, 5)],
    [(5, 5, 20, 1), (9, 9, 30, 1)],
    [(5, 5, 110, 1), (9, 9, 150, 1)],
    [(3, 3, 256, 1), (13, 13, 40, 1)],
    [(6, 6, 30, 7), (7, 7, 12, 1), (3, 9, 9, 16)],
])
@pytest.mark.parametrize("exterior", [False, True])
@pytest.mark.parametrize("precision", ["split_bf16", "fp16", "fp32"])
def test_batch_equals_single_plans(items, exterior, precision, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    made = [_item(k, *it, cuda_device, exterior) for k, it in enumerate(items)]
    bp = scw.BatchedPlan([kw for kw, _ in made], precision=precision)
    for i, (_, dev) in enumerate(made):
        bp.set_layers(i, *dev)
    for _ in range(3):  # launches, capture, replay
        outs = bp.synthesize()
    bp.check()
    for (kw, dev), out in zip(made, outs):
        plan = scw.Plan(precision=precision, **kw)
        plan.set_layers(*dev)
        ref = plan.synthesize()
        plan.check()
        assert torch.equal(ref, out), (kw["U"], kw["illuminations"])
        plan.close()
    bp.close()


@pytest.mark.parametrize("precision", ["split_bf16", "fp16"])
@pytest.mark.parametrize("V,planes,k_split", [(3, 100, 1), (15, 256, 0), (9, 128, 3)])
def test_stall_in_the_wide_contraction_is_reported(precision, V, planes, k_split, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    W, g, a, *_ = wl.random_layer_set(3, V, V, 1)
    plan = scw.Plan(V, V, 1, 1.0, 4.0, 4.0, np.array([0.0, 1.0]), 16, 16, wl.cell_centred_planes(0.0, 1.0, planes),
                    precision=precision, k_split=k_split)
    plan.set_layers(*(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    assert plan.info()["planes_per_layer_pad"] == 128
    ref = plan.synthesize().clone()
    plan.check()
    plan.set_timeout_ns(5_000_000)
    plan.inject_stall(True)
    plan.synthesize()
    with pytest.raises(scw.ScwError) as err:
        plan.check()
    assert err.value.status == 5  # SCW_ERR_TIMEOUT
    plan.inject_stall(False)
    plan.set_timeout_ns(2_000_000_000)
    again = plan.synthesize()
    plan.check()
    assert torch.equal(again, ref)
    plan.close()
