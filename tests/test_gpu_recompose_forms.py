"""GPU: the recomposition's forms agree bit for bit. Plans with index checks run the two-kernel form
(x-pass rows through memory); the others run both directions in one kernel where the plan fits it, or the
register y-pass, or the shared-memory y-pass for long folds. All of them add the same terms in the same
order, so the field may not differ in any bit."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

# U, V, Fx, Fy, planes, extra arguments: every fold length class (V = 1 .. 56: 8 to 56 positions), one and two
# columns per thread, widths from one residue to the widest fused row and beyond, ragged last rounds
CASES = [
    (1, 1, 8, 8, 24, {}), (7, 5, 16, 24, 30, {}), (3, 8, 72, 40, 25, {}), (9, 9, 136, 64, 40, {}),
    (16, 16, 200, 72, 23, {}), (21, 17, 248, 16, 30, {}), (23, 24, 256, 48, 22, {}), (5, 25, 64, 80, 40, {}),
    (13, 33, 128, 32, 30, {}), (11, 41, 256, 24, 24, {}), (4, 48, 104, 40, 28, {}), (3, 49, 64, 64, 24, {}),
    (9, 56, 48, 32, 24, {}), (9, 9, 264, 32, 24, {}), (15, 31, 320, 24, 24, {}), (30, 7, 512, 16, 24, {}),
    (9, 7, 40, 2048, 22, {}), (9, 11, 48, 24, 30, dict(tiles=(2, 3))), (6, 27, 24, 40, 30, dict(tiles=(3, 1))),
    (9, 9, 32, 32, 12, dict(illuminations=3)), (7, 7, 96, 64, 180, {}), (7, 7, 64, 64, 300, dict(k_split=7)),
]


@pytest.mark.parametrize("U,V,Fx,Fy,planes,extra", CASES)
@pytest.mark.parametrize("precision", ["split_bf16", "fp32"])
def test_forms_are_bit_identical(U, V, Fx, Fy, planes, extra, precision, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    L, I = 2, extra.get("illuminations", 1)
    W, g, a, pi, pr, pt = wl.random_layer_set(U * 100 + V, U, V, L)
    if I > 1:
        a, pi, pr, pt = wl.random_illuminations(7, I, U, V, L)
    zb = np.array([0.0, 0.4, 0.7])
    zp = np.concatenate([[-0.2], wl.cell_centred_planes(0.0, 0.7, planes - 2), [0.9]])
    kw = dict(U=U, V=V, L=L, lam=1.0, X=3.1, Y=2.7, z_bounds=zb, Fx=Fx, Fy=Fy, z_planes=zp, x0=0.13, y0=-0.4,
              exterior=True, precision=precision, **dict(dict(k_split=2), **extra))
    dev = [torch.from_numpy(np.ascontiguousarray(x)).to(cuda_device) for x in (W, g, a, pi, pr, pt)]
    fields = []
    for checked in (False, True):
        plan = scw.Plan(debug_bounds=checked, **kw)
        plan.set_layers(*dev)
        fields.append(plan.synthesize())
        plan.check()
        plan.close()
    assert torch.equal(fields[0], fields[1])


def test_batch_of_mixed_folds_equals_single_plans(cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    items, dev = [], []
    for k, (U, V, Fx, Fy, n) in enumerate([(9, 9, 64, 32, 16), (5, 25, 40, 64, 8), (21, 17, 256, 24, 12), (3, 48, 24, 16, 9)]):
        W, g, a, *_ = wl.random_layer_set(70 + k, U, V, 2)
        zb = np.array([0.0, 0.3, 0.8])
        items.append(dict(U=U, V=V, L=2, lam=1.0, X=3.0, Y=3.3, z_bounds=zb, Fx=Fx, Fy=Fy,
                          z_planes=wl.cell_centred_planes(0.0, 0.8, n), k_split=1))
        dev.append(tuple(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    bp = scw.BatchedPlan(items)
    for i, d in enumerate(dev):
        bp.set_layers(i, *d)
    outs = bp.synthesize()
    bp.check()
    for kw, d, out in zip(items, dev, outs):
        plan = scw.Plan(debug_bounds=True, **kw)
        plan.set_layers(*d)
        assert torch.equal(plan.synthesize(), out)
        plan.close()
    bp.close()
