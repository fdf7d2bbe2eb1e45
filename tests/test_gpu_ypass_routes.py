"""GPU: the y-direction of plans that run it as a kernel of its own takes folds of up to 24 positions from registers
and longer ones from shared memory. A batch with folds on both sides of the line launches both kernels and gives
every item the bits of its single plan, at the edges of each kernel's tiles and residue shares."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


# rows wider than the one-kernel form takes; short and tall columns, few and many planes
@pytest.mark.parametrize("Fx,Fy,planes,items_per_fold", [(264, 8, 3, 1), (264, 64, 24, 3), (320, 72, 1, 2), (1024, 64, 8, 4)])
def test_batch_on_both_sides_of_the_line(Fx, Fy, planes, items_per_fold, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    items, dev = [], []
    for k in range(2 * items_per_fold):
        U, V = 5 + k, (24, 25)[k % 2]  # 24 and 32 fold positions
        W, g, a, *_ = wl.random_layer_set(30 + k, U, V, 1)
        items.append(dict(U=U, V=V, L=1, lam=1.0, X=3.0, Y=3.3, z_bounds=np.array([0.0, 0.3]), Fx=Fx, Fy=Fy,
                          z_planes=wl.cell_centred_planes(0.0, 0.3, planes), k_split=1))
        dev.append(tuple(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    bp = scw.BatchedPlan(items)
    for i, d in enumerate(dev):
        bp.set_layers(i, *d)
    outs = bp.synthesize()
    bp.check()
    assert bp.info()["kernels_per_synthesis"] == 5  # phases, contraction, x-pass, both y-pass kernels
    for kw, d, out in zip(items, dev, outs):
        plan = scw.Plan(**kw)
        plan.set_layers(*d)
        assert torch.equal(plan.synthesize(), out)
        # the allocation-free kernel: two FP32 sums of at most 40 terms each, relative error about sqrt(40) 2^-24
        ref = plan.recompose(plan.spectrum())
        assert torch.linalg.vector_norm(out - ref) <= 2e-6 * torch.linalg.vector_norm(ref)
        plan.check()
        plan.close()
    bp.close()
