"""GPU: the truncated DFT's tile width is chosen per batch size (narrow tiles for few samples, wide
ones for many, several tiles per CTA above 300 samples) and only one mode of each conjugate pair is
multiplied. Every output is the same sum in the same order whatever the tile, so a sample's field
and error estimate must not depend on the batch it came in, bit for bit."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

scw = pytest.importorskip("paper_2404_07293_gb300")


@pytest.mark.parametrize("batch", [3, 5, 37, 68, 72, 130, 200, 256, 310])
def test_a_sample_does_not_depend_on_its_batch(batch, cuda_device):
    import torch
    few = wl.phantom_batch(900, 3).astype(np.complex64)
    n = np.repeat(few[:1], batch, axis=0)
    n[0], n[batch // 2], n[-1] = few[0], few[1], few[2]
    s = scw.Surrogate(grid=64, modes=16, layers=2, slices=8, in_grid=32, batch_max=batch, seed=5)
    field, est, _ = s.infer(torch.from_numpy(n).to(cuda_device))
    for b, k in ((0, 0), (batch // 2, 1), (batch - 1, 2)):
        f1, e1, _ = s.infer(torch.from_numpy(few[k:k + 1]).to(cuda_device))
        assert torch.equal(field[b], f1[0]) and torch.equal(est[b], e1[0]), (batch, b)
    s.close()
