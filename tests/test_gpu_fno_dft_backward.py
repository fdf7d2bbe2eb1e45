"""GPU: the backward truncated DFT with the weight gradient at kept-mode counts other than the benchmark's, with enough
samples that a CTA walks several tiles of every tile width. The loss is a mean over samples, so a batch's gradient is the
mean of its halves' gradients: halving the batch scales every value by two, which BF16 keeps, and regroups FP32 sums."""
import numpy as np
import pytest

from oracle import fno
from test_gpu_fno import _case, _compare_grads, _surrogate

pytestmark = pytest.mark.gpu


# tiles of 16 (4 modes), 32 and 48 (8 modes), 96 (12 modes), 144 columns (32 modes); ragged last row and column tiles
@pytest.mark.parametrize("modes,batch", [(4, 322), (8, 324), (8, 620), (12, 326), (32, 146)])
def test_gradient_equals_the_mean_of_the_halves(modes, batch, cuda_device):
    import torch
    sh = fno.FnoShape(width=32, grid=32, modes=modes, layers=2, slices=2, in_grid=16)
    flat, n, E = _case(sh, batch, seed=modes + batch)
    grads = []
    for lo, hi in ((0, batch), (0, batch // 2), (batch // 2, batch)):
        s = _surrogate(sh, hi - lo, "bf16")
        s.set_params(flat)
        s.forward_backward(torch.from_numpy(np.ascontiguousarray(n[lo:hi])).to(cuda_device),
                           torch.from_numpy(np.ascontiguousarray(E[lo:hi])).to(cuda_device))
        grads.append(s.grads().astype(np.float64))
        s.close()
    _compare_grads(grads[0], 0.5 * (grads[1] + grads[2]), sh, 1e-4)
