"""GPU: the surrogate's pixel kernels in BF16 mode have forms chosen by the upsampling factor, the input row and
the slice count (lift by pixel pairs, lift backward and projection sums on the tensor cores, the general
kernels elsewhere). Loss, gradients and field against the FP64 oracle at the edges of each choice."""
import numpy as np
import pytest

from oracle import fno
from test_gpu_fno import TOL, _case, _compare_grads, _surrogate
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,in_grid,slices,batch", [
    (32, 16, 3, 3), (32, 16, 8, 2), (32, 16, 9, 1), (32, 16, 16, 2),  # 2 x 2 upsampling: two and four feature tiles
    (64, 32, 1, 2),                                                    # one slice, two units per row
    (16, 8, 5, 3),                                                     # rows shorter than a unit
    (32, 32, 2, 2), (64, 16, 9, 2), (32, 4, 2, 1),                     # factors 1, 4 and 8
])
def test_pixel_kernel_forms_match_oracle(grid, in_grid, slices, batch, cuda_device):
    import torch
    sh = fno.FnoShape(width=32, grid=grid, modes=4, layers=2, slices=slices, in_grid=in_grid)
    flat, n, E = _case(sh, batch, seed=grid + in_grid + slices)
    s = _surrogate(sh, batch, "bf16")
    s.set_params(flat)
    nd, Ed = torch.from_numpy(n).to(cuda_device), torch.from_numpy(E).to(cuda_device)
    loss = s.forward_backward(nd, Ed)
    g = s.grads().astype(np.float64)
    L, Lf, Lh, gref = fno.loss_and_grads(flat.astype(np.float64), n.astype(np.complex128),
                                          fno.channels_from_field(E.astype(np.complex128)), sh)
    assert abs(loss[1] - Lf) <= TOL["bf16"] * abs(Lf) and abs(loss[2] - Lh) <= TOL["bf16"] * max(abs(Lh), 1.0)
    _compare_grads(g, gref, sh, TOL["bf16"])
    field, _, _ = s.infer(nd)
    ref = fno.field_from_channels(fno.forward(flat.astype(np.float64), n.astype(np.complex128), sh)[0])
    got = field.cpu().numpy()
    assert max(max(rel_l2(got[b], ref[b])) for b in range(batch)) <= TOL["bf16"]
    # inputs off the 16-byte grid take the general forms: the same values up to the order of FP32 sums
    off = torch.empty(nd.numel() + 1, dtype=nd.dtype, device=nd.device)[1:].view(nd.shape)
    offE = torch.empty(Ed.numel() + 1, dtype=Ed.dtype, device=Ed.device)[1:].view(Ed.shape)
    off.copy_(nd)
    offE.copy_(Ed)
    loss2 = s.forward_backward(off, offE)
    assert np.allclose(loss, loss2, rtol=1e-5)
    assert np.linalg.norm(s.grads() - g) <= 1e-4 * np.linalg.norm(g)
    s.close()
