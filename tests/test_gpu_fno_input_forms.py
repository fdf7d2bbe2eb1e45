"""GPU: the surrogate's backward pass takes the lift gradient by one of two kernels, chosen by the address of the input.
Going from one to the other repeats no set-up: the call can be recorded in a graph, with the gradient of a direct call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# 304 is the most partial rows that the tensor-core form writes; 160 and 40 inputs of 16 x 16 and 32 x 32 pixels give
# the general form more, 2 as many
@pytest.mark.parametrize("grid,in_grid,batch", [(32, 16, 160), (64, 32, 40), (32, 16, 2)])
def test_switching_the_form_under_capture(grid, in_grid, batch, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    s = scw.Surrogate(grid=grid, modes=4, layers=2, slices=2, in_grid=in_grid, batch_max=batch, seed=3)
    rng = np.random.default_rng(batch)
    n = torch.from_numpy((1.3 + 0.1 * rng.standard_normal((batch, 2, in_grid, in_grid))).astype(np.complex64)).to(cuda_device)
    t = torch.from_numpy((rng.standard_normal((batch, 3, grid, grid))).astype(np.complex64)).to(cuda_device)
    off = torch.empty(n.numel() + 1, dtype=n.dtype, device=cuda_device)[1:].view(n.shape)  # off the 16-byte grid
    off.copy_(n)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    direct = []
    with torch.cuda.stream(side):
        for x in (n, off):
            s.forward_backward(x, t, read_loss=False)
            direct.append(s.grads())
        for x, want in ((n, direct[0]), (off, direct[1])):  # the call before took the other form
            graph = torch.cuda.CUDAGraph()
            graph.capture_begin(capture_error_mode="thread_local")
            s.forward_backward(x, t, read_loss=False)
            graph.capture_end()
            graph.replay()
            assert np.array_equal(s.grads(), want)
    assert np.linalg.norm(direct[0] - direct[1]) <= 1e-4 * np.linalg.norm(direct[0])
    s.close()
