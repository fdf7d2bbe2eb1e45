"""GPU: the FP32 contraction's spectra against FP64 at the sizes where its loops can go wrong: splits that end
inside a batch of eight modes, splits without any mode, row blocks with a few rows, odd plane counts in
the 8- and the 16-plane form, and the split the plan chooses itself."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the FP32 path's bound (relative L2); a chain of 256 FP32 terms stays near 4e-7


@pytest.mark.parametrize("U,V,planes,k_split", [
    (1, 1, 1, 1), (1, 1, 2, 3), (3, 1, 5, 1), (3, 3, 7, 5), (5, 7, 8, 3), (9, 9, 9, 11), (9, 9, 17, 0), (13, 13, 16, 7),
    (11, 3, 33, 4), (16, 16, 3, 1), (16, 16, 15, 0), (2, 43, 6, 2), (23, 23, 8, 0), (23, 23, 40, 9), (5, 5, 130, 2)])
def test_spectra_match_fp64(U, V, planes, k_split, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    L, lam = 2, 1.0
    W, g, a, *_ = wl.random_layer_set(31 * U + V + planes, U, V, L)
    zb = np.array([0.0, 0.3, 0.8])
    zp = np.concatenate([0.3 * (np.arange(planes) + 0.5) / planes, 0.3 + 0.5 * (np.arange(planes) + 0.5) / planes])
    plan = scw.Plan(U, V, L, lam, 3.0, 3.3, zb, 16, 16, zp, precision="fp32", k_split=k_split)
    plan.set_layers(*(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    S = plan.spectrum().cpu().numpy().astype(np.complex128).reshape(2, planes, 3 * U * V)
    plan.check()
    plan.close()
    M = U * V
    for l in range(L):
        ref_z = np.concatenate([np.full(2 * M, zb[l]), np.full(2 * M, zb[l + 1])])
        z = zp[l * planes:(l + 1) * planes]
        c = a[l][:, None] * np.exp(2j * np.pi / lam * g[l][:, None] * (z[None, :] - ref_z[:, None]))
        ref = (W[l].astype(np.complex128) @ c).T
        err = np.linalg.norm(S[l] - ref) / np.linalg.norm(ref)
        assert err <= TOL, (l, err)
