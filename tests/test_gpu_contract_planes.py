"""GPU: spectra of units with many planes on the tensor cores against FP64: 64 and 128 plane slots, one slot more
or less, layers cut into several units, row tiles with a few rows, splits that leave one or no chunk."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

# relative L2. BF16 pairs: each factor is kept to 2^-18 and the product of the low halves (2^-18) is left out;
# FP16: each factor is rounded to 2^-11
TOL = {"split_bf16": 2e-5, "fp16": 1e-3}


@pytest.mark.parametrize("precision", ["split_bf16", "fp16"])
@pytest.mark.parametrize("U,V,planes,k_split", [
    (1, 1, 65, 1), (1, 1, 128, 1), (3, 3, 64, 2), (3, 3, 66, 2), (5, 7, 100, 3), (7, 7, 17, 1), (7, 7, 127, 4), (9, 9, 129, 5),
    (9, 9, 300, 0), (13, 13, 90, 1), (13, 13, 16, 9), (16, 16, 120, 0), (43, 2, 70, 6), (23, 23, 80, 0), (23, 23, 33, 7)])
def test_spectra_match_fp64(precision, U, V, planes, k_split, cuda_device):
    import torch
    import paper_2404_07293_gb300 as scw
    L, lam = 2, 1.0
    W, g, a, *_ = wl.random_layer_set(17 * U + V + planes, U, V, L)
    zb = np.array([0.0, 0.3, 0.8])
    t = (np.arange(planes) + 0.5) / planes
    plan = scw.Plan(U, V, L, lam, 3.0, 3.3, zb, 16, 16, np.concatenate([0.3 * t, 0.3 + 0.5 * t]), precision=precision, k_split=k_split)
    plan.set_layers(*(torch.from_numpy(x).to(cuda_device) for x in (W, g, a)))
    S = plan.spectrum().cpu().numpy().astype(np.complex128).reshape(2, planes, 3 * U * V)
    plan.check()
    plan.close()
    M = U * V
    for l in range(L):
        ref_z = np.concatenate([np.full(2 * M, zb[l]), np.full(2 * M, zb[l + 1])])
        z = (0.3 * t, 0.3 + 0.5 * t)[l]
        c = a[l][:, None] * np.exp(2j * np.pi / lam * g[l][:, None] * (z[None, :] - ref_z[:, None]))
        ref = (W[l].astype(np.complex128) @ c).T
        err = np.linalg.norm(S[l] - ref) / np.linalg.norm(ref)
        assert err <= TOL[precision], (l, err)
