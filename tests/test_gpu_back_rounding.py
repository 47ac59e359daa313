"""The stand-alone backprojection of stacks (two by two pixels per thread) is no less exact than that of
single planes, which adds every view by one compensated step: it rounds scale (s + e) once."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


# three and four bins per two by two block, stacks on the two by two kernel's side of its bound: six to 32
# plane groups and tiles that fill the SMs (no line of an axis view lies on a pixel edge but for rounding,
# where FP32 and FP64 may take either side)
SIZES = [(127, 121, 24, 1.0), (200, 41, 16, 1.13), (91, 250, 40, 0.93)]


@pytest.mark.parametrize("N,P,V,rho", SIZES)
def test_error_against_single_planes(N, P, V, rho):
    nb = int(1.45 * N / rho) | 1
    y = np.random.default_rng(N).uniform(0.1, 2.0, (P, V, nb)).astype(np.float32)
    ref = oracle.back(oracle.geom(N, P, V, nb, 4, pixel_mm=1.3, bin_mm=1.3 * rho, sens=0.7), -1, y.astype(np.float64))
    err = []
    for planes in (P, 1):
        g = pet.Geometry(N, planes, 1.3, V, nb, 1.3 * rho, 4, 0.7)
        out = torch.empty((P, N, N), device=DEV)
        for z in range(0, P, planes):
            pet.back_subset(g, -1, torch.from_numpy(y[z:z + planes]).to(DEV), out[z:z + planes])
        torch.cuda.synchronize()
        err.append(np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref))
    assert err[0] <= err[1]


# and the largest group count, one group per block row, against the oracle; all views and a subset
@pytest.mark.parametrize("N,P,V,rho", [(34, 2040, 6, 1.0), (129, 128, 9, 0.93), (199, 48, 7, 2.0)])
def test_two_by_two_against_oracle(N, P, V, rho):
    nb = int(1.45 * N / rho) | 1
    g = pet.Geometry(N, P, 1.3, V, nb, 1.3 * rho, 3, 0.7)
    og = oracle.geom(N, P, V, nb, 3, pixel_mm=1.3, bin_mm=1.3 * rho, sens=0.7)
    for i in (-1, 1):
        nv = V if i < 0 else g.subset_size(i)
        y = np.random.default_rng(P).uniform(-1.0, 1.0, (P, nv, nb)).astype(np.float32)
        out = torch.empty((P, N, N), device=DEV)
        pet.back_subset(g, i, torch.from_numpy(y).to(DEV), out)
        torch.cuda.synchronize()
        ref = oracle.back(og, i, y.astype(np.float64))
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max(), i
