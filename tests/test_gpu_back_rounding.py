"""The stand-alone backprojection of stacks (two by two pixels per thread) is no less exact than that of
single planes, which adds every view by one compensated step: it rounds scale (s + e) once."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


# three and four bins per two by two block, few and many views (0.93: at 0.9 the tenth line of an axis view
# lies on a pixel edge but for the rounding of 1.17 / 1.3, and FP32 and FP64 take either side)
@pytest.mark.parametrize("N,P,V,rho", [(64, 9, 96, 1.0), (51, 17, 40, 1.1), (48, 8, 200, 0.93)])
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
