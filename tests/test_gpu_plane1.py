"""Single-plane FP32 scans (csrc/plane1.cu) against the oracle at the sizes where their kernels'
dispatch changes: every count of lanes per pixel, patches cut by the image edge, more views in a
subset than a warp holds at a time, two to four candidate bins, sinograms narrower than the image,
and sub-ray counts on both sides of the closed sums' threshold.

Tolerances as for every FP32 path: 1e-5 per projection (of its largest value), 1e-5 relL2 on the
image after a few subiterations."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")

# (N, V, NB, M, rho, subrays)
GEOMS = [
    (37, 9, 55, 9, 1.0, 1),        # one view per subset: one lane per pixel
    (64, 60, 91, 6, 1.0, 1),       # 10 views per subset
    (65, 70, 93, 2, 1.0, 1),       # 35 views per subset: two rounds of held views
    (131, 24, 150, 3, 1.0, 1),     # 8 lanes, patches cut on both edges
    (50, 20, 31, 4, 1.0, 1),       # the sinogram covers part of the image
    (41, 21, 121, 3, 0.5, 1),      # three candidate bins
    (30, 16, 115, 2, 0.37, 1),     # four candidate bins
    (50, 12, 25, 3, 3.0, 1),       # bins wider than pixels
    (48, 20, 69, 4, 1.0, 5),       # sub-rays walked one by one
    (48, 20, 69, 4, 1.0, 6),       # the fewest taken in closed form
    (47, 18, 27, 3, 2.6, 64),
]


@pytest.mark.parametrize("geom", GEOMS)
def test_single_plane_against_oracle(geom):
    N, V, NB, M, rho, R = geom
    w = synth.Workload("p1", N, 1, 4.0, V, NB, 4.0 * rho, M, 3e6, "ellipses2d",
                       synth.AlgoParams(iterations=3, beta=0.05, **synth.P2_WORKLOAD), seed=N + V, subrays=R)
    scan = synth.make_scan(w)
    g, og = pet.Geometry.from_dict(w.geometry(), scan["sens"]), oracle.geom_from(w.geometry(), scan["sens"])
    x = np.asarray(synth.random_image((1, N, N), seed=V), np.float32)
    xd = torch.from_numpy(x).to(DEV)
    for i in list(range(M)) + [-1]:
        ref = oracle.forward(og, i, x.astype(np.float64))
        out = torch.empty(ref.shape, dtype=torch.float32, device=DEV)
        pet.forward_subset(g, i, xd, out)
        torch.cuda.synchronize()
        den = np.abs(ref).max(axis=-1, keepdims=True)
        assert np.all(np.abs(out.cpu().numpy() - ref) <= 1e-5 * den), i
    counts, gamma = torch.from_numpy(scan["counts"]).to(DEV), torch.from_numpy(scan["gamma"]).to(DEV)
    for prec in (synth.PREC_FP32, synth.PREC_FP32_KAHAN):
        s = pet.State(g, counts, gamma, pet.make_params(w.params, prec), torch.ones((1, N, N), device=DEV))
        for nsub in (1, 5):                       # before and inside the dynamic-nu range
            while s.subiters < nsub:
                s.subiter()
            ref, _ = oracle.reconstruct(og, scan["counts"], scan["gamma"], w.params, np.ones((1, N, N)), nsub=nsub)
            out = torch.empty((1, N, N), dtype=torch.float64, device=DEV)
            s.read_image(out)
            torch.cuda.synchronize()
            err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= 1e-5, (prec, nsub, err)
        s.close()
