"""Bins many pixels wide with several lines each: ring bins whose lines are summed in closed form, line by
line, and (7 and 9 pixels) on both sides of the bound between the two, against the FP64 oracle.
Tolerances as for every FP32 path: 1e-5 of the largest projected and backprojected value, 1e-5 relL2 on
the image after a few subiterations."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("N,P,R", [(48, 1, 32), (29, 9, 6), (61, 1, 64)])
@pytest.mark.parametrize("wide,ring", [(7.0, True), (9.0, True), (70.0, True), (300.0, True), (2000.0, True),
                                       (7.0, False), (9.0, False), (70.0, False)])
def test_wide_bins(wide, ring, N, P, R):
    V, M = 16, 2
    nb = max(4, int(1.45 * N / wide) + 2)
    kw = dict(subrays=R, ring_mm=nb * wide if ring else 0.0)
    g = pet.Geometry(N, P, 1.0, V, nb, wide, M, 0.9, **kw)
    og = oracle.geom(N, P, V, nb, M, pixel_mm=1.0, bin_mm=wide, sens=0.9, **kw)
    x = np.asarray(synth.random_image((P, N, N), seed=N, lo=0.1, hi=2.0), np.float32)
    y = np.asarray(synth.random_image((P, V, nb), seed=R, lo=0.5, hi=1.5), np.float32)
    fwd, back = torch.empty((P, V, nb), device=DEV), torch.empty((P, N, N), device=DEV)
    pet.forward_subset(g, -1, torch.from_numpy(x).to(DEV), fwd)
    pet.back_subset(g, -1, torch.from_numpy(y).to(DEV), back)
    torch.cuda.synchronize()
    for got, ref in ((fwd, oracle.forward(og, -1, x.astype(np.float64))), (back, oracle.back(og, -1, y.astype(np.float64)))):
        assert np.abs(got.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    counts = np.random.default_rng(N).poisson(5.0, (P, V, nb)).astype(np.int32)
    gamma = np.full((P, V, nb), 1.0, np.float32)
    p = synth.AlgoParams(iterations=2, beta=0.05, **synth.P2_WORKLOAD)
    s = pet.State(g, torch.from_numpy(counts).to(DEV), torch.from_numpy(gamma).to(DEV), pet.make_params(p),
                  torch.ones((P, N, N), device=DEV))
    for _ in range(3):
        s.subiter()
    ref, _ = oracle.reconstruct(og, counts, gamma, p, np.ones((P, N, N)), nsub=3)
    img = torch.empty((P, N, N), dtype=torch.float64, device=DEV)
    s.read_image(img)
    torch.cuda.synchronize()
    assert np.linalg.norm(img.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    s.close()
