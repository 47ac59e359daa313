"""The stack kernels at the sizes where their dispatch changes, against the oracle: the tiled TV steps,
the TOF projection and gather of stacks, the 3-D prior with per-voxel sensitivities, the two by two
backprojection, and the FP64 walk on both sides of its integer positions.

Tolerances are those of every path: FP32 1e-5 per projection (of its largest value), of the largest
backprojected value, and relL2 on the image after a few subiterations; FP64 1e-10."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


def rel_l2(got, ref):
    return float(np.linalg.norm(np.asarray(got, np.float64) - ref) / np.linalg.norm(ref))


# single planes and stacks, tiles of 16 and of 32 cut by the image, and step counts around the steps
# per launch (one step runs the untiled kernels)
@pytest.mark.parametrize("N,P", [(15, 1), (33, 1), (17, 2), (64, 9), (130, 41)])
@pytest.mark.parametrize("iters", [1, 2, 5, 11])
def test_tv_steps(N, P, iters):
    g = pet.Geometry(N, P, 2.0, 8, int(1.5 * N) | 1, 2.0, 2, 0.9)
    rng = np.random.default_rng(N + P)
    z, W = f32(rng.uniform(-0.5, 3.0, (P, N, N))), f32(rng.uniform(0.2, 2.0, (P, N, N)))
    px, py = torch.zeros((P, N, N), device=DEV), torch.zeros((P, N, N), device=DEV)
    x = torch.empty((P, N, N), device=DEV)
    pet.tv_prox(g, dev(z), dev(W), 0.3, iters, px, py, x)
    torch.cuda.synchronize()
    ref, (rx, ry) = oracle.tv_prox(z, W, 0.3, iters)
    assert rel_l2(x.cpu().numpy(), ref) <= 1e-5
    assert np.abs(px.cpu().numpy() - rx).max() <= 1e-5 and np.abs(py.cpu().numpy() - ry).max() <= 1e-5


# (N, P, T, TOF bin mm, FWHM mm, rho): planes on both sides of the stack kernel's bound, one to three
# slices of TOF bins, windows narrower and wider than the field, three candidate bins
TOF = [(40, 41, 13, 20.0, 30.0, 1.0), (33, 57, 21, 9.0, 12.0, 1.0), (24, 48, 7, 60.0, 80.0, 0.6),
       (30, 17, 15, 12.0, 25.0, 1.0), (28, 43, 5, 8.0, 10.0, 1.0),
       # TOF bins so short that the field spans hundreds of them: many pixels lie outside all windows
       (80, 9, 64, 0.8, 12.0, 1.0)]


@pytest.mark.parametrize("geom", TOF)
def test_tof_stacks(geom):
    N, P, T, d, fwhm, rho = geom
    nb = int(1.45 * N / rho) | 1
    w = synth.Workload("tof", N, P, 4.0, 21, nb, 4.0 * rho, 5, 4e5 * P, "ellipsoid3d",
                       synth.AlgoParams(iterations=2, beta=0.05, **synth.P2_WORKLOAD), plane_mm=4.0, seed=P,
                       tof_bins=T, tof_bin_mm=d, tof_fwhm_mm=fwhm)
    scan = synth.make_scan(w)
    g, og = pet.Geometry.from_dict(w.geometry(), scan["sens"]), oracle.geom_from(w.geometry(), scan["sens"])
    x = f32(synth.random_image((P, N, N), seed=T))
    ref = oracle.forward(og, 1, x)
    out = torch.empty(ref.shape, device=DEV)
    pet.forward_subset(g, 1, dev(x), out)
    torch.cuda.synchronize()
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    counts, gamma = dev(scan["counts"], torch.int32), dev(scan["gamma"])
    for prec in (synth.PREC_FP32, synth.PREC_FP32_KAHAN):
        s = pet.State(g, counts, gamma, pet.make_params(w.params, prec), torch.ones((P, N, N), device=DEV))
        for _ in range(5):
            s.subiter()
        ref, _ = oracle.reconstruct(og, scan["counts"], scan["gamma"], w.params, np.ones((P, N, N)), nsub=5)
        img = torch.empty((P, N, N), dtype=torch.float64, device=DEV)
        s.read_image(img)
        torch.cuda.synchronize()
        assert rel_l2(img.cpu().numpy(), ref) <= 1e-5, prec
        s.close()


# planes that end inside, at the end and just past a group of eight
@pytest.mark.parametrize("P", [2, 8, 9, 15])
def test_rdp3d_with_detection_factors(P):
    N = 29
    w = synth.Workload("z", N, P, 4.0, 22, 43, 4.0, 4, 5e5 * P, "ellipsoid3d",
                       synth.AlgoParams(iterations=2, beta=0.05, rdp3d=1, **synth.P2_WORKLOAD), plane_mm=4.0, seed=P)
    scan = synth.make_scan(w)
    g, og = pet.Geometry.from_dict(w.geometry(), scan["sens"]), oracle.geom_from(w.geometry(), scan["sens"])
    mult = np.asarray(synth.random_image(scan["gamma"].shape, seed=P, lo=0.4, hi=1.0), np.float32)
    s = pet.State(g, dev(scan["counts"], torch.int32), dev(scan["gamma"]), pet.make_params(w.params),
                  torch.ones((P, N, N), device=DEV), d_mult=dev(mult))
    for _ in range(6):
        s.subiter()
    ref, _ = oracle.reconstruct(og, scan["counts"], scan["gamma"], w.params, np.ones((P, N, N)), nsub=6, mult=mult)
    img = torch.empty((P, N, N), dtype=torch.float64, device=DEV)
    s.read_image(img)
    torch.cuda.synchronize()
    assert rel_l2(img.cpu().numpy(), ref) <= 1e-5


# three and four lines per 2 x 2 block, five (the general kernel), odd sides, all views and a subset
@pytest.mark.parametrize("N,P,rho", [(31, 2, 1.0), (50, 43, 0.95), (27, 9, 0.75), (22, 17, 0.68), (40, 89, 2.0)])
def test_back_two_by_two(N, P, rho):
    V, M, nb = 25, 3, int(1.45 * N / rho) | 1
    g = pet.Geometry(N, P, 2.0, V, nb, 2.0 * rho, M, 0.7)
    og = oracle.geom(N, P, V, nb, M, pixel_mm=2.0, bin_mm=2.0 * rho, sens=0.7)
    for i in (-1, 1):
        nv = V if i < 0 else g.subset_size(i)
        y = f32(synth.random_image((P, nv, nb), seed=P, lo=-1.0, hi=1.0))
        ref = oracle.back(og, i, y)
        out = torch.empty((P, N, N), device=DEV)
        pet.back_subset(g, i, dev(y), out)
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max(), i


@pytest.mark.parametrize("N,P,R", [(1024, 1, 1), (1025, 1, 1), (67, 11, 1), (40, 3, 7)])
def test_fp64_walk(N, P, R):
    V, M, nb = 6, 2, int(1.45 * N) | 1
    g = pet.Geometry(N, P, 2.0, V, nb, 2.0, M, 0.9, subrays=R)
    og = oracle.geom(N, P, V, nb, M, pixel_mm=2.0, bin_mm=2.0, sens=0.9, subrays=R)
    x = synth.random_image((P, N, N), seed=N)
    ref = oracle.forward(og, 0, x)
    out = torch.empty(ref.shape, dtype=torch.float64, device=DEV)
    pet.forward_subset(g, 0, dev(x, torch.float64), out)
    torch.cuda.synchronize()
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
