"""Stacks stepped together by pet.Batch give the bits they give alone, for the classes that the TOF stacks,
the 3-D prior and detection factors make; TV with detection factors against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def make(N, P, T, attn, rdp3d, seed, rho=1.0):
    V, M, nb = 20, 4, int(1.45 * N / rho) | 1
    tof = dict(tof_bins=T, tof_bin_mm=7.0, tof_fwhm_mm=11.0) if T else {}
    g = pet.Geometry(N, P, 1.0, V, nb, rho, M, 0.01, **tof)
    rng = np.random.default_rng(seed)
    shape = (P, V, nb) + ((T,) if T else ())
    counts = torch.from_numpy(rng.poisson(3.0, shape).astype(np.int32)).to(DEV)
    gamma = torch.from_numpy(rng.uniform(0.5, 2.0, shape).astype(np.float32)).to(DEV)
    mult = torch.from_numpy(rng.uniform(0.4, 1.0, shape).astype(np.float32)).to(DEV) if attn else None
    p = synth.AlgoParams(iterations=2, beta=0.05, rdp3d=rdp3d, **synth.P2_WORKLOAD)
    return g, lambda: pet.State(g, counts, gamma, pet.make_params(p), torch.ones((P, N, N), device=DEV), d_mult=mult)


# TOF stacks on both sides of the bound of their projector (planes x TOF bins), two shared-memory shapes of
# it, three candidate bins; the 3-D prior and detection factors with and without TOF
SCANS = [(30, 41, 13, False, 0), (25, 17, 9, False, 0), (22, 9, 5, False, 0), (30, 41, 13, True, 0), (24, 57, 64, True, 0),
         (28, 9, 0, True, 0), (31, 17, 0, False, 1), (20, 10, 0, True, 1), (26, 12, 0, False, 0)]


def test_stacks_in_a_batch():
    scans = [make(*s, seed=k) for k, s in enumerate(SCANS)] + [make(24, 33, 9, False, 0, 99, rho=0.6)]
    alone = []
    for g, new in scans:
        s = new()
        img = torch.empty((g.nplanes, g.n, g.n), device=DEV)
        for _ in range(8):
            s.subiter()
        s.read_image(img)
        torch.cuda.synchronize()
        alone.append(img.cpu().numpy())
        s.close()
    for graph in (False, True):
        stream, batch = torch.cuda.Stream(), pet.Batch(capacity=24, use_graph=graph)
        states = [new() for _, new in scans + scans]
        for k, s in enumerate(states):
            batch.add(s, with_objective=k % 2 == 0, stream=stream)
        while batch.step(stream=stream) > 0:
            pass
        for (g, _), s, want in zip(scans + scans, states, alone + alone):
            img = torch.empty((g.nplanes, g.n, g.n), device=DEV)
            s.read_image(img, stream=stream)
            stream.synchronize()
            np.testing.assert_array_equal(img.cpu().numpy(), want)
        batch.close()


# planes that fill and cut a group of eight, TV steps in one and in several passes; tolerance as for every
# FP32 path
@pytest.mark.parametrize("P,steps", [(1, 10), (9, 3), (16, 12)])
def test_tv_with_detection_factors(P, steps):
    N = 34
    w = synth.Workload("t", N, P, 4.0, 20, 49, 4.0, 4, 5e5 * P, "ellipsoid3d" if P > 1 else "ellipses2d",
                       synth.AlgoParams(iterations=2, beta=0.05, reg=1, tv_iters=steps, **synth.P2_WORKLOAD), plane_mm=4.0, seed=P)
    scan = synth.make_scan(w)
    mult = np.asarray(synth.random_image(scan["gamma"].shape, seed=P, lo=0.4, hi=1.0), np.float32)
    g, og = pet.Geometry.from_dict(w.geometry(), scan["sens"]), oracle.geom_from(w.geometry(), scan["sens"])
    s = pet.State(g, torch.from_numpy(scan["counts"]).to(DEV), torch.from_numpy(scan["gamma"]).to(DEV),
                  pet.make_params(w.params), torch.ones((P, N, N), device=DEV), d_mult=torch.from_numpy(mult).to(DEV))
    for _ in range(6):
        s.subiter()
    ref, _ = oracle.reconstruct(og, scan["counts"], scan["gamma"], w.params, np.ones((P, N, N)), nsub=6, mult=mult)
    img = torch.empty((P, N, N), dtype=torch.float64, device=DEV)
    s.read_image(img)
    torch.cuda.synchronize()
    assert np.linalg.norm(img.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
