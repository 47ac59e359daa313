"""Kernels that share one reconstruction's sums out differently give the same sums.

The single-plane update (csrc/plane1.cu) adds a pixel's views in order whatever the number of lanes per
pixel: with beta = 0 and without nu it gives the bits of the generic update, which the TV variant of
the same scan runs (its proximal step is the identity at beta = 0).  Its projection takes one
compensated step per driving step and joins a ray's chunks in order with their compensations."""
import numpy as np
import pytest
import torch

from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")

# (N, V, NB, M, bin / pixel, subrays, ring radius in pixels)
GEOMS = [
    (203, 72, 297, 2, 1.0, 1, 0),   # one lane per pixel, 36 views: two rounds of held views, patches cut
    (150, 40, 219, 2, 1.0, 1, 0),   # two lanes
    (131, 70, 191, 2, 1.0, 1, 0),   # four lanes, 35 views
    (65, 70, 95, 2, 1.0, 1, 0),     # eight lanes, 35 views
    (37, 9, 55, 9, 1.0, 1, 0),      # one view per subset
    (50, 20, 31, 4, 1.0, 1, 0),     # the sinogram covers part of the image
    (60, 40, 175, 2, 0.5, 1, 0),    # three candidate bins
    (48, 20, 69, 4, 1.0, 5, 0),     # sub-rays taken one by one
    (64, 40, 61, 2, 1.25, 1, 75),   # ring bins
    (150, 60, 119, 3, 1.3, 3, 150),
]


@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("prec", [synth.PREC_FP32, synth.PREC_FP32_KAHAN])
def test_single_plane_update_adds_views_in_order(geom, prec):
    N, V, NB, M, rho, R, ring = geom
    g = pet.Geometry(N, 1, 4.0, V, NB, 4.0 * rho, M, 0.01, subrays=R, ring_mm=4.0 * ring)
    rng = np.random.default_rng(N)
    counts = torch.from_numpy(rng.poisson(4.0, (1, V, NB)).astype(np.int32)).to(DEV)
    gamma = torch.from_numpy(rng.uniform(0.5, 2.0, (1, V, NB)).astype(np.float32)).to(DEV)
    init = torch.from_numpy(rng.uniform(0.5, 2.0, (1, N, N)).astype(np.float32)).to(DEV)
    out = []
    for reg in (0, 1):
        p = synth.AlgoParams(iterations=2, beta=0.0, **dict(synth.P2_WORKLOAD, precond=synth.PRECOND_BSREM))
        p.reg = reg
        s = pet.State(g, counts, gamma, pet.make_params(p, prec), init)
        for _ in range(M + 1):
            s.subiter()
        img = torch.empty((1, N, N), device=DEV)
        s.read_image(img)
        torch.cuda.synchronize()
        out.append(img.cpu().numpy())
        s.close()
    assert not np.array_equal(out[0], init.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("N,S", [(31, 1), (67, 2), (131, 4), (401, 16), (65, 0)])
def test_projection_of_axis_views(N, S):
    # lines along an axis through pixel centres: every length is 1, so the sum is that of a float32 array
    V, nb = 2, N
    g = pet.Geometry(N, 1, 1.0, V, nb, 1.0, 1, 1.0)
    g.set_ray_chunks(S)
    if S == 0:
        S = 4                                        # the default here: at least 16 driving steps per chunk
    x = np.random.default_rng(N).uniform(0.1, 2.0, (N, N)).astype(np.float32)
    y = torch.empty((1, V, nb), device=DEV)
    pet.forward_subset(g, -1, torch.from_numpy(x[None]).to(DEV), y)
    torch.cuda.synchronize()

    def add(v, s, e):
        y = v + e
        t = s + y
        return t, y - (t - s)

    for v, steps in ((0, x), (1, x.T)):              # driven along y, along x: [step][bin]
        s = e = np.zeros(nb, np.float32)
        L = -(-N // S)
        for c in range(S):
            sc = ec = np.zeros(nb, np.float32)
            for k in range(c * L, min(N, (c + 1) * L)):
                sc, ec = add(steps[k], sc, ec)
            if c == 0:
                s, e = sc, ec
            else:
                s, e = add(sc, s, ec + e)
        np.testing.assert_array_equal(y[0, v].cpu().numpy(), s + e)
