"""The update of FP32 stacks with the 3-D prior, detection factors or time of flight rounds an image value
once per subiteration: f - c (scale b + (beta/M) grad R) with one rounding at f's own ulp.

From the same FP32 image a subiteration with a small step leaves the rounding of the result as the only
error that counts: steps of 1e-5 to 1e-3 of f are thousands of ulps, and their own relative error of about
1e-6 is below 1e-2 ulp.  Against the FP64 state the error is then uniform in half an ulp either way,
1 / sqrt(12) = 0.289 ulp rms (two roundings: 0.408)."""
import numpy as np
import pytest
import torch

from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _params(**kw):
    return synth.AlgoParams(iterations=2, **dict(dict(synth.P2_WORKLOAD, precond=synth.PRECOND_BSREM), **kw))


def _inputs(N, P, V, nb, T, seed, attn):
    rng = np.random.default_rng(seed)
    shape = (P, V, nb) + ((T,) if T > 1 else ())
    counts = torch.from_numpy(rng.poisson(4.0, shape).astype(np.int32)).to(DEV)
    gamma = torch.from_numpy(rng.uniform(0.5, 2.0, shape).astype(np.float32)).to(DEV)
    mult = torch.from_numpy(rng.uniform(0.3, 1.0, shape).astype(np.float32)).to(DEV) if attn else None
    init = torch.from_numpy(rng.uniform(0.5, 2.0, (P, N, N)).astype(np.float32)).to(DEV)
    return counts, gamma, mult, init


def _image(g, counts, gamma, mult, init, p, prec, steps, dtype=torch.float32):
    s = pet.State(g, counts, gamma, pet.make_params(p, prec), init, d_mult=mult)
    for _ in range(steps):
        s.subiter()
    img = torch.empty(init.shape, dtype=dtype, device=DEV)
    s.read_image(img)
    torch.cuda.synchronize()
    s.close()
    return img.cpu().numpy()


# planes that fill and cut a group of eight, two to four candidate bins
@pytest.mark.parametrize("rdp3d,attn,T", [(1, False, 0), (0, True, 0), (1, True, 0), (0, False, 9), (0, True, 9)])
@pytest.mark.parametrize("N,P,rho", [(41, 9, 1.0), (30, 17, 0.6), (24, 32, 1.0)])
@pytest.mark.parametrize("prec", [synth.PREC_FP32, synth.PREC_FP32_KAHAN])
def test_one_rounding_per_subiteration(rdp3d, attn, T, N, P, rho, prec):
    V, M, nb = 20, 2, int(1.45 * N / rho) | 1
    tof = dict(tof_bins=T, tof_bin_mm=8.0, tof_fwhm_mm=12.0) if T else {}
    g = pet.Geometry(N, P, 1.0, V, nb, rho, M, 0.01, **tof)
    data = _inputs(N, P, V, nb, T, N + P, attn)
    p = _params(beta=0.2, lambda0=1e-4, rdp3d=rdp3d)
    ref = _image(g, *data, p, synth.PREC_FP64, 1, torch.float64)
    got = _image(g, *data, p, prec, 1)
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    moved = np.abs(ref - data[3].cpu().numpy()) / ulp
    assert np.mean(moved > 50) > 0.9
    assert np.sqrt(np.mean(((got - ref) / ulp) ** 2)) <= 0.31


# A TOF stack's planes against the same data as single planes, which run the general kernels: the same
# operations in FP32.  With compensated sums a ray's rounding may fall to the other side where its sum
# lies next to a border: one of 2^-24 in about a tenth of the rays, 1e-8 of b in all, and steps of at most
# 0.1 f turn that into 2 % of the image values.
@pytest.mark.parametrize("N,P,T", [(33, 17, 9), (40, 41, 13), (24, 48, 21)])
def test_tof_planes_as_single_planes(N, P, T):
    V, M, nb = 18, 2, int(1.45 * N) | 1
    tof = dict(tof_bins=T, tof_bin_mm=8.0, tof_fwhm_mm=12.0)
    one, all_ = (pet.Geometry(N, k, 1.0, V, nb, 1.0, M, 0.01, **tof) for k in (1, P))
    counts, gamma, mult, init = _inputs(N, P, V, nb, T, N + P, True)
    p = _params(beta=0.0, lambda0=0.1)
    for prec, most in ((synth.PREC_FP32, 0.0), (synth.PREC_FP32_KAHAN, 0.05)):
        stack = _image(all_, counts, gamma, mult, init, p, prec, 1)
        for z in (0, P // 2, P - 1):
            plane = _image(one, *(t[z:z + 1].contiguous() for t in (counts, gamma, mult, init)), p, prec, 1)
            assert np.mean(stack[z] != plane[0]) <= most, (prec, z)
