"""The tiled TV steps round as the steps one by one do: a plain restatement in float32 with one rounding per
operation (FMAs through float64) is matched but for rare last bits, whose effect stays at the rounding of
the largest values."""
import numpy as np
import pytest
import torch

from paper_2111_07886_gb300 import pet

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
F = np.float32


def fma(a, b, c):
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(F)


def prox(z, w, b, steps):
    px, py, x, xb, tau = np.zeros_like(z), np.zeros_like(z), z, z, F(0.25) / F(b)
    r = tau / w
    for _ in range(steps):
        gx, gy = np.zeros_like(z), np.zeros_like(z)
        gx[..., :-1] = xb[..., 1:] - xb[..., :-1]
        gy[:, :-1] = xb[:, 1:] - xb[:, :-1]
        qx, qy = fma(F(0.5), gx, px), fma(F(0.5), gy, py)
        n2 = fma(qx, qx, qy * qy)
        s = np.where(n2 > 1, F(1) / np.sqrt(np.maximum(n2, F(1))), F(1)).astype(F)
        px, py = qx * s, qy * s
        left, up = np.zeros_like(z), np.zeros_like(z)
        left[..., 1:], up[:, 1:] = px[..., :-1], py[:, :-1]
        div = ((px - left) + py) - up
        xn = fma(r, z, fma(F(0.25), div, x)) / (F(1) + r)
        xb, x = fma(F(2), xn, -x), xn
    return x, px, py


@pytest.mark.parametrize("N,P", [(40, 1), (35, 9)])
@pytest.mark.parametrize("steps", [2, 10])
def test_steps_round_as_the_operators(N, P, steps):
    g = pet.Geometry(N, P, 2.0, 8, int(1.5 * N) | 1, 2.0, 2, 0.9)
    rng = np.random.default_rng(N)
    z, w = rng.uniform(-0.5, 6.0, (P, N, N)).astype(F), rng.uniform(0.05, 2.0, (P, N, N)).astype(F)
    px, py = torch.zeros((P, N, N), device=DEV), torch.zeros((P, N, N), device=DEV)
    x = torch.empty((P, N, N), device=DEV)
    pet.tv_prox(g, torch.from_numpy(z).to(DEV), torch.from_numpy(w).to(DEV), 0.3, steps, px, py, x)
    torch.cuda.synchronize()
    for got, ref in zip((x, px, py), prox(z, w, 0.3, steps)):
        got = got.cpu().numpy()
        # one value in a hundred may differ per step, by the rounding of a value of its size and its neighbours'
        assert np.mean(got != ref) <= 0.01 * steps
        assert np.abs(got - ref).max() <= steps * 2.0 ** -23 * np.abs(ref).max()
