"""TV scans whose volume leaves no memory for the tiled proximal step's second set of fields run its steps one
by one, with the same bits (the allocation's failure is injected on the host: pet_debug_fail_alloc)."""
import numpy as np
import pytest
import torch

from paper_2111_07886_gb300 import pet, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def fails_next():
    """Whether an injected failure is still waiting for an allocation."""
    try:
        pet.Geometry(8, 1, 1.0, 4, 13, 1.0, 2, 1.0)
    except pet.PetError:
        return True
    return False


# tiles of 16 and of 32 cut by the image, planes that fill and cut a group
@pytest.mark.parametrize("N,P", [(33, 1), (70, 1), (19, 3), (130, 41)])
@pytest.mark.parametrize("iters", [2, 7, 23])
def test_prox_without_memory_for_tiles(N, P, iters):
    rng = np.random.default_rng(N)
    z, w = (torch.from_numpy(rng.uniform(lo, hi, (P, N, N)).astype(np.float32)).to(DEV) for lo, hi in ((-0.5, 3.0), (0.05, 2.0)))
    out = []
    for fail in (0, 1):
        g = pet.Geometry(N, P, 2.0, 8, int(1.5 * N) | 1, 2.0, 2, 0.9)
        px, py, x = torch.zeros_like(z), torch.zeros_like(z), torch.empty_like(z)
        pet.debug_fail_alloc(fail)
        try:
            pet.tv_prox(g, z, w, 0.3, iters, px, py, x)
        finally:
            torch.cuda.synchronize()
            pet.debug_fail_alloc(0)
        out.append([t.cpu().numpy() for t in (x, px, py)])
        g.close()
    assert np.abs(out[0][1]).max() > 0.5
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("P", [1, 11])
def test_state_without_memory_for_tiles(P):
    N, V, M = 37, 20, 4
    g = pet.Geometry(N, P, 2.0, V, 55, 2.0, M, 0.9)
    rng = np.random.default_rng(P)
    counts = torch.from_numpy(rng.poisson(20.0, (P, V, 55)).astype(np.int32)).to(DEV)
    gamma = torch.full((P, V, 55), 1.0, device=DEV)
    p = synth.AlgoParams(iterations=2, beta=0.5, **synth.P2_WORKLOAD)
    p.reg = 1

    def run(fail):
        pet.debug_fail_alloc(fail)
        try:
            s = pet.State(g, counts, gamma, pet.make_params(p), torch.ones((P, N, N), device=DEV))
        except pet.PetError as e:
            assert e.status == pet.ERR_OOM
            return None
        for _ in range(M + 1):
            s.subiter()
        img = torch.empty((P, N, N), device=DEV)
        s.read_image(img)
        torch.cuda.synchronize()
        s.close()
        return img.cpu().numpy()

    want = run(0)
    n = 1
    while (got := run(n)) is None:              # the allocations the state cannot do without
        n += 1
    waiting = fails_next()
    pet.debug_fail_alloc(0)
    assert not waiting                          # one more was asked for, failed and was done without
    np.testing.assert_array_equal(got, want)
