"""The launch forms of the fixed-point LAPs: batches that the resident warps hold
at once (no queue) against batches that run half by fixed stride and half from
the queue, with two tile buffers per warp or one, at the edges of the lane
groups (8, 16, 32) and of the one-tile form.  Every LAP is independent of which
warp solves it, so the results are equal bit for bit; a sample is held to the
oracle: optimum and duals within the tile grid's rounding, 2^-47 of the tile's
magnitude per entry on at most 2 m entries."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _solve(R, torch, cost, u0):
    b, m = cost.shape[:2]
    out = dict(value=torch.empty(b, device="cuda", dtype=torch.float64), n_aug=torch.empty(b, device="cuda", dtype=torch.int32),
               u=torch.empty(b, m, device="cuda", dtype=torch.float64),
               v=torch.empty(b, m, device="cuda", dtype=torch.float64),
               row_to_col=torch.empty(b, m, device="cuda", dtype=torch.int32))
    R.rlt2_lap_batched(cost, u0=u0, dual_mode=1, **out)
    return out


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("m", [1, 7, 8, 9, 16, 17, 19, 20, 23, 24, 27, 30, 31, 32])
def test_large_batches_equal_small_ones(m, warm):
    torch = pytest.importorskip("torch")
    from paper_1710_03732_gb300 import rlt2 as R
    batch = 45001 if m <= 8 else 25001 if m <= 16 else 12001
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    cost = 100 * torch.randn(batch, m, m, generator=g, device="cuda", dtype=torch.float64)
    cost[::3] = torch.round(cost[::3] / 20)  # ties
    cost[5::97] = 0.0
    cost[6::89] *= -0.0
    u0 = 50 * torch.randn(batch, m, generator=g, device="cuda", dtype=torch.float64) if warm else None
    big = _solve(R, torch, cost, u0)
    for a in range(0, batch, 1000):
        small = _solve(R, torch, cost[a:a + 1000].contiguous(), u0[a:a + 1000].contiguous() if warm else None)
        for k, x in small.items():
            assert torch.equal(x, big[k][a:a + 1000]), k
    for i in list(range(0, batch, batch // 40)) + [batch - 1]:
        c = cost[i].cpu().numpy()
        ref = O.lap(c, canonical=True)
        tol = 2 * m * 2.0**-47 * max(np.abs(c).max(), 1e-300)
        assert abs(big["value"][i].item() - ref.value) <= tol
        assert np.abs(big["u"][i].cpu().numpy() - ref.u).max() <= tol
        assert np.abs(big["v"][i].cpu().numpy() - ref.v).max() <= tol
