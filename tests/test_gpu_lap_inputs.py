"""Inputs that choose between forms of the batched LAP launches: tiles on 8-byte
and on 16-byte boundaries, all-zero tiles beside others in one warp of a batch of
nodes, and calls between a producer and a consumer on the caller's stream, also
captured into a graph behind work of another stream."""
import numpy as np
import pytest

import oracle as O
from paper_1710_03732_gb300 import instances as I

pytestmark = pytest.mark.gpu


def _outputs(torch, b, m):
    return dict(value=torch.empty(b, device="cuda", dtype=torch.float64), u=torch.empty(b, m, device="cuda", dtype=torch.float64),
                v=torch.empty(b, m, device="cuda", dtype=torch.float64),
                row_to_col=torch.empty(b, m, device="cuda", dtype=torch.int32),
                n_aug=torch.empty(b, device="cuda", dtype=torch.int32))


@pytest.mark.parametrize("batch", [300, 30001])  # held at once, and through the queue
@pytest.mark.parametrize("m", [2, 4, 8, 10, 16, 18, 20])
def test_tiles_on_eight_byte_boundaries(m, batch):
    torch = pytest.importorskip("torch")
    from paper_1710_03732_gb300 import rlt2 as R
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    flat = 100 * torch.randn(batch * m * m + 1, generator=g, device="cuda", dtype=torch.float64)
    u0 = 30 * torch.randn(batch, m, generator=g, device="cuda", dtype=torch.float64)
    shifted = flat[1:].view(batch, m, m)
    aligned = shifted.clone()
    assert shifted.data_ptr() % 16 == 8 and aligned.data_ptr() % 16 == 0
    for start in (None, u0):
        a, b = _outputs(torch, batch, m), _outputs(torch, batch, m)
        R.rlt2_lap_batched(aligned, u0=start, dual_mode=1, **a)
        R.rlt2_lap_batched(shifted, u0=start, dual_mode=1, **b)
        for k in a:
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("warm", [0, 1])
@pytest.mark.parametrize("n", [6, 9, 10, 14, 18, 20])
def test_zero_tiles_beside_others_in_batched_nodes(n, warm, mode):
    """One solve of nodes whose tiles are zero at random places, so that the LAPs of
    one warp (four, two or one, n - 2 up to 8, 16, 32) differ in kind: as the oracle's
    duals for sampled tiles, zero for the zero ones, and as rlt2_iterate's."""
    from paper_1710_03732_gb300 import rlt2 as R
    m, T = n - 2, O.num_tiles(n)
    inst = I.random_instance(n, 17, with_b=True)
    rng = np.random.default_rng([n, warm])
    D = rng.normal(0, 100, (T, m, m))
    zero = rng.random(T) < 0.4
    zero[:4] = True
    D[zero] = 0.0
    D[5 % T, 0, 0] = 5e-324 if zero[5 % T] else D[5 % T, 0, 0]  # nearly zero
    zero[5 % T] = False
    prm = R.params(dual_mode=mode, warm=warm, feas_tol=0.0)
    many, single = ([R.Context(inst.F, inst.D, inst.B, prm=prm) for _ in range(2)] for _ in range(2))
    for group in (many, single):
        for c in group:
            c.import_state(D.reshape(-1), c.export_state()[1])
    assert (R.rlt2_iterate_many(many, 1) == 1).all()
    for a, b in zip(many, single):
        b.iterate(1)
        da, db = a.duals(), b.duals()
        for k in da:
            assert np.array_equal(da[k], db[k]), k
        xi, psi = da["xi"].reshape(T, m), da["psi"].reshape(T, m)
        assert not xi[zero].any() and not psi[zero].any()
        for t in rng.permutation(np.flatnonzero(~zero))[:12]:
            ref = O.lap(D[t], canonical=True)
            # rounding of the tile's grid, 2^-47 of its magnitude on at most 2 m entries
            tol = 2 * m * 2.0**-47 * max(np.abs(D[t]).max(), 1e-300)
            assert np.abs(xi[t] - ref.u).max() <= tol and np.abs(psi[t] - ref.v).max() <= tol
    for c in many + single:
        c.close()


@pytest.mark.parametrize("batch,m", [(400, 7), (300, 18), (40000, 12)])
def test_between_kernels_of_the_callers_stream(batch, m):
    torch = pytest.importorskip("torch")
    from paper_1710_03732_gb300 import rlt2 as R
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    base = 50 * torch.randn(batch, m, m, generator=g, device="cuda", dtype=torch.float64)
    scales = [1.0, -2.0, 0.5, 3.0]
    want = []
    for f in scales:
        o = _outputs(torch, batch, m)
        R.rlt2_lap_batched(base * f, dual_mode=1, **o)
        torch.cuda.synchronize()
        want.append(o["value"] + o["u"].sum(1))
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    cost, o = torch.empty_like(base), _outputs(torch, batch, m)
    got = [torch.empty(batch, device="cuda", dtype=torch.float64) for _ in scales]
    torch.cuda.synchronize()

    def chain():  # each step overwrites the costs that the step before reads
        for f, out in zip(scales, got):
            torch.mul(base, f, out=cost)
            R.rlt2_lap_batched(cost, dual_mode=1, **o)
            torch.add(o["value"], o["u"].sum(1), out=out)

    with torch.cuda.stream(s):
        for _ in range(5):
            chain()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    # captured: the first call's costs come from another stream
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        other.wait_stream(s)
        with torch.cuda.stream(other):
            torch.mul(base, scales[0], out=cost)
        o["value"].zero_()
        s.wait_stream(other)
        R.rlt2_lap_batched(cost, dual_mode=1, **o)
        torch.add(o["value"], o["u"].sum(1), out=got[0])
        chain()
    for x in got:
        x.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
