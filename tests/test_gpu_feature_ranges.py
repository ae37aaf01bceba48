"""Features of tiles whose scale leaves FP32's comfortable range: differences so
large that the scale overflows (its inverse is 0) or so small that the inverse does
(zero differences then scale to NaN), beside ordinary ones.  The values follow from
the definition: FP32 truncation, column minima, one product per entry, a bitonic
sort of 32 lanes by IEEE minNum and maxNum (a NaN loses to a number), BF16."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _bf(x):
    """BF16 rounding, to nearest even."""
    b = np.asarray(x, dtype=np.float32).view(np.uint32).astype(np.uint64)
    r = (((b + 0x7FFF + ((b >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32)
    return np.where(np.isnan(x), np.float32(np.nan), r)


def _sort(rows):
    """Rows of 32 lanes through the network."""
    v, lane = rows.copy(), np.arange(32)
    k = 2
    while k <= 32:
        j = k >> 1
        while j:
            o = v[:, lane ^ j]
            v = np.where(((lane & j) == 0) == ((lane & k) == 0), np.fmin(v, o), np.fmax(v, o))
            j >>= 1
        k <<= 1
    return v


def _features(tile, prev):
    m = len(prev)
    f = np.array([O.f32_trunc(x) for x in tile.reshape(-1)], dtype=np.float32).reshape(m, m)
    p = np.array([O.f32_trunc(x) for x in prev], dtype=np.float32)
    red = f - f.min(0)
    s = red.max()
    inv = np.float32(1) / (s if s > 0 else np.float32(1))
    rows = np.full((m, 32), np.inf, dtype=np.float32)
    rows[:, :m] = red * inv
    out = np.zeros((m, 34), dtype=np.float32)
    out[:, :m] = _sort(rows)[:, :m]
    out[:, 32] = p * inv
    out[:, 33] = np.float32(m) / np.float32(32)
    return _bf(out)


@pytest.mark.parametrize("kind", ["plain", "tiny", "huge", "mixed"])
@pytest.mark.parametrize("m", [2, 3, 8, 9, 16, 17, 18, 31, 32])
def test_features_over_the_range(m, kind):
    torch = pytest.importorskip("torch")
    from paper_1710_03732_gb300 import rlt2 as R
    rng = np.random.default_rng([m, len(kind)])
    nt = 24
    tiles = rng.normal(0, 100, (nt, m, m))
    tiny = 2.0**-126 * (1 + rng.integers(0, 40, (nt, m, m)) * 2.0**-23)
    huge = rng.uniform(-1, 1, (nt, m, m)) * 3.3e38
    if kind == "tiny":
        tiles = tiny
    elif kind == "huge":
        tiles = huge
    elif kind == "mixed":
        tiles[0::4], tiles[1::4] = tiny[0::4], huge[1::4]
        tiles[2::4] = 0.0
    prev = rng.normal(0, 3, (nt, m))
    net = R.Mlp(64, seed=1)
    net.add_samples(torch.from_numpy(tiles).cuda(), torch.from_numpy(np.zeros((nt, m))).cuda(), torch.from_numpy(prev).cuda())
    X, _ = net.samples()
    net.close()
    with np.errstate(all="ignore"):
        ref = np.concatenate([_features(c, p) for c, p in zip(tiles, prev)])
    assert np.array_equal(X, ref, equal_nan=True)
