"""GPU parity of the tree's top-k selection where its lower bound is tight or useless: plateaus, rows of few distinct values, masked
vocabularies, infinities, segments that end early, more children than warps."""
import numpy as np
import pytest

from test_gpu_tree_build import _both, _probs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [3, 511, 513, 4100, 9000])
@pytest.mark.parametrize("branching,T", [((1, 1), 3), ((3, 2, 1), 12), ((8, 1), 10), ((9, 2), 20)])
@pytest.mark.parametrize("kind", ["plateau", "two", "masked", "spikes", "inf", "negative"])
def test_selection_bounds(V, branching, T, kind):
    branching = tuple(min(b, V) for b in branching)
    rng = np.random.default_rng(V + T)
    q = _probs(rng, 2, T, V)
    if kind == "plateau":
        q[:] = 0.25
    elif kind == "two":
        q[:] = rng.integers(0, 2, q.shape)
    elif kind == "masked":
        q[rng.random(q.shape) < 0.98] = -np.inf
        q[:, :, 0] = 0.5  # (some entry in every row)
    elif kind == "spikes":
        q[:] = 0.0
        q[:, :, rng.integers(0, V, 2)] = 1.0
    elif kind == "inf":
        q[:, :, :: max(1, V // 7)] = np.inf
    else:
        q = -q - np.float32(3.0e38)
    _both(q, branching, rng.integers(0, V, 2).astype(np.int32), np.array([7, 90], dtype=np.int32))
