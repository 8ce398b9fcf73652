"""GPU parity of the tree's top-k selection where its lower bound is tight or useless: plateaus, rows of few distinct values, masked
vocabularies, infinities, negative values, NaN (which never ranks), segments that end early, more children than warps, and as many
entries above the bound as the list holds."""
import numpy as np
import pytest

from test_gpu_tree_build import _both, _probs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [3, 511, 513, 4100, 9000])
@pytest.mark.parametrize("branching,T", [((1, 1), 3), ((3, 2, 1), 12), ((8, 1), 10), ((9, 2), 20)])
@pytest.mark.parametrize("kind", ["plateau", "two", "masked", "spikes", "inf", "negative", "nan"])
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
    elif kind == "negative":
        q = -1 - rng.random(q.shape, dtype=np.float32)
    shown = q.copy()
    if kind == "nan":  # the oracle sees them as -inf: there are other entries enough
        shown[:, :, 5::7] = np.nan
        q[:, :, 5::7] = -np.inf
    _both(shown, branching, rng.integers(0, V, 2).astype(np.int32), np.array([7, 90], dtype=np.int32), ranked=q)


@pytest.mark.parametrize("V", [4096, 4097, 8192])
@pytest.mark.parametrize("reach", [127, 128, 129])
def test_as_many_entries_reach_the_bound_as_the_list_holds(V, reach):
    # two children: the second greatest of the warps' maxima is the bound.  Tokens 1024 j + 0 .. 31 of a segment are one warp's, with
    # four loads per thread (V a multiple of 4) or sixteen; token 200 is another's and holds the bound itself.
    rng = np.random.default_rng(reach)
    q = (rng.random((2, 3, V)) * 0.1).astype(np.float32)
    first = (np.arange(4)[:, None] * 1024 + np.arange(32)).reshape(-1)
    for row in q.reshape(-1, V):
        at = rng.permutation(first)[: reach - 1]
        row[at] = 0.6 + 0.3 * rng.permutation(reach - 1).astype(np.float32) / reach
        row[200] = 0.5
    assert (q[:, :, :4096] >= 0.5).sum(-1).tolist() == [[reach] * 3] * 2
    _both(q, (2,), np.array([1, 2], dtype=np.int32), None)
