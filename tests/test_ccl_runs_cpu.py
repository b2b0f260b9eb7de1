"""The labelling kernels' run-based union rule (pixels start at their run's first
pixel within a 32-pixel segment; overlapping runs of two rows are joined where
the overlap begins), replayed in random order on random masks, gives the
8-connected components with their smallest index as label."""
import numpy as np
import pytest

nd = pytest.importorskip("scipy.ndimage")


def run_rule_labels(mask, rng):
    H, W = mask.shape
    f, n = mask.ravel(), mask.size
    lab = np.full(n, -1)
    for i in np.flatnonzero(f):
        lab[i] = lab[i - 1] if i % 32 and i % W and f[i - 1] else i

    def root(x):
        while lab[x] != x:
            x = lab[x]
        return x

    def unite(a, b):
        a, b = root(a), root(b)
        lab[max(a, b)] = min(a, b)

    for i in rng.permutation(np.flatnonzero(f)):
        x, y = i % W, i // W
        left = x > 0 and f[i - 1]
        if left and i % 32 == 0:
            unite(i, i - 1)
        if y == 0:
            continue
        up_left = x > 0 and f[i - W - 1]
        if f[i - W]:
            if not (left and up_left):
                unite(i, i - W)
        else:
            if up_left and not left:
                unite(i, i - W - 1)
            if x < W - 1 and f[i - W + 1] and not f[i + 1]:
                unite(i, i - W + 1)
    return np.array([root(i) if f[i] else -1 for i in range(n)])


@pytest.mark.parametrize("density", [0.1, 0.4, 0.6, 0.9, 1.0])
def test_run_rule_gives_eight_connected_labels(density):
    rng = np.random.default_rng(int(density * 100))
    for _ in range(40):
        mask = rng.random((rng.integers(1, 16), rng.integers(1, 80))) < density
        comp, k = nd.label(mask, np.ones((3, 3)))
        want = np.full(mask.size, -1)
        for c in range(1, k + 1):
            at = np.flatnonzero(comp.ravel() == c)
            want[at] = at[0]
        np.testing.assert_array_equal(run_rule_labels(mask, rng), want)
