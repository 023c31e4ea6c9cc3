"""Product orders whose coordinates are clustered, equal or in any order of labels: both ways of
ranking them (one CTA up to 8192 elements, tiles of 4096 beyond) against the oracle, every N_k, and the time
that they take against that of spread-out coordinates."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as m
    return m


def _coords(shape, n):
    rng = np.random.default_rng(n)
    if shape == "equal":
        c = np.full((2, n), 77)
    elif shape == "outlier":
        c = rng.integers(0, 5000, (2, n))
        c[:, n // 2] = 2 ** 31 - 1
    elif shape == "one_v":
        c = np.stack([rng.integers(0, 2 ** 31, n), np.full(n, 123456)])
    elif shape == "duplicates":  # in u, in v and in both, far apart in the labels
        c = rng.integers(0, 2 ** 31, (2, n))
        c[0, : n // 3] = c[0, 2 * n // 3: 2 * n // 3 + n // 3]
        c[1, n // 4: n // 2] = c[1, n // 2: n // 2 + n // 2 - n // 4]
        c[:, : n // 8] = c[:, n - n // 8:]
    else:
        c = rng.integers(0, 2 ** 31, (2, n))
    return np.ascontiguousarray(c[:, np.argsort(c.sum(0), kind="stable")], dtype=np.int32)


def _call(cs, kind, coords):
    """A function that counts, and its histogram."""
    import torch
    n = coords.shape[1]
    c = torch.from_numpy(coords).cuda()
    hist = torch.full((cs.hist_len(n),), -5, dtype=torch.int64, device="cuda")
    ws = torch.full((cs.coords_abundance_workspace(kind, n),), 255, dtype=torch.uint8, device="cuda")
    return (lambda: cs.coords_abundance(kind, n, c, hist, ws)), hist


@pytest.mark.parametrize("kind", [1, 5])
@pytest.mark.parametrize("n", [1025, 8191, 8192, 8193, 12288, 12289])
@pytest.mark.parametrize("shape", ["equal", "outlier", "one_v", "duplicates"])
def test_histogram(cs, oracle, kind, n, shape):
    c = _coords(shape, n)
    want = oracle.interval_abundance(oracle.causal_matrix(kind, c))
    assert want.sum() > 0 or shape in ("equal", "one_v")
    f, hist = _call(cs, kind, c)
    f()
    assert (hist.cpu().numpy() == want).all()
    # any order of the labels
    f, hist = _call(cs, kind, np.ascontiguousarray(c[:, np.random.default_rng(1).permutation(n)]))
    f()
    assert (hist.cpu().numpy() == want).all()


@pytest.mark.parametrize("shape", ["equal", "outlier", "one_v"])
@pytest.mark.parametrize("n", [3000, 8192])
def test_time_does_not_depend_on_the_distribution(cs, shape, n):
    """The ranks of clustered coordinates, sorted, take some times those of spread-out ones, not n times."""
    import torch

    def best(f):
        f()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(3):
                f()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    spread, _ = _call(cs, 1, _coords("uniform", n))
    clustered, _ = _call(cs, 1, _coords(shape, n))
    assert best(clustered) < 5.0 * best(spread)
