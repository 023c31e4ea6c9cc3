"""The smeared sums at the edges of their terms: fewer abundances than the
polynomial's degree, one and several terms per thread, powers with bits below
and above the lanes', cutoffs from tens of terms to the whole histogram.
Against the binary128 oracle at the actions' bound, 1e-12 of max(1, |S|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = (1e-6, 1e-4, 0.003, 0.0625, 0.3, 0.75, 0.999)


@pytest.mark.parametrize("dim", [2, 3, 4])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 33, 34, 36, 1500, 4100, 70001])
def test_smeared_actions(oracle, dim, n):
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    rng = np.random.default_rng(n)
    # at most the abundances of a chain, some of them none
    h = (n - 1 - np.arange(n - 1)) * (rng.random(n - 1) < 0.8)
    hist = torch.from_numpy(h.astype(np.int64)).cuda()
    out = torch.zeros(16, dtype=torch.float64, device="cuda")
    br = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = torch.empty(cs.action_workspace_bytes(), dtype=torch.uint8, device="cuda")
    eps = EPS + (0.0, 1.0)
    for _ in range(2):  # back to back: the second call must not overtake the first
        cs.action_device(dim, n, hist, list(eps), out, br, ws)
    got = out.cpu().numpy()
    for e, ep in enumerate(eps):
        want, bracket = oracle.action(dim, n, h.astype(np.int64), ep)
        assert int(br[0]) == bracket
        assert abs(got[e] - want) <= 1e-12 * max(1.0, abs(want)), (ep, got[e], want)


def test_captured_action(oracle):
    """The dependent launch inside a CUDA graph, between other kernels, replayed back to back."""
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    buf = cs.allocate(0, 700)
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        cs.run(buf, 5, eps=EPS, stream=st)
        st.synchronize()
        with torch.cuda.graph(g, stream=st):
            cs.run(buf, 4, eps=EPS, stream=st)
            cs.run(buf, 5, eps=EPS, stream=st)
    buf.actions.zero_()
    for _ in range(5):
        g.replay()
    torch.cuda.synchronize()
    h = oracle.interval_abundance(oracle.causal_matrix(0, oracle.sprinkle(0, 700, 5)))
    assert (buf.hist.cpu().numpy() == h).all()
    for e, ep in enumerate(EPS):
        want, bracket = oracle.action(2, 700, h, ep)
        assert int(buf.bracket[0]) == bracket
        assert abs(float(buf.actions[e]) - want) <= 1e-12 * max(1.0, abs(want)), ep
