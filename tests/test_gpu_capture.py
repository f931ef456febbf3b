"""The first library call on a stream made while that stream is being captured: the words that the
searches expect at 0 are 0 for a call outside the graph too, before any replay."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,W", [(0, 300, 136), (0, 40, 64), (3, 300, 136)])
def test_first_call_under_capture(n, H, W):
    from paper_2410_21207_gb300 import binding as sc
    rng = np.random.default_rng(H + n)
    # memory that the workspace's words may be made of holds no zeros
    junk = [torch.full((1 << k,), -1, dtype=torch.int32, device="cuda") for k in range(3, 20)]
    del junk
    torch.cuda.empty_cache()
    maps = [rng.integers(0, 65536, size=(H, W)).astype(np.uint16) for _ in range(max(n, 1))]
    dev = [torch.from_numpy(m).cuda() for m in maps]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())

    def call():
        return sc.find_seam_multi(dev) if n else sc.find_seam(dev[0])

    def same(seams, costs):
        for k, m in enumerate(maps):
            ref, cost = oracle.dp_seam(m)
            np.testing.assert_array_equal((seams[k] if n else seams).cpu().numpy(), ref)
            assert int(costs.cpu()[k]) == cost

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        captured = call()
    with torch.cuda.stream(s):
        eager = call()
        sc.check()
    same(*eager)
    for _ in range(2):
        with torch.cuda.stream(s):
            g.replay()
            sc.check()
        same(*captured)
