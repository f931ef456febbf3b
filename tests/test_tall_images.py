"""Narrow images of more rows than one CTA has shared memory for: a batch plan carves them on another
configuration, a cluster or the per-seam path, and a server on a cluster."""
import numpy as np
import pytest

import oracle
from paper_2410_21207_gb300 import binding as sc


def test_route_of_images_taller_than_any_configuration():
    """7,168 rows are the most a one-CTA configuration has room for; clusters of 8-row tiles 7,392."""
    cs, shape, _ = sc.batch_route([(7168, 20, 1, 18, 7168)], 0.0, 152)
    assert cs == [0]
    cs, shape, _ = sc.batch_route([(7169, 20, 1, 18, 7169), (7392, 20, 1, 18, 7392), (7393, 20, 1, 18, 7393),
                                   (8192, 20, 1, 18, 8192), (100, 20, 1, 18, 100)], 0.0, 152)
    assert cs == [1, 1, -1, -1, 0] and shape[:2] == [0, 0]
    # with both passes as well: 11 CTAs would cover the second pass's columns, but not the first one's rows
    cs, _, _ = sc.batch_route([(8192, 20, 1, 18, 8190)], 0.0, 152)
    assert cs == [-1]


@pytest.mark.gpu
@pytest.mark.parametrize("W,H", [(8, 8192), (9, 7393), (9, 7169)])
def test_tall_images_in_a_batch(W, H):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(H)
    imgs = [rng.integers(0, 256, size=s, dtype=np.uint8) for s in ((H, W, 3), (40, 60, 3))]
    targets = [(W - 2, H), (50, 40)]
    outs = sc.carve_batch([torch.from_numpy(i).cuda() for i in imgs], targets)
    sc.check()
    for i, (tw, th), o in zip(imgs, targets, outs):
        np.testing.assert_array_equal(o.cpu().numpy(), oracle.carve(i, tw, th))


# the one-CTA kernel of the server has room for 1,664 to 1,728 rows; a request that no kernel took stayed at
# the queue's front for good
@pytest.mark.gpu
def test_served_at_every_height():
    pytest.importorskip("torch")
    rng = np.random.default_rng(4)
    srv = sc.Server(budget_bytes=256 << 20, max_batch=8, streams=2)
    jobs = []
    for H in (1664, 1665, 1696, 1697, 1728, 1729, 4096, 300):
        for W in (24, 1000) if H < 1800 else (24,):
            im = rng.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
            jobs.append((im, srv.submit(im, W - 3, H)))
    srv.drain(60)
    for im, t in jobs:
        np.testing.assert_array_equal(srv.result(t), oracle.carve(im, im.shape[1] - 3, im.shape[0]))
    assert srv.stats()["device_errors"] == 0
    srv.close()
