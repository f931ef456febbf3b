"""Narrow images of more rows than one CTA has shared memory for: a batch plan carves them on another
configuration, a cluster or the per-seam path, and a server on a cluster."""
import numpy as np
import pytest

import oracle
from paper_2410_21207_gb300 import binding as sc


def test_route_of_images_taller_than_any_configuration():
    """7,232 rows are the most a one-CTA configuration has room for; clusters of 8-row tiles 7,392."""
    cs, shape, _ = sc.batch_route([(7232, 20, 1, 18, 7232)], 0.0, 152)
    assert cs == [0]
    cs, shape, _ = sc.batch_route([(7233, 20, 1, 18, 7233), (7392, 20, 1, 18, 7392), (7393, 20, 1, 18, 7393),
                                   (8192, 20, 1, 18, 8192), (100, 20, 1, 18, 100)], 0.0, 152)
    assert cs == [1, 1, -1, -1, 0] and shape[:2] == [0, 0]
    # with both passes as well: 11 CTAs would cover the second pass's columns, but not the first one's rows
    cs, _, _ = sc.batch_route([(8192, 20, 1, 18, 8190)], 0.0, 152)
    assert cs == [-1]


# the most rows each configuration has room for, and one row more (which the next one in the list takes)
@pytest.mark.gpu
@pytest.mark.parametrize("H,cfg", [(1728, (15, 16)), (1729, (15, 8)), (2560, (15, 8)), (2561, (12, 8)), (3680, (12, 8)),
                                   (3681, (8, 16))])
def test_default_configuration_by_height(H, cfg):
    torch = pytest.importorskip("torch")
    img = np.random.default_rng(H).integers(0, 256, size=(H, 24, 3), dtype=np.uint8)
    plan = sc.BatchPlan([torch.from_numpy(img).cuda()], [(22, H)])
    info = plan.info()
    assert (info["compute_warps"], info["tile_rows"], info["batched"]) == (*cfg, 1)
    out = plan.run()[0]
    sc.check()
    np.testing.assert_array_equal(out.cpu().numpy(), oracle.carve(img, 22, H))
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("W,H", [(8, 8192), (9, 7393), (9, 7233)])
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
