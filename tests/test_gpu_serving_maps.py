"""Requests whose launches reuse one place in the server's memory: every image's energies must be read
through its own tensor map, not through an earlier one that lay at the same address."""
import numpy as np
import pytest

import oracle
from paper_2410_21207_gb300 import binding as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tables_reuse_their_addresses():
    """A small arena and one request or a few at a time: the descriptor tables of successive launches, of
    both kernels and of different sizes, fall on the same addresses."""
    if not torch.cuda.is_available():
        pytest.fail("the -m gpu tests need a CUDA GPU")
    rng = np.random.default_rng(11)
    srv = sc.Server(budget_bytes=64 << 20, max_batch=4, streams=2)
    for k in range(24):
        sizes = [(int(rng.integers(1500, 1700)), int(rng.integers(20, 60)))] if k % 4 == 3 else \
            [(int(rng.integers(16, 300)), int(rng.integers(8, 200))) for _ in range(1 + k % 3)]
        imgs = [rng.integers(0, 256, size=(H, W, 3), dtype=np.uint8) for W, H in sizes]
        tickets = [srv.submit(im, im.shape[1] - 4, im.shape[0]) for im in imgs]
        srv.drain(60)
        for im, t in zip(imgs, tickets):
            np.testing.assert_array_equal(srv.result(t), oracle.carve(im, im.shape[1] - 4, im.shape[0]))
            srv.release(t)
    assert srv.stats()["device_errors"] == 0
    srv.close()
