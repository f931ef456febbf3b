"""The energy straight from HWC bytes equals the oracle's for every channel count, byte alignment of the
image, width modulo the kernel's 4 columns, and at its 4-row groups' edges."""
import numpy as np
import pytest

import oracle
from paper_2410_21207_gb300 import binding as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 3, 4])
@pytest.mark.parametrize("H,W", [(1, 1), (1, 6), (4, 4), (5, 7), (8, 130), (9, 257), (3, 2051), (64, 512)])
def test_energy_of_any_alignment(C, H, W):
    rng = np.random.default_rng(C * 1000003 + H * 1009 + W)
    for offset in range(4):
        img = rng.integers(0, 256, size=(H, W, C)).astype(np.uint8)
        buf = torch.zeros(H * W * C + 8, dtype=torch.uint8, device="cuda")
        view = buf[offset:offset + H * W * C].view(H, W, C)
        view.copy_(torch.from_numpy(img))
        got = sc.energy(view).cpu().numpy()
        np.testing.assert_array_equal(got, oracle.energy(img), err_msg=f"offset {offset}")
