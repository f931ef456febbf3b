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


def test_outputs_inside_the_input():
    """An output that overlaps the input gets the same result as one that does not: the energy over its own
    image, a seam over its own map (a width the search reads in place otherwise)."""
    rng = np.random.default_rng(9)
    img = rng.integers(0, 256, size=(40, 64, 3)).astype(np.uint8)
    buf = torch.zeros(40 * 64 * 3 + 16, dtype=torch.uint8, device="cuda")
    buf[:img.size].copy_(torch.from_numpy(img.reshape(-1)))
    lib, st = sc.load(), torch.cuda.current_stream().cuda_stream
    assert lib.sc_energy(buf.data_ptr(), 40, 64, 3, buf.data_ptr(), st) == 0
    sc.check()
    got = buf[:40 * 64 * 2].cpu().numpy().view(np.uint16).reshape(40, 64)
    np.testing.assert_array_equal(got, oracle.energy(img))
    for H in (100, 400):
        e = rng.integers(0, 2041, size=(H, 128)).astype(np.uint16)
        m = torch.from_numpy(e).cuda()
        assert lib.sc_find_seam(m.data_ptr(), H, 128, m.data_ptr(), None, st) == 0
        sc.check()
        got = m.cpu().numpy().reshape(-1)[:2 * H].view(np.int32)
        np.testing.assert_array_equal(got, oracle.dp_seam(e)[0])
