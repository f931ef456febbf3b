"""The two-ended seam search: the upper half of a map swept downwards, the lower half upwards, joined
in the middle. The identity it rests on is checked in numpy on the CPU, the kernel on the GPU, both
against the oracle's Algorithm 3, at the sizes where the halves, tiles and super-tiles have edges."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")


def _maps(H, W):
    rng = np.random.default_rng(H * 8191 + W)
    yield "uniform", rng.integers(0, 2041, size=(H, W))
    yield "ties", rng.integers(0, 2, size=(H, W))
    yield "constant", np.full((H, W), 3)


def _sweep(e):
    """Costs and leftmost directions of every cell from row 0 downwards."""
    H, W = e.shape
    m = np.full((H, W + 2), 1 << 40, dtype=np.int64)
    d = np.zeros((H, W), dtype=np.int64)
    m[0, 1:-1] = e[0]
    for i in range(1, H):
        three = np.stack([m[i - 1, :-2], m[i - 1, 1:-1], m[i - 1, 2:]])
        d[i] = np.argmin(three, axis=0) - 1
        m[i, 1:-1] = e[i] + three.min(axis=0)
    return m, d


@pytest.mark.parametrize("H,W", [(2, 1), (2, 7), (3, 2), (9, 5), (16, 31), (41, 12)])
def test_seam_from_both_ends_is_algorithm_3s(H, W):
    for kind, e in _maps(H, W):
        e = e.astype(np.uint16)
        h0 = (H + 1) // 2
        m0, d0 = _sweep(e[:h0])
        m1, d1 = _sweep(e[h0:][::-1])
        up, dn = m0[-1, 1:-1], m1[-1]
        three = np.stack([dn[:-2], dn[1:-1], dn[2:]])
        j = int(np.argmin(up + three.min(axis=0)))
        seam = np.empty(H, dtype=np.int32)
        c = j
        for i in range(h0 - 1, -1, -1):
            seam[i] = c
            c += int(d0[i, c]) if i else 0
        c = j + int(np.argmin(three[:, j])) - 1
        for r in range(H - h0 - 1, -1, -1):
            seam[H - 1 - r] = c
            c += int(d1[r, c]) if r else 0
        ref, cost = oracle.dp_seam(e)
        assert int(up[j] + three[:, j].min()) == cost, kind
        np.testing.assert_array_equal(seam, ref, err_msg=kind)


# 192 rows are the fewest swept from both ends; 128 columns a CTA (up to 2048), 384 (up to 6144), 640;
# 32-row tiles and super-tiles in each half; 2300 x 8192: the ancestor tables do not fit shared memory
@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [(191, 129), (192, 1), (192, 128), (193, 129), (194, 2), (255, 300), (256, 2048),
                                 (257, 2049), (319, 130), (321, 6144), (383, 6145), (1079, 1919), (2300, 8192)])
def test_two_ended_search_parity(H, W):
    from paper_2410_21207_gb300 import binding as sc
    for kind, e in _maps(H, W):
        e = e.astype(np.uint16)
        ref, cost = oracle.dp_seam(e)
        for _ in range(2):   # the arrival counter is back at zero
            seam, c = sc.find_seam(torch.from_numpy(e).cuda())
            sc.check()
            assert int(c.cpu()[0]) == cost, kind
            np.testing.assert_array_equal(seam.cpu().numpy(), ref, err_msg=f"{H}x{W} {kind}")


# maps read in place (rows of a multiple of 8 columns from a 16-byte boundary) and the same maps 2 bytes off
# it (copied first), at both sides of the 24-bit range: H * max(e) = 2^24 - H (fast) and 2^24 (wide-cost);
# 128 rows: one cluster, 512: both ends; then an ordinary map on the same workspace
@pytest.mark.gpu
@pytest.mark.parametrize("H,W,emax", [(512, 64, 32767), (512, 64, 32768), (512, 2056, 32768), (128, 264, 65535),
                                      (256, 8, 65535), (264, 136, 65535)])
def test_maps_in_place_at_the_range_limit(H, W, emax):
    from paper_2410_21207_gb300 import binding as sc
    rng = np.random.default_rng(H + W + emax)
    near = rng.integers(emax - 3, emax, size=(H, W), endpoint=True).astype(np.uint16)
    near[H // 2, W // 2] = emax
    plain = rng.integers(0, 2041, size=(H, W)).astype(np.uint16)
    for e in (near, plain, near, plain):
        ref, cost = oracle.dp_seam(e)
        buf = torch.zeros(H * W + 8, dtype=torch.uint16, device="cuda")
        for off in (0, 1):
            view = buf[off:off + H * W].view(H, W)
            view.copy_(torch.from_numpy(e))
            seam, c = sc.find_seam(view)
            sc.check()
            assert int(c.cpu()[0]) == cost
            np.testing.assert_array_equal(seam.cpu().numpy(), ref)


# forward energy from both ends: 256 columns a CTA, 16-row tiles, 32-row super-tiles; planes of one row count
# only (the lower half's first step reads the row below the last one)
@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [(191, 40), (192, 1), (193, 2), (207, 255), (223, 256), (225, 257), (255, 2049),
                                 (320, 4096), (1079, 515)])
def test_forward_from_both_ends(H, W):
    from paper_2410_21207_gb300 import binding as sc
    rng = np.random.default_rng(H * 4099 + W)
    for kind, hi in (("image", 256), ("ties", 2), ("planes", 0)):
        if hi:
            planes = oracle.forward_costs(rng.integers(0, hi, size=(H, W, 3)).astype(np.uint8))
        else:   # any values, entries without a predecessor included
            planes = tuple(rng.integers(0, 4000, size=(H, W)).astype(np.uint16) for _ in range(3))
        ref, cost = oracle.dp_seam_forward(*planes)
        seam, c = sc.find_seam_forward(*[torch.from_numpy(p).cuda() for p in planes])
        sc.check()
        assert int(c.cpu()[0]) == cost, kind
        np.testing.assert_array_equal(seam.cpu().numpy(), ref, err_msg=f"{H}x{W} {kind}")


# both passes; wider than tall, square and taller than wide (rows below the planes' last one exist or not), and
# rows wider than the refresh keeps in registers
@pytest.mark.gpu
@pytest.mark.parametrize("H,W,tw,th", [(200, 260, 240, 194), (230, 230, 210, 215), (300, 210, 200, 280),
                                       (193, 2070, 2040, 193)])
def test_forward_carve_from_both_ends(H, W, tw, th):
    from paper_2410_21207_gb300 import binding as sc
    rng = np.random.default_rng(H + W)
    for hi in (256, 2):
        img = rng.integers(0, hi, size=(H, W, 3)).astype(np.uint8)
        out, log, cost = sc.carve_forward(torch.from_numpy(img).cuda(), tw, th, with_log=True)
        sc.check()
        r_out, r_log, r_cost = oracle.carve_forward(img, tw, th, with_log=True)
        np.testing.assert_array_equal(log.cpu().numpy(), r_log)
        np.testing.assert_array_equal(cost.cpu().numpy(), r_cost)
        np.testing.assert_array_equal(out.cpu().numpy(), r_out)
