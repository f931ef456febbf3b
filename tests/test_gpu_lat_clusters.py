"""A plan's heaviest image on clusters that sweep it from both ends, alone (the larger clusters) and beside
230 images of a few pixels (the smaller ones), at the widths where the cluster changes: two CTAs up to 768
columns (a CTA covers each half alone), an odd number, whose last CTA sweeps nothing, 8 warps and 12, both
passes, few rows (one half only up to 16), and the widest (16 CTAs)."""
import numpy as np
import pytest

import oracle
from paper_2410_21207_gb300 import binding as sc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,tw,th", [
    (2, 40, 1, 40), (640, 33, 620, 33), (641, 70, 630, 70), (767, 64, 760, 64), (768, 97, 760, 90), (769, 97, 760, 97),
    (1023, 16, 1015, 16), (1024, 17, 1016, 17), (1025, 48, 1015, 48), (1151, 130, 1140, 130), (1152, 200, 1140, 195),
    (1153, 65, 1145, 65), (1408, 40, 1400, 40), (1409, 40, 1400, 40), (1537, 96, 1530, 96), (2176, 31, 2170, 31),
    (2305, 50, 2300, 50), (3841, 34, 3836, 34), (5121, 32, 5116, 32), (6144, 20, 6139, 20), (300, 1000, 292, 994)])
def test_one_image_on_its_cluster(W, H, tw, th):
    rng = np.random.default_rng(W * 31 + H)
    for hi in (256, 2):   # ordinary values, and many ties
        img = rng.integers(0, hi, size=(H, W, 3), dtype=np.uint8)
        ref, log = oracle.carve(img, tw, th, with_log=True)[:2]
        dot = torch.full((2, 3, 1), 7, dtype=torch.uint8, device="cuda")
        for beside in (0, 230) if W > 2 else (0,):   # (two columns are no heavier than the rest)
            plan = sc.BatchPlan([torch.from_numpy(img).cuda()] + [dot] * beside, [(tw, th)] + [(2, 2)] * beside,
                                autotune=2, with_log=True)
            assert plan.info()["cluster_path"] == 1
            cs = sc.batch_route([(H, W, 3, tw, th)] + [(2, 3, 1, 2, 2)] * beside, 1.4, 152)[0]
            w = W if th == H else max(W, H)
            assert cs[0] == (max(2, -(-w // 384)) if beside or w > 5120 else 2 * -(-w // 640))
            for _ in range(2):
                out = plan.run()[0]
                sc.check()
                np.testing.assert_array_equal(plan.logs[0].cpu().numpy(), log)
                np.testing.assert_array_equal(out.cpu().numpy(), ref)
            plan.close()
