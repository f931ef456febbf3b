"""sc_batch_route tells what a plan launches: for images of every width, the cluster sizes and shapes it
reports are those of the layout that a plan's launches are made from (called in the library through its
own header, by a small program built here; no device call)."""
import os
import random
import shutil
import subprocess

import pytest

from paper_2410_21207_gb300 import binding as sc
from paper_2410_21207_gb300 import build

CSRC = os.path.join(os.path.dirname(build.__file__), "csrc")
PROGRAM = r"""
#include <cstdio>
#include "sc_host.h"
#include "sc_batch_cl.h"
int main() {
  float thr; int sms, n;
  if (scanf("%f %d %d", &thr, &sms, &n) != 3) return 1;
  std::vector<sc_image_desc> d(n);
  for (auto &x : d) { x = {}; if (scanf("%d %d %d %d %d", &x.H, &x.W, &x.C, &x.target_w, &x.target_h) != 5) return 1; }
  sc::BatchCfg c{15, 16};
  c.thr_bal = thr;
  c.sms = sms;
  sc::BatchSetup b;
  sc::batch_layout(d.data(), n, c, nullptr, b);
  std::vector<int> cs(n, 0), shape(n, 0);
  for (auto &g : b.cl) {
    const sc::ClOps o = sc::cl_ops(g.shape);
    for (int k : g.index) {
      if (sc::batch_cl_cols(g.cs, g.shape) < sc::batch_need_width(d[k])) return 2;   // not covered
      cs[k] = g.cs;
      shape[k] = o.tile_rows == 8 ? 0 : 1;
    }
  }
  for (int k : b.fallback) cs[k] = -1;
  for (int k = 0; k < n; ++k) printf("%d %d\n", cs[k], shape[k]);
  return 0;
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    lib = build.build()
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", os.path.join(cuda, "include"), str(d / "layout.cc"), lib,
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(d / "layout")], check=True)

    def run(sizes, thr, sms):
        text = f"{thr} {sms} {len(sizes)}\n" + "\n".join(" ".join(map(str, s)) for s in sizes)
        out = subprocess.run([str(d / "layout")], input=text, capture_output=True, text=True, check=True).stdout
        rows = [tuple(map(int, ln.split())) for ln in out.splitlines()]
        return [r[0] for r in rows], [r[1] for r in rows]
    return run


@pytest.mark.parametrize("thr", [0.0, 0.5, 1.4])
def test_reported_clusters_are_those_of_the_layout(layout, thr):
    rng = random.Random(int(thr * 10))
    sizes = []
    # (no width that only the one-CTA configurations of 8-row tiles cover: the default one is laid out here)
    for k, W in enumerate(w for w in range(200, 8192, 83) if not 1440 < w <= 1680):
        H = rng.randrange(200, 1200)
        sizes.append((H, W, 3, W - rng.randrange(20, 180), H - (rng.randrange(1, 20) if k % 3 == 0 else 0)))
    cs, shape, _ = sc.batch_route(sizes, thr, 16)
    assert (cs, shape) == layout(sizes, thr, 16)


def test_every_balanced_image_up_to_6144_columns_has_a_latency_cluster(layout):
    """One image alone is above any share and has the SMs: 2 ceil(width / 640) CTAs up to 16; where that is
    more, and beside 230 light images, max(2, ceil(width / 384))."""
    light = [(40, 30, 3, 29, 40)] * 230
    for W in (100, 640, 641, 700, 768, 769, 1152, 1153, 1408, 1409, 1536, 1537, 2500, 5120, 5121, 5200, 6144):
        size = [(600, W, 3, W - 50, 600)]
        two, fewer = 2 * -(-W // 640), max(2, -(-W // 384))
        cs, shape, _ = sc.batch_route(size, 1.4, 152)
        assert (cs, shape) == ([two if two <= 16 else fewer], [1]), W
        assert layout(size, 1.4, 152) == (cs, shape), W
        cs, shape, _ = sc.batch_route(size + light, 1.4, 152)
        assert (cs, shape) == ([fewer] + [0] * 230, [1] + [0] * 230), W
        assert layout(size + light, 1.4, 152) == (cs, shape), W
    cs, shape, _ = sc.batch_route([(600, 6145, 3, 6100, 600)], 1.4, 152)
    assert (cs, shape) == ([9], [0])
