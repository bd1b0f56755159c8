"""The autotuner times no two configurations that are the same kernel: large launches with
tile 16 have one adjoint for every batch depth (CPU only)."""
import os
import re

import pytest

from paper_2506_05558_gb300 import autotune, gs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def test_rule_is_the_kernels():
    src = open(os.path.join(ROOT, "paper_2506_05558_gb300", "csrc", "render.cu")).read()
    a, b = re.search(r"constexpr int kBwdMinTiles = (\d+) \* (\d+);", src).groups()
    assert int(a) * int(b) == autotune.ROWS_TILES


@pytest.mark.parametrize("sizes,tried", [([(1920, 1080)], []), ([(640, 480)] * 2, [32, 64, 128]), ([(1216, 640)], []),
                                         ([(1200, 640)], [32, 64, 128])])
def test_batch_depths_of_one_kernel_are_not_compared(monkeypatch, sizes, tried):
    seen = []

    def fake(g, cams, sizes, targets, cfg, steps=3, device="cuda"):
        seen.append((cfg.tile, cfg.bwd_batch))
        return {8: 3.0, 16: 2.0, 32: 4.0}[cfg.tile] - 0.01 * len(seen)  # each a little faster: noise

    monkeypatch.setattr(autotune, "time_config", fake)
    cfg, _ = autotune.tune(None, None, sizes, None, gs.config(), steps=1, device="cpu")
    assert cfg.tile == 16 and [b for t, b in seen if b] == tried
    assert cfg.bwd_batch == (tried[-1] if tried else 0)
