"""Bytes of workspace per node: a solve at the size that just fits the device must not stop fitting because of
a faster kernel's copies.  FP64 needs none beyond the 227.5 B of the vectors and levels, FP32 and mixed
precision in 3D one padded copy of kappa (4 B times the pitch over the row) beyond 247.5 and 263.5 B."""
import pytest

from paper_1903_12522_gb300 import cmcg


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [256, 512, 900])
def test_3d(n, order):
    g = cmcg.make_grid((n, n, n), 0.01, order)
    pad = 4.0 * ((n + 4) // 4 * 4) / (n + 1)
    for precision, base in ((cmcg.FP64, 227.51), (cmcg.FP32, 247.51 + pad), (cmcg.MIXED, 263.51 + pad)):
        per_node = cmcg.cmcg_workspace_size(g, cmcg.make_options(precision)) / (n + 1) ** 3
        assert per_node <= base + 0.07, (precision, per_node)  # 0.07: flags of where the source is not zero


@pytest.mark.parametrize("n", [1500, 3000])
def test_2d_past_the_chip(n):
    g = cmcg.make_grid((n, n), 0.01)
    for precision, base in ((cmcg.FP64, 230.95), (cmcg.FP32, 250.95), (cmcg.MIXED, 266.95)):
        assert cmcg.cmcg_workspace_size(g, cmcg.make_options(precision)) / (n + 1) ** 2 <= base
