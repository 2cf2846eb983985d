"""Every plan of a 2D step loop in one launch has the kernel that it needs: the grid's own stencil, room
for all of a band's nodes, and shared memory that a CTA can have.  Host code only."""
import pytest

from paper_1903_12522_gb300 import cmcg

# short and long rows and columns; the widths around which a grid of three rows leaves one CTA
WIDTHS = sorted({*range(2, 40), *range(56, 72), *range(500, 530), 700, 783, *range(1000, 1030), 1100, *range(1350, 1370),
                 *range(2040, 2060), *range(2700, 2900, 3), 2727, 2728, 2729, 2730, 2891, 2892, *range(4080, 4110), 5800, 8200})


@pytest.mark.parametrize("elem", [4, 8])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("bands_max", [152, 100, 16, 5, 1])
def test_every_plan_has_its_kernel(elem, order, bands_max):
    planned = 0
    for nx in WIDTHS:
        for ny in (2, 3, 4, 5, 8, 17, 40, 128, 300, 444, 768, 1024):
            for n in ((nx, ny), (ny, nx)):
                g = cmcg.make_grid(n, 0.01, order)
                bands, rows, cluster, per_item, reach, npt, threads, smem = cmcg.cmcg_band_plan_selftest(g, elem, bands_max)
                if bands == 0:
                    continue
                planned += 1
                assert npt > 0, n
                assert reach == order // 2, n
                assert (per_item == 4) == (elem == 4 and order == 2), n
                items = (n[0] + 1 + per_item - 1) // per_item
                assert rows * items <= npt * threads, n
                assert smem <= 227 * 1024, n
                assert bands <= bands_max and bands * rows >= n[1] + 1, n
                assert bands == 1 or ((n[1] + 1) // bands >= reach + 1 and (cluster == bands) == (bands <= 16)), n
    assert planned > 100
