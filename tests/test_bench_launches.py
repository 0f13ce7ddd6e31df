"""The bench's count of shadow-map kernels follows the library's grouping of lights, which depends on the
triangle count and the map size."""
import pytest

import bench
import paper_2012_03325_gb300 as ep


@pytest.mark.parametrize("triangles,size,maps,launches", [
    (200192, 512, 64, 1 + 2 * 8),   # 9 lights per group
    (200192, 512, 9, 1 + 2), (200192, 512, 10, 1 + 4),
    (100, 512, 64, 1 + 2 * 2),      # 32 per group
    (5000000, 64, 64, 1 + 2 * 8),   # 8 per group
    (1000, 64, 0, 0), (0, 64, 5, 1)])
def test_shadow_map_launches(triangles, size, maps, launches):
    assert bench.shadow_map_launches(ep, triangles, size, maps) == launches
