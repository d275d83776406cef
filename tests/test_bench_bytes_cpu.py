"""The bytes behind the bandwidths that bench.py prints: of the active cells alone, so that a
fraction of the peak is never above what was moved."""
import bench
import pytest

from paper_1812_03191_gb300 import inputs as I


def test_printed_bandwidths_count_the_active_cells():
    cfg = I.precision()
    n, G, band = cfg["n"], cfg["G"], cfg["params"]["band"]
    kinds = {"source": (10.0, 310), "sweep": (68.5, 930), "commmean": (4.0, 150),
             "commup": (6.0, 150), "dt": (1.5, 100)}
    t = bench.kernel_hbm_table(cfg, kinds, 4, True, 6800.0, active=True)
    assert set(t) == {"source", "sweep", "commmean", "commup"}

    def gbs(elements, kind):
        ms, launches = kinds[kind]
        return 4 * elements / (ms / launches / 1e3) / 1e9

    # rho, e, phi, v3 -> v3; x: rho, e, v3 -> 5, y and z: rho, e, pi3, v_d -> 5
    assert t["source"]["gbs"] == pytest.approx(gbs(9 * n**3, "source"), abs=0.1)
    assert t["sweep"]["gbs"] == pytest.approx(gbs((10 + 11 + 11) / 3 * n**3, "sweep"), abs=0.1)
    # coarse cells within the band of the child's frontier: 8 cells of rho and e, 4 faces of v
    near = sum(min(min(i, n // 2 - 1 - i) for i in (x, y, z)) < band
               for x in range(n // 2) for y in range(n // 2) for z in range(n // 2))
    assert t["commmean"]["gbs"] == pytest.approx(gbs((28 + 5) * near, "commmean"), abs=0.1)
    # fine ghosts, and the coarse cells that their stencils reach
    hosts = (n // 2 + G + 2) ** 3 - (n // 2 - 2) ** 3
    assert t["commup"]["gbs"] == pytest.approx(
        gbs(5 * ((n + 2 * G) ** 3 - n**3 + hosts), "commup"), abs=0.1)
    # never above the count over the level step's whole margin
    whole = bench.kernel_hbm_table(cfg, kinds, 4, True, 6800.0)
    assert all(t[k]["gbs"] < whole[k]["gbs"] for k in t)


def test_pool_bytes_of_one_coarse_step():
    # three levels: 1 + 2 + 4 level steps; two of the finest's four follow another
    assert bench.pool_bytes_per_step(32, 3, "sweep", 4) == pytest.approx(7 * 32 * 4 * 32**3)
    assert bench.pool_bytes_per_step(32, 3, "source", 4) == pytest.approx(5 * 9 * 4 * 32**3)
    assert bench.pool_bytes_per_step(32, 1, "source", 4) == pytest.approx(9 * 4 * 32**3)
