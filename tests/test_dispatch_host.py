"""Rules that pick a kernel's form, without a GPU."""
import pytest

from paper_2310_03921_gb300 import gap


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
def test_a_forced_tile_variant_reaches_the_gradient_product(variant):
    """Few atoms split the gradient product's K over SMs on a tile of its own; a forced variant runs it whole, on the
    forced tile (240 atoms, 300 points, D = 252: the parity test of the variants)."""
    parts = gap.lib().gap_test_contract_parts
    assert parts(240, 512, 256, 2) > 1
    try:
        gap.test_tc_force_variant(variant)
        assert parts(240, 512, 256, 2) == 1
        assert parts(240, 512, 256, 3) > 1  # three planes have one tile
    finally:
        gap.test_tc_force_variant(-1)
    assert parts(240, 512, 256, 2) > 1


def test_block_roofline_counts_the_clusters_sms():
    import bench
    r = bench.alu_rooflines({"solve_block": 0.04}, n_atoms=1000, n_pairs=30000, n_max=8, l_max=6, D=252, M=2000,
                            fp32_peak=80.0, fp64_peak=1.2, hbm=6800.0, n_sm=152, n_fact=2)["solve_block"]
    assert r["sms"] == 8 and r["frac_of_sms"] == pytest.approx(r["frac"] / 8)
