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
