"""The tuner sweeps what reaches a launch at its k."""
import pytest

from paper_2308_07173_gb300 import autotune


@pytest.mark.parametrize("k,names", [
    (10, {"occupancy", "rho_scale", "slots", "probe"}),
    (24, {"occupancy", "rho_scale", "slots", "probe"}),
    (25, {"occupancy", "rho_scale", "probe"}),
    (32, {"occupancy", "rho_scale", "probe"}),
    (33, {"occupancy", "rho_scale", "warps", "tile"}),
])
def test_swept_parameters(k, names):
    assert set(autotune.swept(k)) == names
    given = {"tile": (16, 32), "warps": (4,), "occupancy": (12.0,)}
    assert autotune.swept(k, given) == given
