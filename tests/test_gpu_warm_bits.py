"""The droplet fill rounds the fall of the profile, (rho_in - rho_v) / 2 tanh(2 s / W), before it
subtracts it from the mean density, as it always did: contracted into one operation the field
changes by some units in the last place everywhere in the vapour."""
import numpy as np
import pytest

from tests import pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(97, 130), (64, 16), (200, 65)])
def test_the_fall_of_the_profile_is_rounded(nx, ny):
    """Where the fall lies above a power of two 2^k, it is a multiple of 2^(k - 52), as is the
    mean, and so is their difference, the density, whose own last place is smaller in the
    vapour.  The rest population is 4/9 of the density, rounded: the multiple next to it must
    give that very number."""
    from paper_1211_6932_gb300.warm import WarmParams
    c = pairs.case(nx, ny, tr=0.7, sigma=0.114)
    rl, rv = pairs.maxwell(c)
    drops = np.array([[0.27 * nx, 0.53 * ny, 9.4], [0.74 * nx, 0.26 * ny, 6.3]])
    with pairs.gpu_lattice(c, "fp64") as L:
        L.init_droplets(drops, WarmParams(rl, rv, 4.2))
        f0 = L.get_populations()[0]
    k = int(np.floor(np.log2(0.5 * (rl - rv) * 0.95)))
    unit = 2.0 ** (k - 52)
    rho = f0 * 2.25
    sel = (0.5 * (rl + rv) - rho > 2.0 ** k * 1.0001) & (f0 != (4.0 / 9.0) * rv)
    assert sel.sum() > 200 and unit >= 4 * np.spacing(rho[sel].min())
    near = np.round(rho[sel] / unit) * unit
    assert np.array_equal((4.0 / 9.0) * near, f0[sel])
