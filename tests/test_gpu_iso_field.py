"""The isosurface field on grids on both sides of the size where it changes from eight lanes per
corner to one thread (160,000 corners), ragged last blocks, with boundary and soft particles
among the candidates: within the bar of the field's parity test of the oracle's field."""
import numpy as np
import pytest

import oracle
from oracle import iso as oiso
from paper_2511_15908_gb300 import scenes

from test_gpu_iso import sph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cube_over_h", [2.0, 1.0, 0.47, 0.3])
def test_field_matches_oracle_on_both_walks(sph, cube_over_h):  # noqa: F811
    sc = scenes.tiny(seed=2, n=(9, 9, 9))
    h, rho0 = sc.params["h"], sc.params["rho0"]
    cube = float(np.float32(cube_over_h * h))
    hi = np.asarray(sc.params["lo"], float) + 56.0 * 0.3 * h          # up to ~56^3 corners
    sc.params = dict(sc.params, hi=tuple(float(v) for v in np.maximum(hi, sc.params["hi"])))
    sim = sph.Simulation(sc)
    dims, origin = sph.iso_grid(sc.params, cube)
    f = sim.iso_field(cube).cpu().numpy()
    x = np.ascontiguousarray(sc.fluid_x, np.float32)
    m = np.full(len(x), float(oracle.particle_mass(rho0, sc.fluid_spacing)))
    want = oiso.field(x, m, np.ones(len(x), np.int32), h, dims, origin, np.float32(cube))
    assert np.abs(f - want).max() <= 1e-5 * rho0
    assert want.max() > 0.5 * rho0
    sim.close()
