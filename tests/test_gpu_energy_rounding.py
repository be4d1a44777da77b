"""The kinetic energy of single degrees of freedom, to the rounding of its own arithmetic.

The device keeps 1 / m (one rounding, 2^-53) and forms m v^2 / 2 from the reciprocal of that (held to one unit
in the last place, 2^-52), v v and the product (2^-53 each): 5 x 2^-53 = 5.6e-16 at most, held to 6e-16.  The
other degrees of freedom are at rest and add exact zeros."""
import numpy as np
import pytest

from paper_2603_13190_gb300 import ldpm, specimen
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL

pytestmark = pytest.mark.gpu
SPEC = specimen.make_cube_specimen(8.0, 2.0, 4.0, 60, seed=60)


def energies(mass, inertia, speeds):
    """W_kin with one degree of freedom moving, for each of `speeds` [n][3]: particle, DOF, velocity."""
    N = SPEC.n_particles
    m = ldpm.Model(SPEC, dict(WORKLOAD_MATERIAL), precision="fp64", dt=1e-9, mass=mass, inertia=inertia)
    out = []
    for p, d, v in speeds:
        vel = np.zeros((N, 6))
        vel[int(p), int(d)] = v
        m.set_state(np.zeros((N, 6)), vel, None, 0)
        out.append(m.energy()[0][2])
    m.close()
    return np.array(out)


def reference(mass, inertia, speeds):
    m6 = np.concatenate([np.repeat(mass[:, None], 3, 1), inertia], 1)
    return np.array([0.5 * m6[int(p), int(d)] * v * v for p, d, v in speeds])


def test_kinetic_energy_over_the_exponent_range():
    rng = np.random.default_rng(4)
    N = SPEC.n_particles
    mass, inertia = 2.0 ** rng.uniform(-500, 500, N), 2.0 ** rng.uniform(-500, 500, (N, 3))
    mass[:20], inertia[:20] = rng.uniform(1e-12, 1e-9, 20), rng.uniform(1e-12, 1e-8, (20, 3))
    inertia[20:24, 0] = [1.0, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0), 2.0 ** -300]
    speeds = [(p, d, rng.uniform(1.0, 2.0)) for p in range(N) for d in (0, 3, 4, 5)]
    got, ref = energies(mass, inertia, speeds), reference(mass, inertia, speeds)
    assert np.all(np.abs(got - ref) <= 6e-16 * ref), np.max(np.abs(got - ref) / ref)


def test_masses_next_to_the_ends_of_the_range():
    """Masses whose reciprocals are the largest normal numbers or subnormal.  A subnormal 1 / m has lost up to
    its own rounding unit (2^-1074 m, 5e-16 at 1e308): 1.2e-15 there."""
    N = SPEC.n_particles
    inertia = np.ones((N, 3))
    inertia[0] = [1e-308, 1.2e-308, 2.3e-308]
    inertia[1] = [1e308, 5e307, 3e307]
    speeds = [(0, 3, 1e100), (0, 4, 1e100), (0, 5, 1e100), (1, 3, 1e-100), (1, 4, 1e-100), (1, 5, 1e-100)]
    got, ref = energies(np.ones(N), inertia, speeds), reference(np.ones(N), inertia, speeds)
    assert np.all(np.abs(got - ref) <= 1.2e-15 * ref), (got, ref)
