"""The FP64 passes decide with cheap bounds whether a facet can have reached a boundary of the law, and
evaluate the boundary only there.  The bounds have to hold for every material and state the library takes:
FP64 trajectories and gradients against the oracle, which always evaluates the whole law, over materials that
put the boundaries where the workloads' material does not.  Trajectories at the FP64 1e-9, per element;
gradients at 1e-8 along dense parameter directions, as the other adjoint tests."""
import numpy as np
import pytest

import oracle
from paper_2603_13190_gb300 import ldpm, specimen, workloads
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL
from parity import assert_elementwise

pytestmark = pytest.mark.gpu
MAT = dict(WORKLOAD_MATERIAL)
STEPS = 60

# kappa_c2 < 0 with H_c0 < H_c1 / 2: H_c falls below zero as r_DV grows, and sigma_bc below sigma_c0
SOFTENING_COMPACTION = dict(MAT, kc1=0.0, kc2=-0.3, Hc0_E0=0.1, Hc1_E0=0.6)


def cube():
    return specimen.make_cube_specimen(8.0, 2.0, 4.0, 60, seed=60)


def loading(spec, kind):
    if kind == "tension":
        return workloads.uniaxial_tension_bc(spec, velocity=1500.0, ramp_time=1e-6)
    return workloads.confined_compression_bc(spec, velocity=6000.0, ramp_time=1e-6)


def pair(mat, kind):
    """(specimen, conditions, step, oracle) of the loaded cube."""
    spec = cube()
    bc = loading(spec, kind)
    dt = 0.7 * oracle.Oracle(spec, mat, 1e-7, bc).critical_dt()
    return spec, bc, dt, oracle.Oracle(spec, mat, dt, bc)


def check_trajectory(mat, kind):
    spec, bc, dt, o = pair(mat, kind)
    m = ldpm.Model(spec, mat, precision="fp64", dt=dt, bc=bc)
    o.step(STEPS)
    m.step(STEPS)
    got, ref = m.get_state(), o.get_state()
    m.close()
    for name, g, r in zip(("q", "v", "hist"), got, ref):
        assert_elementwise(g, r, 1e-9, kind + " " + name)
    return ref


def check_gradient(mat, kind, steps=40):
    spec, bc, dt, o = pair(mat, kind)
    seed = np.zeros((spec.n_particles, 6))
    seed[spec.face_nodes(2, 1), 2] = 1.0
    rng = np.random.default_rng(3)
    D = rng.standard_normal((3, 3, spec.n_facets)) * np.array([mat["E0"], mat["alpha"], mat["sigma_t"]])[None, :, None]
    J, dJ = o.tangent(steps, seed, D[:, 0], D[:, 1], D[:, 2])
    m = ldpm.Model(spec, mat, precision="fp64", dt=dt, bc=bc)
    Jg, *g = m.adjoint(steps, seed, ckpt_every=16)
    m.close()
    np.testing.assert_allclose(Jg, J, rtol=1e-11)
    np.testing.assert_allclose(np.einsum("dpf,pf->d", D, np.array(g)), dJ, rtol=1e-8)


def test_negative_hardening_modulus():
    """H_c < 0 takes sigma_bc below sigma_c0: a trial above -sigma_c0 is not inside for that alone."""
    mat = SOFTENING_COMPACTION
    h = check_trajectory(mat, "compression")[2]
    assert np.sum((h[:, 0] < -0.5 * mat["sigma_c0"]) & (h[:, 0] > -0.98 * mat["sigma_c0"])) > 200
    check_gradient(mat, "compression")
