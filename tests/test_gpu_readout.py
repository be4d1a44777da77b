"""Read-outs at the sizes where their kernels can go wrong: the history conversion (blocks of 128 facets,
5 values each, through shared memory), the energy reduction (8 lanes per particle, at most 304 blocks of
32 particles, then a stride), and the adjoint's kept workspace over calls of changing size."""
import numpy as np
import pytest

import oracle
from paper_2603_13190_gb300 import ldpm, specimen, workloads
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL
from parity import assert_elementwise

pytestmark = pytest.mark.gpu
MAT = dict(WORKLOAD_MATERIAL)


def cube(n):
    return specimen.shuffled(specimen.make_cube_specimen(10.0, 2.0, 4.0, n, seed=n), seed=3)


@pytest.mark.parametrize("spec", [specimen.single_tet_specimen(), cube(60), cube(121)], ids=["12", "n60", "n121"])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-14), ("mixed", 2e-6)])
def test_history_survives_a_round_trip(spec, prec, tol):
    """Tractions set as (t_N, tangential vector, e_max) come back: exact up to the rounding of the frame and
    of its two tangential components.  A frame vector carries up to 8 units in the last place (reciprocal
    root, division and products of the basis) and enters twice, for two vectors: 32 units, 2e-6 in mixed
    mode and 4e-15 (held to 1e-14) in FP64."""
    rng = np.random.default_rng(9)
    F = spec.n_facets
    d = spec.x[spec.facet_pj] - spec.x[spec.facet_pi]
    n = d / np.linalg.norm(d, axis=1)[:, None]
    t = rng.standard_normal((F, 3)) * 10.0 ** rng.integers(-6, 3, (F, 1))
    t -= (t * n).sum(1)[:, None] * n
    h = np.concatenate([rng.standard_normal((F, 1)), t, rng.random((F, 1)) * 1e-3], 1)
    h[::17] = 0.0
    if prec == "mixed":
        h[:, [0, 4]] = h[:, [0, 4]].astype(np.float32)
    m = ldpm.Model(spec, MAT, precision=prec, dt=1e-9)
    m.set_state(np.zeros((spec.n_particles, 6)), np.zeros((spec.n_particles, 6)), h)
    got = m.get_state()[2]
    m.close()
    assert np.array_equal(got[:, [0, 4]], h[:, [0, 4]])
    scale = np.linalg.norm(h[:, 1:4], axis=1)[:, None]
    assert np.all(np.abs(got[:, 1:4] - h[:, 1:4]) <= tol * scale)


@pytest.mark.parametrize("n,edge", [(60, 10.0), (330, 14.0), (11000, 38.0)])
def test_energy_reduction_below_at_and_past_one_stride(n, edge):
    spec = specimen.make_cube_specimen(edge, 2.0, 4.0, n, seed=5)
    bc = workloads.uniaxial_tension_bc(spec, velocity=100.0, ramp_time=1e-6)
    dt = 1.0e-7
    o = oracle.Oracle(spec, MAT, dt, bc)
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc)
    o.step(6)
    m.step(6)
    eg, rg = m.energy()
    eo, ro = o.energy()
    assert_elementwise(eg[:3], eo[:3], 1e-9, "energies")
    assert_elementwise(rg, ro, 1e-9, "reactions")
    m.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_adjoint_workspace_over_changing_calls(prec):
    spec = cube(70)
    bc = workloads.uniaxial_tension_bc(spec, velocity=40.0, ramp_time=1e-5)
    seed = np.zeros((spec.n_particles, 6))
    seed[spec.face_nodes(2, 1), 2] = 1.0
    m = ldpm.Model(spec, MAT, precision=prec, dt=1.0e-7, bc=bc)
    start = ldpm.ldpm_save_checkpoint(m.h)
    for K, C in ((20, 20), (30, 4), (7, 3), (20, 20)):  # grows, shrinks, comes back
        ldpm.ldpm_load_checkpoint(m.h, start)
        got = m.adjoint(K, seed, ckpt_every=C)
        fresh = ldpm.Model(spec, MAT, precision=prec, dt=1.0e-7, bc=bc)
        ref = fresh.adjoint(K, seed, ckpt_every=C)
        fresh.close()
        assert got[0] == ref[0] and all(np.array_equal(x, y) for x, y in zip(got[1:], ref[1:])), (K, C)
    m.close()
