"""The FP64 edge tiles (5 tetrahedra per warp) and the energy reduction (304 blocks of 32 particles, then a
stride) at every remainder, with the counts asserted: specimens whose tetrahedra, and whose tetrahedra padded
to 32 (the kernels' own count), leave each remainder modulo 5, per-facet parameters that differ from facet to
facet in the forward and the reverse pass, rows longer than the slot table in the reverse particle pass, and
particle counts one below, at and one past one stride.  FP64 trajectories at 1e-9 per element, gradients along
dense directions at 1e-8 (FP64) and 2e-3 (mixed) of the largest, as the other tests of these passes: the
directions are alike, so a small derivative is one where larger terms cancel."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2603_13190_gb300 import ldpm, specimen, workloads
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL
from parity import assert_elementwise

pytestmark = pytest.mark.gpu
MAT = dict(WORKLOAD_MATERIAL)
P0 = np.array([MAT["E0"], MAT["alpha"], MAT["sigma_t"]])
# particles and seed of 8 mm cubes, their tetrahedra and those padded to 32
CUBES = [(38, 0, 141, 160), (82, 1, 252, 256), (46, 2, 173, 192), (90, 1, 269, 288), (54, 0, 195, 224)]


def test_the_cubes_leave_every_remainder():
    assert sorted(t % 5 for _, _, t, _ in CUBES) == [0, 1, 2, 3, 4] == sorted(p % 5 for _, _, _, p in CUBES)


def loading(spec, kind):
    if kind == "tension":
        return workloads.uniaxial_tension_bc(spec, velocity=1500.0, ramp_time=1e-6)
    return workloads.confined_compression_bc(spec, velocity=6000.0, ramp_time=1e-6)


def parameters(spec, seed):
    return [P0[j] * np.random.default_rng(10 * seed + j).uniform(0.8, 1.2, spec.n_facets) for j in range(3)]


def gradient_along(spec, bc, dt, par, prec, steps, seed_dof=2):
    """(device, oracle) objective and directional derivatives along three dense directions."""
    seed = np.zeros((spec.n_particles, 6))
    seed[spec.face_nodes(2, 1), seed_dof] = 1.0
    D = np.random.default_rng(3).standard_normal((3, 3, spec.n_facets)) * P0[None, :, None]
    o = oracle.Oracle(spec, MAT, dt, bc)
    m = ldpm.Model(spec, MAT, precision=prec, dt=dt, bc=bc)
    for k in (o, m):
        if par:
            k.set_facet_params(*par)
    J, dJ = o.tangent(steps, seed, D[:, 0], D[:, 1], D[:, 2])
    Jg, *g = m.adjoint(steps, seed, ckpt_every=16)
    m.close()
    return (Jg, np.einsum("dpf,pf->d", D, np.array(g))), (J, dJ)


@pytest.mark.parametrize("kind", ["tension", "compression"])
@pytest.mark.parametrize("cube", CUBES, ids=["T%d" % c[2] for c in CUBES])
def test_unequal_parameters_at_every_remainder(cube, kind):
    n, seed, tets, padded = cube
    spec = specimen.make_cube_specimen(8.0, 2.0, 4.0, n, seed=seed)
    assert spec.n_tets == tets and (tets + 31) // 32 * 32 == padded
    bc = loading(spec, kind)
    dt = 0.7 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    par = parameters(spec, seed)
    o = oracle.Oracle(spec, MAT, dt, bc)
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc)
    for k in (o, m):
        k.set_facet_params(*par)
        k.step(60)
    ref = o.get_state()
    # the boundaries are reached: softened facets, or yielded and sliding ones
    if kind == "tension":
        assert (ref[2][:, 4] > 2.0 * MAT["sigma_t"] / MAT["E0"]).sum() > 10
    else:
        assert (ref[2][:, 0] < -1.01 * MAT["sigma_c0"]).sum() > 10
    for name, g, r in zip(("q", "v", "hist"), m.get_state(), ref):
        assert_elementwise(g, r, 1e-9, name)
    m.close()
    (Jg, got), (J, dJ) = gradient_along(spec, bc, dt, par, "fp64", 60)
    np.testing.assert_allclose(Jg, J, rtol=1e-11)
    assert np.abs(got - dJ).max() <= 1e-8 * np.abs(dJ).max()


@pytest.mark.parametrize("kind", ["tension", "compression"])
def test_unequal_parameters_in_the_mixed_gradient(kind):
    """Slow loading, so that few facets are within FP32's rounding of a switch of branch."""
    spec = specimen.make_cube_specimen(10.0, 2.0, 4.0, 120, seed=31)
    bc = workloads.uniaxial_tension_bc(spec, velocity=20.0 if kind == "tension" else -20.0, ramp_time=1e-5)
    dt = 0.9 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    (Jg, got), (J, dJ) = gradient_along(spec, bc, dt, parameters(spec, 7), "mixed", 200)
    np.testing.assert_allclose(Jg, J, rtol=1e-5)
    assert np.abs(got - dJ).max() <= 2e-3 * np.abs(dJ).max()


@pytest.mark.parametrize("prec,rtol", [("fp64", 1e-8), ("mixed", 2e-3)])
def test_gradient_with_rows_past_the_slot_table(prec, rtol):
    """Widely graded sizes: particles with more than 40 (tetrahedron, vertex) shares, up to 9 per lane."""
    spec = specimen.shuffled(specimen.make_cube_specimen(12.0, 0.8, 5.0, 800, seed=11), seed=2)
    cnt = np.bincount(np.asarray(spec.tets).ravel(), minlength=spec.n_particles)
    assert cnt.max() > 64 and np.sum(cnt > 40) >= 5
    bc = workloads.uniaxial_tension_bc(spec, velocity=20.0, ramp_time=1e-5)
    dt = 0.9 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    (Jg, got), (J, dJ) = gradient_along(spec, bc, dt, None, prec, 40)
    np.testing.assert_allclose(Jg, J, rtol=1e-11 if prec == "fp64" else 1e-5)
    assert np.abs(got - dJ).max() <= rtol * np.abs(dJ).max()


@pytest.mark.parametrize("n", [9727, 9728, 9729, 2 * 9728 + 1])
def test_energies_next_to_one_stride(n):
    """A cube and isolated particles, up to 304 x 32 = 9728 and past it."""
    base = specimen.make_cube_specimen(8.0, 2.0, 4.0, 60, seed=60)
    rng = np.random.default_rng(n)
    extra = n - base.n_particles
    spec = dataclasses.replace(base, x=np.concatenate([base.x, rng.uniform(0.0, 8.0, (extra, 3))]),
                               diameter=np.concatenate([base.diameter, np.full(extra, 2.0)]))
    mass, inertia = rng.uniform(1e-10, 1e-8, n), rng.uniform(1e-10, 1e-8, (n, 3))
    bc = workloads.free_bc(n)
    bc.mask[:] = rng.integers(0, 3, (n, 6))
    bc.vel[:] = rng.standard_normal((n, 6))
    bc.v0[:] = rng.standard_normal((n, 6))
    o = oracle.Oracle(spec, MAT, 1e-9, bc, mass=mass, inertia=inertia)
    m = ldpm.Model(spec, MAT, precision="fp64", dt=1e-9, bc=bc, mass=mass, inertia=inertia)
    for k in (o, m):
        k.step(3)
    (eg, rg), (eo, ro) = m.energy(), o.energy()
    m.close()
    assert_elementwise(eg[:3], eo[:3], 1e-9, "energies")
    assert_elementwise(rg, ro, 1e-9, "reactions")
