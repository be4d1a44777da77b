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


def in_unit(mat, s):
    """The material with stresses and density in a unit 1 / s as large (the motion is the same)."""
    return dict(mat, **{n: mat[n] * s for n in ("rho", "E0", "sigma_t", "sigma_c0", "sigma_N0")})


@pytest.mark.parametrize("kind", ["tension", "compression"])
@pytest.mark.parametrize("e", [-130, -70, 70, 130])
def test_stress_units_beyond_single_precision(kind, e):
    """At 2^+-70 the squares of the tractions, at 2^+-130 the moduli, leave the range of FP32."""
    check_trajectory(in_unit(MAT, 2.0 ** e), kind)
    check_gradient(in_unit(MAT, 2.0 ** e), kind)


def test_per_facet_parameters_beyond_single_precision():
    """Ordinary material constants, per-facet moduli and strengths below the range of FP32."""
    mat = dict(MAT, rho=MAT["rho"] * 2.0 ** -140)
    spec = cube()
    bc = loading(spec, "tension")
    par = [np.full(spec.n_facets, MAT[n] * 2.0 ** -140) for n in ("E0", "sigma_t")]
    dt = 0.7 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    o = oracle.Oracle(spec, mat, dt, bc)
    o.set_facet_params(par[0], None, par[1])
    o.step(STEPS)
    m = ldpm.Model(spec, mat, precision="fp64", dt=dt, bc=bc)
    m.set_facet_params(par[0], None, par[1])
    m.step(STEPS)
    ref = o.get_state()
    assert (ref[2][:, 4] > 2.0 * MAT["sigma_t"] / MAT["E0"]).sum() > 10
    for name, g, r in zip(("q", "v", "hist"), m.get_state(), ref):
        assert_elementwise(g, r, 1e-9, name)
    m.close()


def test_parameters_taken_back():
    """Out-of-range parameters set and taken back again leave the material's own law."""
    spec, bc, dt, o = pair(MAT, "tension")
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc)
    m.set_facet_params(np.full(spec.n_facets, 1e-40), None, np.full(spec.n_facets, 1e-44))
    m.set_facet_params(None, None, None)
    o.step(STEPS)
    m.step(STEPS)
    for name, g, r in zip(("q", "v", "hist"), m.get_state(), o.get_state()):
        assert_elementwise(g, r, 1e-9, name)
    m.close()


def test_vanishing_strain_of_softened_facets():
    """Strains of 1e-27, whose squares are below the range of FP32, on facets that have softened and carry
    traction: the boundary still depends on the direction of the strain.  Masses hold the particles still."""
    spec = cube()
    N, F = spec.n_particles, spec.n_facets
    mass, inertia = np.full(N, 1e30), np.full((N, 3), 1e30)
    rng = np.random.default_rng(8)
    q = rng.standard_normal((N, 6)) * 1e-27
    d = spec.x[spec.facet_pj] - spec.x[spec.facet_pi]
    n = d / np.linalg.norm(d, axis=1)[:, None]
    t = rng.standard_normal((F, 3))
    t -= (t * n).sum(1)[:, None] * n
    e0 = MAT["sigma_t"] / MAT["E0"]
    h = np.concatenate([rng.uniform(0.2, 0.9, (F, 1)) * MAT["sigma_t"], t, e0 * rng.uniform(1.0, 8.0, (F, 1))], 1)
    args = dict(mass=mass, inertia=inertia)
    o = oracle.Oracle(spec, MAT, 1e-8, None, **args)
    m = ldpm.Model(spec, MAT, precision="fp64", dt=1e-8, **args)
    for k in (o, m):
        k.set_state(q, np.zeros((N, 6)), h, 0)
        k.step(1)
    got, ref = m.get_state()[2], o.get_state()[2]
    m.close()
    assert np.sum(np.abs(ref[:, 0]) < 0.5 * np.abs(h[:, 0])) > 50  # capped
    # tangential components: strains enter through differences of 1e-27 numbers exactly as larger ones would
    assert_elementwise(got, ref, 1e-9, "hist")


@pytest.mark.parametrize("n_t,r_s,l_t", [(0.2, 0.0, 120.0), (0.2, 0.5, 120.0), (20.0, 0.5, 120.0), (20.0, 50.0, 120.0),
                                         (50.0, 50.0, None), (400.0, 0.0, 120.0), (400.0, 50.0, 120.0), (2.0, 0.0, None)])
def test_traction_next_to_the_fracture_boundary(n_t, r_s, l_t):
    """Softened facets with a traction within 3e-3 to 1e-5 of the boundary on either side, near pure tension
    (where the powers (2 omega / pi)^n_t vary most) and in mixed mode, for softening exponents up to 400, shear
    softening far steeper than the tensile one, and l_t a thousandth above the longest edge (None)."""
    spec = cube()
    N, F = spec.n_particles, spec.n_facets
    d = spec.x[spec.facet_pj] - spec.x[spec.facet_pi]
    l = np.linalg.norm(d, axis=1)
    mat = dict(MAT, n_t=n_t, r_s=r_s, l_t=l_t if l_t else 1.001 * l.max())
    args = dict(mass=np.full(N, 1e30), inertia=np.full((N, 3), 1e30))
    e0 = mat["sigma_t"] / mat["E0"]
    o = oracle.Oracle(spec, mat, 1e-8, None, **args)
    m = ldpm.Model(spec, mat, precision="fp64", dt=1e-8, **args)
    rng = np.random.default_rng(12)
    zero = np.zeros((N, 6))
    off = rng.choice([1e-5, 5e-5, 3e-4, 1e-3, 3e-3], F) * rng.choice([-1.0, 1.0], F)
    for shear in (1e-4, 3e-3, 0.1, 1.0):
        q = np.zeros((N, 6))
        q[:, :3] = spec.x @ (0.2 * e0 * (np.eye(3) + shear * rng.standard_normal((3, 3))))
        # e_max where the boundary has fallen to exp(-0.1) .. exp(-4) of sigma_0
        e = o.strains(q)[0].reshape(F, 3)
        om = np.arctan2(e[:, 0], np.sqrt(mat["alpha"] * (e[:, 1] ** 2 + e[:, 2] ** 2)))
        s0 = 2 * mat["sigma_t"] / (np.sin(om) + np.sqrt(np.sin(om) ** 2 + 4 * mat["alpha"] * (np.cos(om) / mat["r_st"]) ** 2))
        Hs, Ht = r_s * mat["E0"] / mat["alpha"], 2 * mat["E0"] / (mat["l_t"] / l - 1)
        H0 = Hs + (Ht - Hs) * np.maximum(2 * om / np.pi, 0) ** n_t
        h = np.zeros((F, 5))
        h[:, 0] = 100.0 * mat["sigma_t"]
        h[:, 4] = s0 / mat["E0"] * np.minimum(1.0 + rng.uniform(0.1, 4.0, F) * mat["E0"] / np.maximum(H0, 1e-9), 50.0)
        o.set_state(q, zero, h, 0)
        o.step(1)
        t = o.get_state()[2]  # the boundary, as the cap of a traction far above it
        cap = np.sqrt(t[:, 0] ** 2 + (t[:, 1:4] ** 2).sum(1) / mat["alpha"])
        h[:, 0] = np.where(t[:, 0] > 0, cap * (1.0 + off), 0.0)
        for k in (o, m):
            k.set_state(q, zero, h, 0)
            k.step(1)
        got, ref = m.get_state()[2], o.get_state()[2]
        assert np.sum(ref[:, 0] > 1e-3 * mat["sigma_t"]) > F // 3
        assert_elementwise(got, ref, 1e-9, "shear %g" % shear)
    m.close()


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("kind", ["tension", "compression"])
def test_history_without_a_maximum_strain(kind, sign):
    """A NaN e_max (of either sign) takes the facet's strain when it is next in tension, as in the oracle: it
    does not stand for a strain above all others, which would switch softening off for good."""
    spec, bc, dt, o = pair(MAT, kind)
    h = np.zeros((spec.n_facets, 5))
    h[::3, 4] = np.copysign(np.nan, sign)
    zero = np.zeros((spec.n_particles, 6))
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc)
    for k in (o, m):
        k.set_state(zero, zero, h, 0)
        k.step(STEPS)
    got, ref = m.get_state(), o.get_state()
    m.close()
    assert np.sum(~np.isnan(ref[2][::3, 4])) > 10  # some have been in tension
    assert np.array_equal(np.isnan(got[2]), np.isnan(ref[2]))
    for name, g, r in zip(("q", "v", "hist"), got, ref):
        assert_elementwise(np.nan_to_num(g), np.nan_to_num(r), 1e-9, name)
