"""The FP64 step's edge tiles (5 tetrahedra per warp) where they can go wrong: specimens whose tetrahedra
leave different remainders modulo the tile, facets on the law's boundaries (collected and evaluated apart)
beside facets off them, per-facet parameters, and batches whose tiles straddle two specimens.  Against the
oracle, per element, at the FP64 trajectories' 1e-9."""
import numpy as np
import pytest

import oracle
from paper_2603_13190_gb300 import ldpm, specimen, workloads
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL
from parity import assert_elementwise

pytestmark = pytest.mark.gpu
MAT = dict(WORKLOAD_MATERIAL)
STEPS = 60


def cube(k):
    return specimen.make_cube_specimen(8.0, 2.0, 4.0, 50 + 9 * k, seed=60 + k)


def loading(spec, kind):
    if kind == "tension":
        return workloads.uniaxial_tension_bc(spec, velocity=1500.0, ramp_time=1e-6)
    return workloads.confined_compression_bc(spec, velocity=6000.0, ramp_time=1e-6)


def compare(got, ref, what):
    for name, g, r in zip(("q", "v", "hist"), got, ref):
        assert_elementwise(g, r, 1e-9, what + " " + name)


@pytest.mark.parametrize("kind", ["tension", "compression"])
@pytest.mark.parametrize("k", range(5))
def test_boundaries_and_remainders_match_the_oracle(k, kind):
    spec = cube(k)
    bc = loading(spec, kind)
    par = [MAT[n] * np.random.default_rng(k + j).uniform(0.8, 1.2, spec.n_facets) for j, n in
           enumerate(("E0", "alpha", "sigma_t"))] if k == 4 else [None] * 3
    dt = 0.7 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    o = oracle.Oracle(spec, MAT, dt, bc)
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc)
    if k == 4:
        o.set_facet_params(*par)
        m.set_facet_params(*par)
    o.step(STEPS)
    m.step(STEPS)
    ref = o.get_state()
    # the loading has to reach the boundaries: softened facets, or yielded and sliding ones
    if kind == "tension":
        assert (ref[2][:, 4] > 2.0 * MAT["sigma_t"] / MAT["E0"]).sum() > 10
    else:
        assert (ref[2][:, 0] < -1.01 * MAT["sigma_c0"]).sum() > 10
    compare(m.get_state(), ref, "%s %d (T %% 5 = %d)" % (kind, k, spec.n_tets % 5))
    m.close()


def test_single_tetrahedron_and_straddling_batch():
    specs = [specimen.single_tet_specimen()] + [cube(k) for k in range(3)]
    bcs = [workloads.free_bc(4)] + [loading(s, "tension") for s in specs[1:]]
    bcs[0].v0[:] = 50.0 * np.random.default_rng(5).standard_normal((4, 6)) * np.array([1, 1, 1, 0.5, 0.5, 0.5])
    mats = [dict(MAT, sigma_t=MAT["sigma_t"] * (1 + 0.1 * i)) for i in range(4)]
    dts = [0.6 * oracle.Oracle(s, m, 1e-7, b).critical_dt() for s, m, b in zip(specs, mats, bcs)]
    b = ldpm.Batch(specs, mats, "fp64", dts=dts, bcs=bcs)
    b.step(STEPS)
    for i in range(4):
        o = oracle.Oracle(specs[i], mats[i], dts[i], bcs[i])
        o.step(STEPS)
        compare(b.get_state(i), o.get_state(), "specimen %d" % i)
    b.close()
