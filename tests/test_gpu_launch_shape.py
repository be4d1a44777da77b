"""Launch shapes: tetrahedra per facet-pass block (8, 16, 32) have no part in the results of FP64 steps, and an
autotuned handle, whose shape depends on timings, differs by the lanes per particle alone."""
import numpy as np
import pytest

import oracle
from paper_2603_13190_gb300 import ldpm, specimen, workloads
from paper_2603_13190_gb300.workloads import WORKLOAD_MATERIAL
from parity import assert_elementwise

pytestmark = pytest.mark.gpu
MAT = dict(WORKLOAD_MATERIAL)


@pytest.fixture(scope="module")
def setup():
    spec = specimen.shuffled(specimen.make_cube_specimen(10.0, 2.0, 4.0, 120, seed=9), seed=1)
    bc = workloads.uniaxial_tension_bc(spec, velocity=1500.0, ramp_time=1e-6)
    dt = 0.7 * oracle.Oracle(spec, MAT, 1e-7, bc).critical_dt()
    return spec, bc, dt


def run(setup, **kw):
    spec, bc, dt = setup
    m = ldpm.Model(spec, MAT, precision="fp64", dt=dt, bc=bc, **kw)
    m.step(80)
    out = m.get_state()[:3], m.launch_shape()
    m.close()
    return out


@pytest.mark.parametrize("tets", [16, 32])
def test_tets_per_block_leave_fp64_steps_alone(setup, monkeypatch, tets):
    ref, shape = run(setup)
    assert tuple(shape) == (8, 8)
    monkeypatch.setenv("LDPM_TETS_PER_BLOCK", str(tets))
    got, shape = run(setup)
    assert tuple(shape) == (tets, 8)
    assert all(np.array_equal(g, r) for g, r in zip(got, ref))


def test_autotuned_fp64_handle_differs_by_its_lanes_alone(setup, monkeypatch):
    got, shape = run(setup, autotune=True)
    assert shape[0] == 8 and shape[1] in (8, 16)
    monkeypatch.setenv("LDPM_GATHER_LANES", str(shape[1]))
    ref, _ = run(setup)
    # the launch mode is timed as well; the two modes agree to rounding
    for name, g, r in zip(("q", "v", "hist"), got, ref):
        assert_elementwise(g, r, 1e-9, name)
