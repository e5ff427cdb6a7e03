"""The step that lbm_step picks for a float32 lattice beyond the small ones --
the wavefront launch with a lag that fits the plane, or the two passes --
against the two halves of a step, bit for bit: lattices on either side of the
rule (short in z, long lags, ragged tiles), fractions per component, moving
walls, a change of reservoirs on the way."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_11524_gb300 import build, lbm, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    lbm.load()


def _lattice(shape, per_component):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, 4)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.75, F_ext=(1e-5, 2e-5, -1e-5),
                    ns_per_component=per_component)
    g.set_geometry(ns, gads, ns[::-1, ::-1].copy() if per_component else None)
    rng = np.random.default_rng(5)
    ra = rng.uniform(0.02, 0.98, shape)
    g.init_equilibrium(ra, 1.0 - ra)
    return g


# lags 34 (170 planes are five of them, 169 are not), 53 on ragged tiles, 17
SHAPES = [(170, 64, 64), (169, 64, 64), (266, 39, 33), (96, 96, 96)]


@pytest.mark.parametrize("per_component", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_the_chosen_step_equals_the_two_halves(shape, per_component):
    a, b = _lattice(shape, per_component), _lattice(shape, per_component)
    assert a.wavefront()[0] == 0
    for n, rho in ((1, 1.0), (2, 1.02), (3, 1.04)):
        for g in (a, b):
            g.set_bc(0, 2, rho, 0.01)
            g.set_bc(3, 1, 0.5, 0.5, (0.01, 0.0, 0.02))
        a.step(n)
        for _ in range(n):
            lbm.lbm_density(b.ctx)
            lbm.lbm_collide_stream(b.ctx)
    assert a.t == b.t
    assert bytes(a.save()) == bytes(b.save())
    for k, v in a.fields().items():
        assert np.array_equal(v, b.fields()[k]), k
    assert lbm.lbm_fault_word(a.ctx) == 0
    a.close()
    b.close()
