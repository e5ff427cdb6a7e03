"""The prefetching fused pass where its blocks walk runs of 4, 8 and 16 planes
(a last, shorter run among them): the ring of five density planes comes round
several times and the copies' offsets wrap, which small lattices, whose runs
are one or two planes, do not reach.  Every prefetching shape against the
plain pass, bit for bit, after each of three steps."""
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


def _run(shape, by):
    """Planes per block: the longest run that makes 152 x 24 / by blocks."""
    nz, ny, nx = shape
    columns = ((nx + 31) // 32) * ((ny + by - 1) // by)
    return next((zc for zc in (16, 8, 4, 2) if columns * -(-nz // zc) >= 152 * 24 // by), 1)


def _states(shape, storage, per_component, cfg):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, 5)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.75, F_ext=(1e-5, 2e-5, -1e-5),
                    storage=storage, rho0=(0.5, 0.5), ns_per_component=per_component)
    g.set_geometry(ns, gads, ns[::-1, ::-1].copy() if per_component else None)
    g.set_bc(1, 1, 1.04, 0.01)
    rng = np.random.default_rng(6)
    ra = rng.uniform(0.02, 0.98, shape)
    g.init_equilibrium(ra, 1.0 - ra)
    g.set_launch_config(0, cfg, cfg)
    out = []
    for _ in range(3):
        g.step(1)
        out.append(bytes(g.save()))
    assert lbm.lbm_fault_word(g.ctx) == 0
    g.close()
    return out


@pytest.mark.parametrize("storage,per_component", [("f32", False), ("f16", True), ("bf16l", False)])
@pytest.mark.parametrize("shape,run", [((41, 127, 90), 4), ((75, 127, 90), 8), ((147, 127, 90), 16)])
def test_long_runs_equal_the_plain_pass(shape, run, storage, per_component):
    assert {_run(shape, by) for by in (2, 4, 8)} == {run} and shape[0] % run
    ref = _states(shape, storage, per_component, 0)
    for cfg in range(5, lbm.LBM_COLLIDE_CONFIGS):
        assert _states(shape, storage, per_component, cfg) == ref, cfg
