"""The prefetching fused pass copies whole rows of 32 nodes and walks runs of
planes: the lattices where a row, its edge node or a run can go wrong (widths
around a tile, single rows and planes, wraps, runs of one plane and more)
against the plain pass, bit for bit."""
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


def _states(shape, storage, per_component, cfg, steps=3):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, 5)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.75, F_ext=(1e-5, 2e-5, -1e-5),
                    storage=storage, rho0=(0.5, 0.5), ns_per_component=per_component)
    g.set_geometry(ns, gads, ns[::-1, ::-1].copy() if per_component else None)
    if nx > 2:
        g.set_bc(1, 1, 1.04, 0.01)
    g.set_populations(synth.random_state(shape, 6))
    g.set_launch_config(0, cfg, cfg)
    out = []
    for _ in range(steps):
        g.step(1)
        out.append(g.populations())
    g.close()
    return out


SHAPES = [(1, 1, 1), (1, 1, 2), (3, 1, 31), (2, 3, 32), (5, 2, 33), (1, 9, 64), (37, 3, 65),
          (17, 33, 40), (70, 40, 96)]


@pytest.mark.parametrize("per_component", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16l"])
@pytest.mark.parametrize("shape", SHAPES)
def test_prefetching_shapes_equal_the_plain_pass(shape, storage, per_component):
    ref = _states(shape, storage, per_component, 0)
    for cfg in range(5, lbm.LBM_COLLIDE_CONFIGS):
        for t, (got, want) in enumerate(zip(_states(shape, storage, per_component, cfg), ref)):
            assert np.array_equal(got, want), (cfg, t + 1)
