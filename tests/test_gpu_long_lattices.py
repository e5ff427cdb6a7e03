"""Lattices longer than a grid has blocks along y or z (65,535): every launch
shape steps them, with the results of the shape made for them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_11524_gb300 import build, lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    lbm.load()


def _lattice(shape, storage):
    nz, ny, nx = shape
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.6, F_ext=(0, 1e-5, 2e-5), storage=storage,
                    rho0=(0.5, 0.5))
    rng = np.random.default_rng(7)
    g.set_geometry(rng.choice([0.0, 0.3, 1.0], shape), np.full(shape, 0.1))
    ra = rng.uniform(0.02, 0.98, shape)
    g.init_equilibrium(ra, 1.0 - ra)
    return g


@pytest.mark.parametrize("storage", ["f32", "f16", "f16l"])
@pytest.mark.parametrize("shape", [(1, 131073, 1), (1, 262140, 1), (65537, 1, 2), (131070, 1, 1)])
def test_every_shape_steps_a_long_lattice(shape, storage):
    ref = _lattice(shape, storage)
    ref.set_launch_config(0, 6, 6)
    ref.step(3)
    want = ref.populations()
    fields = ref.fields()
    ref.close()
    for cfg in [None, (0, 8, 9), (1, 7, 7), (2, 5, 0), (1, 1, 2), (2, 2, 3), (0, 3, 4)]:
        g = _lattice(shape, storage)
        if cfg:
            g.set_launch_config(*cfg)
        g.step(3)
        assert np.array_equal(g.populations(), want), cfg
        if cfg in (None, (1, 7, 7)):
            for k, v in g.fields().items():
                assert np.array_equal(v, fields[k]), (cfg, k)
            assert g.observables()["nonfinite"] == 0
        g.close()
