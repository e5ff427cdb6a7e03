"""Several steps of a small lattice per launch (the cluster and the
cooperative variant) against the two passes step by step, bit for bit: tile
counts around each variant's limits, storages, both parities, reservoirs that
change on the way, more steps than one launch takes; and a wait that runs
out, reported and recovered from."""
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


def _lattice(shape, storage, per_component=False):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, 8)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.75, F_ext=(1e-5, 2e-5, -1e-5),
                    storage=storage, rho0=(0.5, 0.5), ns_per_component=per_component)
    g.set_geometry(ns, gads, ns[::-1, ::-1].copy() if per_component else None)
    g.set_populations(synth.random_state(shape, 9))
    return g


def _halves(g, n):
    for _ in range(n):
        lbm.lbm_density(g.ctx)
        lbm.lbm_collide_stream(g.ctx)


def _same(a, b):
    assert a.t == b.t
    assert np.array_equal(a.populations(), b.populations()), a.t
    for k, v in a.fields().items():
        assert np.array_equal(v, b.fields()[k]), k
    assert bytes(a.save()) == bytes(b.save())


# tiles: 1, 2, 15, 16, 17 (two warps a block), 127, 128 (the cluster's last),
# 129, 351 (three x-tiles, ragged), 1217 (a second tile for some warps), 4608
SHAPES = [(1, 1, 1), (1, 2, 33), (5, 3, 32), (1, 16, 7), (17, 1, 31), (127, 1, 20), (16, 4, 64),
          (43, 3, 32), (9, 13, 70), (1217, 1, 5), (48, 48, 48)]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f16l", "bf16l"])
@pytest.mark.parametrize("shape", SHAPES)
def test_small_lattices_equal_the_two_passes(shape, storage):
    a, b = _lattice(shape, storage), _lattice(shape, storage)
    for n in (1, 2, 5):                      # starts at both parities
        a.step(n)
        _halves(b, n)
    _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(1, 7, 40), (6, 30, 33)])
def test_reservoir_changes_fractions_per_component_and_many_steps(shape):
    a, b = _lattice(shape, "f32", True), _lattice(shape, "f32", True)
    for n, rho in ((3, 1.0), (4, 1.02), (520, 1.04)):
        for g in (a, b):
            g.set_bc(0, 2, rho, 0.01)
            g.set_bc(3, 1, 0.5, 0.5, (0.01, 0.0, 0.02))
        a.step(n)
        _halves(b, n)
        _same(a, b)
    a.close()
    b.close()


def test_a_wait_that_runs_out_is_reported_and_recovered_from():
    shape = (6, 30, 33)                      # 360 tiles: the cooperative variant
    a, b = _lattice(shape, "f32"), _lattice(shape, "f32")
    a.step(2)
    kept = a.save()
    lbm.lbm_set_wavefront_limits(a.ctx, 2000, 0)
    a.step(4)
    with pytest.raises(lbm.LbmError) as e:
        a.observables(allow_nan=True)
    assert e.value.status == lbm.LBM_EINTERNAL
    with pytest.raises(lbm.LbmError):
        a.step(1)
    lbm.lbm_set_wavefront_limits(a.ctx, 0, -1)
    a.load(kept)
    a.step(4)
    _halves(b, 6)
    _same(a, b)
    a.close()
    b.close()
