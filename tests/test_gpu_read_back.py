"""Read-backs: small ones through the host-mapped buffer, larger ones through
the staging planes in several rounds, the density fields without the velocity
pass, reductions of lattices with fewer blocks than the full grid -- against
each other and against sums formed on the host."""
import threading

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


def _lattice(shape, storage="f32", seed=3):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, seed)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.1), G=1.75, storage=storage, rho0=(0.5, 0.5))
    g.set_geometry(ns, gads)
    f = synth.random_state(shape, seed + 1).astype(np.float32)
    g.set_populations(f)
    return g, f


# 6,898 nodes are the last whose 38 populations fit the buffer of 1 MB, 5,461
# the last whose fields fit their share of 128 KB
SHAPES = [(1, 1, 1), (3, 5, 33), (1, 43, 127), (1, 2, 2731), (1, 2, 3449), (1, 1, 6899),
          (40, 48, 64)]


@pytest.mark.parametrize("shape", SHAPES)
def test_populations_and_density_fields(shape):
    g, f = _lattice(shape)
    assert np.array_equal(g.populations(), f)
    for steps in (1, 1):
        g.step(steps)
        pops = g.populations()
        full = g.fields()
        only = {k: np.empty(shape, np.float32) for k in ("rho_a", "rho_b", "p")}
        lbm.lbm_read_fields(g.ctx, only["rho_a"], only["rho_b"], None, only["p"])
        for k, v in only.items():
            assert np.array_equal(v, full[k]), k
        # the library sums in direction order, in float32
        for s, k in enumerate(("rho_a", "rho_b")):
            rho = pops[s, 0].copy()
            for i in range(1, 19):
                rho += pops[s, i]
            assert np.array_equal(rho, full[k]), k
        # FP64 sums of n float32 values: a few ulps of the sum of magnitudes
        mass = g.observables()["mass"]
        for s, k in enumerate(("rho_a", "rho_b")):
            want = full[k].astype(np.float64).sum()
            assert abs(mass[s] - want) <= 1e-13 * abs(want)
    g.close()


@pytest.mark.parametrize("storage", ["f16", "bf16l"])
def test_sixteen_bit_populations_of_both_read_back_paths_agree(storage):
    """The same tiles read as a small lattice and as part of a larger one."""
    small, f = _lattice((4, 6, 64), storage)
    big = lbm.Lattice(64, 6, 120, tau=(0.9, 1.1), G=1.75, storage=storage, rho0=(0.5, 0.5))
    big.set_geometry(np.zeros((120, 6, 64)))
    big.set_populations(np.tile(f, (1, 1, 30, 1, 1)))
    assert np.array_equal(big.populations()[:, :, :4], small.populations())
    big.close()
    small.close()


def test_two_threads_read_at_once():
    lats = []
    for k in range(2):
        with torch.cuda.stream(torch.cuda.Stream()):
            lats.append(_lattice((6, 20, 70), seed=20 + k)[0])
    torch.cuda.synchronize()
    want = [(g.fields(), g.populations(), g.observables()["mass"]) for g in lats]
    bad = []

    def work(k):
        for _ in range(50):
            fields, pops, mass = lats[k].fields(), lats[k].populations(), lats[k].observables()["mass"]
            if not (all(np.array_equal(fields[n], want[k][0][n]) for n in fields)
                    and np.array_equal(pops, want[k][1]) and np.array_equal(mass, want[k][2])):
                bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for g in lats:
        g.close()


@pytest.mark.parametrize("shape", [(3, 5, 33), (9, 31, 70), (40, 48, 64)])
@pytest.mark.parametrize("without", [None, "rho_b", "u", "p"])
def test_pinned_and_pageable_destinations_agree(shape, without):
    g, _ = _lattice(shape, "f16l")
    g.step(3)
    want = g.fields()
    n = int(np.prod(shape))

    def pinned(count):            # one value in, so that no array starts on a vector's boundary
        return torch.empty(count + 1, dtype=torch.float32, pin_memory=True).numpy()[1:]

    out = {k: pinned(n * (3 if k == "u" else 1)) for k in want if k != without}
    for v in out.values():
        v[...] = -1.0
    lbm.lbm_read_fields(g.ctx, out.get("rho_a"), out.get("rho_b"), out.get("u"), out.get("p"))
    for k, v in out.items():
        assert np.array_equal(v, want[k].reshape(-1)), k
    g.close()
