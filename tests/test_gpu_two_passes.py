"""The two-pass step, asked for, at the benchmark's full size against the
launches that may replace it (lbm_step's own choice and the wavefront step),
bit for bit, and several lattices on streams and threads of their own, one in
each launch lbm_step chooses, against the halves of a step."""
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


def test_two_passes_of_the_full_size_electrode():
    case = synth.electrode((256, 256, 256))
    saved = []
    for wave in (0, None, 1, 2):             # None: the library's choice
        g = lbm.Lattice(256, 256, 256, tau=case.tau, G=case.G, F_ext=case.F_ext, rho0=(0.5, 0.5))
        g.set_geometry(case.ns, case.gads2)
        for face, (L, r1, r2) in case.reservoirs.items():
            g.set_bc(face, L, r1, r2)
        g.init_equilibrium(case.rho_a, case.rho_b)
        if wave is not None:
            g.set_wavefront(wave)
        g.step(2)
        saved.append(bytes(g.save()))
        assert lbm.lbm_fault_word(g.ctx) == 0
        g.close()
    assert all(s == saved[0] for s in saved[1:])


def _lattice(shape, storage, seed):
    nz, ny, nx = shape
    ns, gads = synth.random_geometry(shape, seed)
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.2), G=1.75, F_ext=(1e-5, 2e-5, -1e-5),
                    storage=storage, rho0=(0.5, 0.5))
    g.set_geometry(ns, gads)
    g.set_bc(0, 2, 1.02, 0.01)
    ra = np.random.default_rng(seed).uniform(0.02, 0.98, shape)
    g.init_equilibrium(ra, 1.0 - ra)
    return g


def test_lattices_on_streams_and_threads_of_their_own():
    # one cluster, blocks of one tile a warp, of several tiles a warp, wavefront
    kinds = [((1, 64, 64), "f32"), ((32, 32, 32), "f16l"), ((40, 40, 40), "f32"), ((96, 96, 96), "f32")]
    lats = []
    for k, (shape, storage) in enumerate(kinds):
        with torch.cuda.stream(torch.cuda.Stream()):
            lats.append(_lattice(shape, storage, k))
    torch.cuda.synchronize()
    errors = []

    def work(g):
        try:
            for n in (1, 20, 300, 7):
                g.step(n)
            lbm.lbm_sync(g.ctx, 60.0)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(g,)) for g in lats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for k, (shape, storage) in enumerate(kinds):
        ref = _lattice(shape, storage, k)
        for _ in range(328):
            lbm.lbm_density(ref.ctx)
            lbm.lbm_collide_stream(ref.ctx)
        assert bytes(lats[k].save()) == bytes(ref.save()), kinds[k]
        ref.close()
        lats[k].close()
