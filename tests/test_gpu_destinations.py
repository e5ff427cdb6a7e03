"""Host arrays that lbm_read_fields and lbm_get_populations are handed: where
they lie and how they are aligned decides how the results travel, never what
they are."""
import ctypes

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


# through the read-back buffer, and too large for it
SHAPES = [(3, 5, 33), (40, 48, 64)]


def _lattice(shape):
    nz, ny, nx = shape
    g = lbm.Lattice(nx, ny, nz, tau=(0.9, 1.1), G=1.75)
    ns, gads = synth.random_geometry(shape, 3)
    g.set_geometry(ns, gads)
    g.set_populations(synth.random_state(shape, 4))
    g.step(3)
    return g


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_pinned_arrays_at_any_byte(shape, offset):
    g = _lattice(shape)
    want = g.fields()

    def at(n):
        raw = torch.zeros(4 * n + 4, dtype=torch.uint8, pin_memory=True).numpy()
        return raw[offset:offset + 4 * n].view(np.float32)

    n = int(np.prod(shape))
    out = {k: at(3 * n if k == "u" else n) for k in want}
    assert not out["p"].flags.aligned
    lbm.lbm_read_fields(g.ctx, out["rho_a"], out["rho_b"], out["u"], out["p"])
    for k, v in out.items():
        assert np.array_equal(v, want[k].reshape(-1)), k
    g.close()


@pytest.mark.parametrize("shape", SHAPES)
def test_device_addresses_are_the_runtimes_to_refuse(shape):
    """The copy to the array decides, as for a large lattice: it is refused, or
    made; the process lives and so does the lattice."""
    g = _lattice(shape)
    want = g.fields()["rho_a"].reshape(-1)
    d = torch.zeros(38 * want.size, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    at = ctypes.cast(d.data_ptr(), ctypes.POINTER(ctypes.c_float))
    st = lbm.load().lbm_read_fields(g.ctx, at, None, None, None)
    assert st in (lbm.LBM_OK, lbm.LBM_ECUDA)
    if st == lbm.LBM_OK:
        assert np.array_equal(d[:want.size].cpu().numpy(), want)
    assert lbm.load().lbm_get_populations(g.ctx, at) == st
    assert np.array_equal(g.fields()["rho_a"].reshape(-1), want)
    g.close()
