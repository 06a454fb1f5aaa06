"""Values at void nodes take no part in a step: with NaN, infinities or huge
numbers there, the tissue of a masked grid steps bitwise as with zeros, at the
edges of tiles (64 columns, 7 rows) and of chunks, and void nodes keep them."""
import numpy as np
import pytest

from paper_1605_06015_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_06015_gb300 import bbx as b
    return b


@pytest.mark.parametrize("shape,frac,aniso,ty", [((1, 15, 66), 0.7, True, 7), ((1, 29, 129), 0.6, False, 14),
                                                 ((5, 8, 65), 0.8, True, 7), ((9, 15, 130), 0.5, True, 14),
                                                 ((4, 29, 64), 0.9, False, 28), ((2, 7, 17), 0.3, True, 7)])
def test_void_values_take_no_part(bbx, shape, frac, aniso, ty):
    nz, ny, nx = shape
    mask, fib = wl.random_geometry(nx, ny, nz, 9, tissue_frac=frac, aniso=aniso)
    rng = np.random.default_rng(10)
    st = rng.uniform(0.0, 1.0, (2, nz, ny, nx)).astype(np.float32)
    bad = rng.choice(np.array([np.nan, np.inf, -np.inf, 3e38], np.float32), size=st.shape)
    out = []
    for fill in (np.zeros_like(bad), bad):
        G = bbx.Grid(nx, ny, nz, 0.3, mask)
        G.set_fibres(fib, 1.0, 0.25 if aniso else 1.0)
        G.set_tiling(ty, 4)
        G.set_ionic_model(bbx.BBX_BARKLEY)
        s = np.where(mask != 0, st, fill)
        G.write_all(s)
        G.step(0.005, 3)
        got = G.read_all()
        assert np.array_equal(got[:, mask == 0].view(np.uint32), s[:, mask == 0].view(np.uint32))
        out.append((got[:, mask != 0], G.step_total()))
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32)) and out[0][1] == out[1][1]
