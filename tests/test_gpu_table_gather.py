"""Tabulated kernels whose warps gather table entries together (tile rows 7)
against those whose lanes read their own (tile rows 14): the same entries and
the same interpolation, so one step from a state with another V at every node,
beyond both ends of the table too, is bitwise the same."""
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


@pytest.mark.parametrize("model,shape,masked", [("br", (1, 15, 66), False), ("br", (5, 29, 129), False), ("br", (4, 15, 67), True),
                                                ("mrl", (1, 8, 1), False), ("mrl", (5, 15, 130), False)])
def test_gathered_entries_equal_own_entries_bitwise(bbx, model, shape, masked):
    nz, ny, nx = shape
    rng = np.random.default_rng(31)
    S = 8 if model == "br" else 11
    st = rng.uniform(0.0, 1.0, (S,) + shape).astype(np.float32)
    st[0] = rng.uniform(-140.0, 100.0, shape)  # (the table: -120 .. 80)
    st[0].reshape(-1)[:4] = [-120.0, 80.0, 79.99, -119.99]
    st[1] = 10 ** rng.uniform(-7.2, -5.2, shape)
    mask = (rng.random(shape) < 0.7).astype(np.uint8) if masked else None
    if masked:
        st[0][mask == 0] = np.nan
    out = []
    for ty in (7, 14):
        G = bbx.Grid(nx, ny, nz, 0.2, mask)
        # (masked: isotropic, where the two heights differ in how they gather)
        G.set_fibres(None if masked else wl.rotational_fibres(nx, ny, nz), 0.1, 0.1 if masked else 0.025)
        G.set_tiling(ty, 4)
        G.set_ionic_model(bbx.BBX_BR if model == "br" else bbx.BBX_BR_MRL)
        if model == "br":
            G.set_tabulation(True)
        G.set_wsum_elision(False)
        G.write_all(st)
        G.step(0.02, 1)
        out.append(G.read_all())
    sel = np.ones(shape, bool) if mask is None else mask != 0
    assert np.isfinite(out[0][:, sel]).all()
    assert np.array_equal(out[0][:, sel], out[1][:, sel])
