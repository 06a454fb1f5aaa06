"""Small isotropic sheets step many steps in one cluster's registers and shared
memory; the arithmetic is the tiled kernel's, so n steps in one call are
bitwise n calls of one step (tiled): state, activation map, time; the total to
FP64 rounding.  Shapes: every number of rows a thread can own, odd widths,
the fewest rows (one per CTA), bands of unequal height, and the first shape
past each limit (which the tiled kernel takes)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_06015_gb300 import bbx as b
    return b


@pytest.mark.parametrize("nx,ny,model", [(1, 16, "fhn"), (2, 17, "barkley"), (15, 15, "fhn"), (33, 31, "zfk"), (200, 200, "fhn"),
                                         (199, 201, "barkley"), (128, 500, "fhn"), (300, 300, "diffusion"), (511, 333, "fhn"),
                                         (96, 1000, "barkley"), (512, 512, "fhn"), (2000, 16, "fhn"), (2049, 17, "zfk"),
                                         (640, 640, "fhn")])
def test_resident_steps_equal_tiled_steps_bitwise(bbx, nx, ny, model):
    mid = {"fhn": bbx.BBX_FHN, "barkley": bbx.BBX_BARKLEY, "zfk": bbx.BBX_ZFK, "diffusion": bbx.BBX_DIFFUSION}[model]
    rng = np.random.default_rng(nx + ny)
    S = bbx.NVARS[mid]
    st = rng.uniform(-0.2, 1.2, (S, 1, ny, nx)).astype(np.float32)
    reg = (rng.random((1, ny, nx)) < 0.3).astype(np.uint8)
    out = []
    for one in (False, True):
        G = bbx.Grid(nx, ny, 1, 0.5)
        G.set_fibres(None, 1.0, 1.0)
        G.set_ionic_model(mid)
        G.set_threshold(0.5)
        G.set_stimulus(reg, 4.0, 0.015, 0.04)
        G.write_all(st)
        for n in (7, 2, 4):
            if one:
                for _ in range(n):
                    G.step(0.01, 1)
            else:
                G.step(0.01, n)
        out.append((G.read_all(), G.read_activation(), G.get_time(), G.step_total()))
    a, b = out
    assert np.array_equal(a[0].view(np.uint32), b[0].view(np.uint32))
    assert np.array_equal(a[1], b[1]) and a[2] == b[2]
    # both sum doubles (or float pairs) of the same floats
    assert abs(a[3] - b[3]) <= 1e-12 * np.abs(a[0][0]).sum()
