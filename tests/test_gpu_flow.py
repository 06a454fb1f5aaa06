"""Several time steps in one launch: a call of bbx_step (or bbx_batch_step)
with n steps on unmasked grids runs them in one launch whose CTAs wait for one
another plane by plane.  The arithmetic of a node does not depend on it, so
the state, the activation map, the time and the total are bitwise those of n
calls with one step each (one launch per step)."""
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


def _grid(bbx, model, shape, fibres, ty, setup=None, seed=3):
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    h, dt = {bbx.BBX_BR: (0.2, 0.02), bbx.BBX_FHN: (0.5, 0.01)}.get(model, (0.3, 0.005))
    G = bbx.Grid(nx, ny, nz, h)
    fib = None
    if fibres == "smooth":
        fib = wl.smooth_fibres(nx, ny, nz, h)
    elif fibres == "rotational":
        fib = wl.rotational_fibres(nx, ny, nz)
    d = (0.1, 0.025) if model == bbx.BBX_BR else (1.0, 0.25)
    G.set_fibres(fib, d[0], d[1] if fib is not None else d[0])
    G.set_ionic_model(model)
    if setup:
        setup(G)
    G.set_tiling(ty, 16)
    G.set_timestep(dt)
    V = G.read_state(0)
    span = 60.0 if model == bbx.BBX_BR else 1.0
    G.write_state(0, (V + span * rng.random((nz, ny, nx))).astype(np.float32))
    return G, dt


def _lie(G):
    G.set_scheme(1)


def _stim(G):
    nz, ny, nx = G.shape
    reg = np.zeros((nz, ny, nx), np.uint8)
    reg[:, : ny // 2] = 1
    G.set_stimulus(reg, 5.0, 0.012, 0.031)


# sizes at the edges of tiles (64 columns, 7 / 14 / 28 rows) and of a share
# (columns with more and with fewer planes than a CTA takes), one CTA alone,
# remainders in every direction
CASES = [
    ("one tile", "fhn", (1, 5, 9), "none", 7, None, 9),
    ("sheet", "fhn", (1, 200, 200), "none", 14, None, 21),
    ("sheet, tall tiles", "fhn", (1, 301, 65), "none", 28, None, 8),
    ("sheet, anisotropic", "barkley", (1, 97, 130), "smooth", 7, None, 7),
    ("flat", "barkley", (2, 29, 63), "smooth", 14, None, 6),
    ("slab", "barkley", (19, 37, 100), "rotational", 14, None, 10),
    ("tall, pieces across columns", "barkley", (131, 71, 70), "rotational", 7, None, 5),
    ("isotropic block", "zfk", (33, 64, 129), "none", 14, None, 70),
    ("one variable", "diffusion", (17, 30, 64), "smooth", 7, None, 11),
    ("stimulus window", "barkley", (12, 44, 65), "smooth", 14, _stim, 9),
    ("Lie scheme", "barkley", (9, 50, 128), "smooth", 14, _lie, 4),
    ("Beeler-Reuter", "br", (15, 45, 96), "rotational", 7, None, 6),
]


@pytest.mark.parametrize("name,model,shape,fibres,ty,setup,n", CASES, ids=[c[0] for c in CASES])
def test_steps_of_one_launch_equal_single_steps_bitwise(bbx, name, model, shape, fibres, ty, setup, n):
    mid = {"fhn": bbx.BBX_FHN, "barkley": bbx.BBX_BARKLEY, "br": bbx.BBX_BR, "zfk": bbx.BBX_ZFK,
           "diffusion": bbx.BBX_DIFFUSION}[model]
    A, dt = _grid(bbx, mid, shape, fibres, ty, setup)
    B, _ = _grid(bbx, mid, shape, fibres, ty, setup)
    for _ in range(2):  # the second call starts from the parity the first one left
        A.step(dt, n)
        for _ in range(n):
            B.step(dt, 1)
        assert np.array_equal(A.read_all().view(np.uint32), B.read_all().view(np.uint32))
        assert np.array_equal(A.read_activation(), B.read_activation())
        assert A.get_time() == B.get_time()
        # (a small isotropic sheet's steps of one launch sum the total in another order)
        assert abs(A.step_total() - B.step_total()) <= 1e-12 * np.abs(A.read_state(0)).sum()


def test_halo_planes_are_read_but_never_waited_for(bbx):
    A, dt = _grid(bbx, bbx.BBX_BARKLEY, (21, 40, 70), "smooth", 14)
    B, _ = _grid(bbx, bbx.BBX_BARKLEY, (21, 40, 70), "smooth", 14)
    for G in (A, B):
        G.set_halo_planes(1, 1)
    A.step(dt, 6)
    for _ in range(6):
        B.step(dt, 1)
    assert np.array_equal(A.read_all(), B.read_all())
    assert A.step_total() == B.step_total()


# n: one launch, and one more than a launch takes
@pytest.mark.parametrize("n,planar", [(2, True), (5, False), (67, True)])
def test_batch_steps_of_one_launch_equal_single_steps_bitwise(bbx, n, planar):
    shapes = [(1, 33, 70), (1, 129, 64), (1, 17, 200)] if planar else [(20, 40, 64), (12, 30, 100), (7, 15, 65)]
    m = bbx.BBX_FHN if planar else bbx.BBX_BARKLEY

    def make():
        gs = [_grid(bbx, m, s, "none", 14, None, seed=20 + i)[0] for i, s in enumerate(shapes)]
        return gs, bbx.Batch(gs)

    ga, A = make()
    gb, B = make()
    A.step(n)
    for _ in range(n):
        B.step(1)
    A.sync()
    B.sync()
    for a, b in zip(ga, gb):
        assert np.array_equal(a.read_all(), b.read_all())
        assert np.array_equal(a.read_activation(), b.read_activation())
        assert a.get_time() == b.get_time() and a.get_time()[1] == n
        assert a.step_total() == b.step_total()
    A.close()
    B.close()


@pytest.mark.parametrize("model,shape", [("barkley", (9, 30, 70)), ("fhn", (1, 64, 96)), ("fhn", (1, 900, 700))])
def test_captured_steps_replay(bbx, model, shape):
    """A call captured into a CUDA graph replays as the same call made again."""
    torch = pytest.importorskip("torch")
    mid = bbx.BBX_BARKLEY if model == "barkley" else bbx.BBX_FHN
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        A, dt = _grid(bbx, mid, shape, "none", 14)
        A.step(dt, 4)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            A.step(dt, 4)
        for _ in range(3):
            g.replay()
        s.synchronize()
    B, _ = _grid(bbx, mid, shape, "none", 14)
    for _ in range(16):
        B.step(dt, 1)
    assert np.array_equal(A.read_all(), B.read_all())
    assert A.get_time() == B.get_time()
