"""Which kernels a call of bbx_step takes: by the grid's size and the number of
steps, or as bbx_debug_route asks for; every route gives the results of calls
of one step bitwise."""
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


def _sheet(bbx, nx, ny, model, seed=1):
    mid = {"fhn": bbx.BBX_FHN, "barkley": bbx.BBX_BARKLEY, "zfk": bbx.BBX_ZFK, "diffusion": bbx.BBX_DIFFUSION}[model]
    G = bbx.Grid(nx, ny, 1, 0.5)
    G.set_fibres(None, 1.0, 1.0)
    G.set_ionic_model(mid)
    rng = np.random.default_rng(seed)
    G.write_all(rng.uniform(-0.2, 1.2, (bbx.NVARS[mid], 1, ny, nx)).astype(np.float32))
    G.set_threshold(0.5)
    G.set_stimulus((rng.random((1, ny, nx)) < 0.3).astype(np.uint8), 4.0, 0.015, 0.04)
    return G


def _same(a, b):
    assert np.array_equal(a.read_all().view(np.uint32), b.read_all().view(np.uint32))
    assert np.array_equal(a.read_activation(), b.read_activation())
    assert a.get_time() == b.get_time()
    assert abs(a.step_total() - b.step_total()) <= 1e-12 * np.abs(a.read_state(0)).sum()


def _one_by_one(G, dt, n):
    for _ in range(n):
        G.step(dt, 1)


@pytest.mark.parametrize("nx,ny,model,n,resident", [(64, 64, "fhn", 2, True), (400, 400, "fhn", 4, False),
                                                    (400, 400, "fhn", 5, True), (512, 512, "barkley", 14, False),
                                                    (512, 512, "barkley", 15, True), (520, 520, "fhn", 70, False),
                                                    (512, 512, "zfk", 4, False), (512, 512, "zfk", 6, True), (560, 560, "zfk", 10, False)])
def test_short_calls_on_large_sheets_take_tiles(bbx, nx, ny, model, n, resident):
    A, B = _sheet(bbx, nx, ny, model), _sheet(bbx, nx, ny, model)
    A.step(0.01, n)
    assert A.debug_launches()[2] == (1 if resident else 0) and A.debug_launches()[3] == 0
    _one_by_one(B, 0.01, n)
    assert B.debug_launches() == [n, 0, 0, 0]
    _same(A, B)


# the shapes of the register-resident kernel (every number of rows a thread owns), in calls too
# short to take it by themselves, asked for by the switch or by the hook
@pytest.mark.parametrize("ask", ["set_resident", "debug_route"])
@pytest.mark.parametrize("nx,ny,model", [(1, 16, "fhn"), (200, 200, "barkley"), (300, 300, "diffusion"), (511, 333, "fhn"),
                                         (400, 400, "barkley"), (512, 512, "fhn"), (513, 511, "barkley"), (560, 560, "zfk")])
def test_resident_calls_asked_for(bbx, ask, nx, ny, model):
    A, B = _sheet(bbx, nx, ny, model), _sheet(bbx, nx, ny, model)
    if ask == "set_resident":
        A.set_resident(True)
    else:
        A.debug_route(bbx.BBX_ROUTE_REGISTERS)
    for n in (3, 2):
        A.step(0.01, n)
        _one_by_one(B, 0.01, n)
    assert A.debug_launches() == [0, 0, 2, 0]
    _same(A, B)


@pytest.mark.parametrize("nx,ny", [(200, 200), (900, 700)])
def test_one_launch_a_step_asked_for(bbx, nx, ny):
    A, B = _sheet(bbx, nx, ny, "fhn"), _sheet(bbx, nx, ny, "fhn")
    A.debug_route(bbx.BBX_ROUTE_STEPS)
    A.step(0.01, 30)
    assert A.debug_launches() == [30, 0, 0, 0]
    _one_by_one(B, 0.01, 30)
    _same(A, B)
    with pytest.raises(bbx.BbxError):
        A.debug_route(4)


def _block(bbx, model, shape, fibres, ty, setup=None):
    from test_gpu_flow import _grid
    mid = {"fhn": bbx.BBX_FHN, "barkley": bbx.BBX_BARKLEY, "br": bbx.BBX_BR, "zfk": bbx.BBX_ZFK,
           "diffusion": bbx.BBX_DIFFUSION}[model]
    return _grid(bbx, mid, shape, fibres, ty, setup)


@pytest.mark.parametrize("model,shape,fibres,ty,n,several", [
    ("fhn", (1, 900, 700), "none", 14, 5, False), ("fhn", (1, 900, 700), "none", 28, 64, False),
    ("barkley", (1, 130, 200), "smooth", 14, 8, False), ("barkley", (1, 130, 200), "smooth", 14, 9, True),
    ("barkley", (16, 64, 64), "rotational", 14, 7, False), ("barkley", (16, 64, 64), "rotational", 14, 8, True),
    ("fhn", (96, 96, 96), "none", 28, 64, False), ("barkley", (128, 128, 128), "rotational", 7, 2, False),
    ("barkley", (128, 128, 128), "rotational", 7, 3, True), ("fhn", (128, 128, 128), "none", 14, 6, False),
    ("fhn", (1, 2048, 2048), "none", 28, 2, True), ("br", (9, 40, 64), "rotational", 7, 30, False)])
def test_short_calls_on_small_grids_take_one_launch_a_step(bbx, model, shape, fibres, ty, n, several):
    A, dt = _block(bbx, model, shape, fibres, ty)
    B, _ = _block(bbx, model, shape, fibres, ty)
    A.step(dt, n)
    assert A.debug_launches() == ([0, 1, 0, 0] if several else [n, 0, 0, 0])
    _one_by_one(B, dt, n)
    assert B.debug_launches() == [n, 0, 0, 0]
    _same(A, B)


from test_gpu_flow import CASES  # noqa: E402

SEVERAL = [c for c in CASES if c[1] != "br"] + [
    ("sheet, 28 rows", "fhn", (1, 900, 700), "none", 28, None, 9),
    ("isotropic block, 28 rows", "fhn", (21, 71, 130), "none", 28, None, 6),
    ("anisotropic block, 28 rows", "barkley", (33, 57, 65), "smooth", 28, None, 7),
    ("two columns, 28 rows", "zfk", (40, 29, 64), "none", 28, None, 5)]


@pytest.mark.parametrize("name,model,shape,fibres,ty,setup,n", SEVERAL, ids=[c[0] for c in SEVERAL])
def test_several_steps_a_launch_asked_for(bbx, name, model, shape, fibres, ty, setup, n):
    """The cases of several steps a launch, and tiles of 28 rows, whatever the grid's size chooses; mixed
    with launches of one step, whose totals are summed from another plan's pieces."""
    A, dt = _block(bbx, model, shape, fibres, ty, setup)
    B, _ = _block(bbx, model, shape, fibres, ty, setup)
    A.debug_route(bbx.BBX_ROUTE_SEVERAL)
    for m in (n, 1, n):  # the second call starts from the parity the first one left
        A.step(dt, m)
        _one_by_one(B, dt, m)
        _same(A, B)
    assert A.debug_launches()[:3] == [1 + 2 * (n % 64 == 1), 2 * (-(-n // 64)) - 2 * (n % 64 == 1), 0]


def test_captured_one_step_launches_between_calls_of_several(bbx):
    """A replay of captured one-step launches after a call of several steps leaves its own total."""
    torch = pytest.importorskip("torch")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        A, dt = _block(bbx, "barkley", (16, 64, 64), "rotational", 14)
        B, _ = _block(bbx, "barkley", (16, 64, 64), "rotational", 14)
        A.step(dt, 2)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            A.step(dt, 12)
        A.step(dt, 12)
        A.step(dt, 20)
        g.replay()
        s.synchronize()
        _one_by_one(B, dt, 46)
        s.synchronize()
        _same(A, B)
        assert A.debug_launches() == [2 + 12, 2, 0, 0]


@pytest.mark.parametrize("kind", ["sheet", "slab"])
def test_refused_launches_fall_back_to_one_launch_a_step(bbx, kind):
    def make():
        return (_sheet(bbx, 150, 120, "fhn"), 0.01) if kind == "sheet" else _block(bbx, "barkley", (16, 64, 64), "rotational", 14)

    (A, dt), (B, _) = make(), make()
    A.step(dt, 20)
    A.debug_refuse_launches(True)
    A.step(dt, 21)
    A.debug_refuse_launches(False)
    A.step(dt, 3)
    _one_by_one(B, dt, 44)
    _same(A, B)
    k = 2 if kind == "sheet" else 1
    assert A.debug_launches()[k] == 1 and sum(A.debug_launches()) == 25


def test_refused_batch_launches_fall_back(bbx):
    def make():
        gs = [_sheet(bbx, nx, ny, "fhn", seed=nx) for nx, ny in ((70, 33), (64, 129), (200, 17))]
        for g in gs:
            g.set_timestep(0.01)
        return gs, bbx.Batch(gs)

    (ga, A), (gb, B) = make(), make()
    ga[1].debug_refuse_launches(True)
    for n in (5, 130, 1, 18):
        A.step(n)
        for _ in range(n):
            B.step(1)
    A.sync()
    B.sync()
    for a, b in zip(ga, gb):
        _same(a, b)
        assert a.get_time()[1] == 154
    A.close()
    B.close()


@pytest.mark.parametrize("nx,ny,resident", [(200, 200, False), (500, 500, False), (64, 64, True), (2100, 12, True)])
def test_autotuning_times_the_tiles_of_a_resident_sheet(bbx, nx, ny, resident):
    """The resident kernels have no tiles: tuned with them, the height would be left to chance."""
    A = _sheet(bbx, nx, ny, "fhn")
    if resident:
        A.set_resident(True)
    st = A.read_all()
    assert A.autotune(0.01) > 0.0
    assert A.debug_launches() == [3 * (2 + 6), 0, 0, 0]
    assert np.array_equal(A.read_all(), st) and A.get_time() == (0.0, 0)
    A.step(0.01, 20)
    assert A.debug_launches()[0] == 24 and sum(A.debug_launches()) == 25


@pytest.mark.parametrize("model,aniso,heights", [("mrl", True, 2), ("fca", True, 2), ("mrl", False, 1), ("br", True, 1)])
def test_autotuning_of_tables_keeps_to_seven_rows_only_where_they_gather(bbx, model, aniso, heights):
    """Masked anisotropic grids of eleven variables gather table entries with 14 rows and not with 7."""
    from paper_1605_06015_gb300 import workloads as wl
    nx, ny, nz = 70, 20, 8
    mask, fib = wl.random_geometry(nx, ny, nz, 5, tissue_frac=0.7)
    G = bbx.Grid(nx, ny, nz, 0.2, mask)
    G.set_fibres(fib if aniso else None, 0.1, 0.025 if aniso else 0.1)
    G.set_ionic_model({"mrl": bbx.BBX_BR_MRL, "fca": bbx.BBX_BR_FCA, "br": bbx.BBX_BR}[model])
    if model == "br":
        G.set_tabulation(True)
    G.autotune(0.02)
    assert G.debug_launches() == [heights * 2 * (2 + 6), 0, 0, 0]  # two depths (4, 8)


@pytest.mark.parametrize("model", ["mrl", "fca"])
def test_gathered_entries_of_a_masked_anisotropic_grid(bbx, model):
    """14 rows (gathered) against 7 (each lane its own entries): the same entries, bitwise."""
    from paper_1605_06015_gb300 import workloads as wl
    nx, ny, nz = 130, 29, 5
    mask, fib = wl.random_geometry(nx, ny, nz, 6, tissue_frac=0.7)
    rng = np.random.default_rng(32)
    st = rng.uniform(0.0, 1.0, (11, nz, ny, nx)).astype(np.float32)
    st[0] = rng.uniform(-140.0, 100.0, (nz, ny, nx))  # (the table: -120 .. 80)
    st[1] = 10 ** rng.uniform(-7.2, -5.2, (nz, ny, nx))
    out = []
    for ty in (7, 14):
        G = bbx.Grid(nx, ny, nz, 0.2, mask)
        G.set_fibres(fib, 0.1, 0.025)
        G.set_tiling(ty, 4)
        G.set_ionic_model(bbx.BBX_BR_MRL if model == "mrl" else bbx.BBX_BR_FCA)
        G.write_all(st)
        G.step(0.02, 1)
        out.append(G.read_all()[:, mask != 0])
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("shape,fibres", [((16, 64, 64), "rotational"), ((20, 70, 66), "none"), ((1, 300, 200), "smooth"),
                                          ((130, 100, 90), "none")])
def test_autotuned_plans_of_one_and_of_several_steps(bbx, shape, fibres):
    """The two plans have tile rows of their own; calls that mix them give the results of one-step calls,
    the total of a call from its own plan's pieces, and settings changed in between reach both."""
    A, dt = _block(bbx, "barkley", shape, fibres, 14)
    B, _ = _block(bbx, "barkley", shape, fibres, 14)
    A.autotune(dt)
    for k, n in enumerate((64, 1, 70, 2)):
        if k == 2:
            for G in (A, B):
                G.set_stimulus((np.random.default_rng(8).random(shape) < 0.2).astype(np.uint8), 3.0, 0.0, 1.0)
                G.set_threshold(0.4)
        A.step(dt, n)
        _one_by_one(B, dt, n)
        _same(A, B)
    A.autotune(dt)
    A.set_scheme(1)
    B.set_scheme(1)
    A.step(dt, 24)
    _one_by_one(B, dt, 24)
    _same(A, B)
