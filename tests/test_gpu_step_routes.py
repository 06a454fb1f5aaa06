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
