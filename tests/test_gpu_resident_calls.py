"""Calls of several steps on small isotropic sheets, which run in one cluster's
registers and shared memory (k_resident_pairs), against calls of one step."""
import math

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


def _sheet(bbx, nx, ny, model, seed=1, lo=-0.2, hi=1.2):
    mid = {"fhn": bbx.BBX_FHN, "barkley": bbx.BBX_BARKLEY, "zfk": bbx.BBX_ZFK, "diffusion": bbx.BBX_DIFFUSION}[model]
    G = bbx.Grid(nx, ny, 1, 0.5)
    G.set_fibres(None, 1.0, 1.0)
    G.set_ionic_model(mid)
    st = np.random.default_rng(seed).uniform(lo, hi, (bbx.NVARS[mid], 1, ny, nx)).astype(np.float32)
    return G, st


@pytest.mark.parametrize("nx,ny", [(1, 16), (33, 31), (200, 200), (333, 257)])
def test_total_is_the_sum_of_the_state(bbx, nx, ny):
    """The sums of a thread, a warp and a block are kept in three floats (2^-70 of the sum of the
    magnitudes an addition); 2 + 5 + 16 additions in FP64 over a warp's three, the warps and the CTAs remain:
    2^-53 each."""
    G, st = _sheet(bbx, nx, ny, "diffusion", lo=-1e4, hi=1e4)
    G.write_all(st)
    G.step(0.01, 30)
    V = G.read_state(0).astype(np.float64).ravel()
    assert abs(G.step_total() - math.fsum(V)) <= 24 * 2.0 ** -53 * math.fsum(np.abs(V))


@pytest.mark.parametrize("nx,ny,model,n", [(33, 31, "fhn", 4), (100, 90, "barkley", 7), (199, 201, "zfk", 20), (300, 300, "fhn", 31),
                                           (200, 200, "diffusion", 8), (511, 333, "fhn", 100)])
def test_other_buffer_holds_the_state_before_the_last_step(bbx, nx, ny, model, n):
    """A program that owns both buffers finds in them the last two states, as after n calls of one
    step, and its values beside the rows are left alone."""
    import torch
    got = []
    for one in (False, True):
        G, st = _sheet(bbx, nx, ny, model)
        px = G.get_info()["px"]
        bufs = [torch.full((st.shape[0], 1, ny, px), 7.0, device="cuda") for _ in range(2)]
        G.bind_state(*bufs)
        G.write_all(st)
        for b in bufs:
            b[..., nx:] = 7.0
        for _ in range(n if one else 1):
            G.step(0.01, 1 if one else n)
        G.step_total()
        cur = 0 if G.state_device_ptr(0) == bufs[0].data_ptr() else 1
        got.append([bufs[cur].cpu().numpy(), bufs[cur ^ 1].cpu().numpy()])
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("nx,ny,model", [(2100, 17, "fhn"), (2051, 40, "zfk"), (150, 12, "barkley"), (2100, 15, "fhn"), (7, 8, "diffusion")])
def test_sheets_in_shared_memory(bbx, nx, ny, model):
    """Sheets that the registers' kernel does not take (more than 2048 columns; 8 to 15 rows, a
    cluster of 8): the kernel in shared memory, to rounding as calls of one step."""
    A, st = _sheet(bbx, nx, ny, model)
    B, _ = _sheet(bbx, nx, ny, model)
    reg = (np.random.default_rng(2).random((1, ny, nx)) < 0.3).astype(np.uint8)
    for G in (A, B):
        G.write_all(st)
        G.set_threshold(0.5)
        G.set_stimulus(reg, 4.0, 0.015, 0.04)
    A.set_resident(True)
    for n in (7, 2, 4):
        A.step(0.01, n)
        for _ in range(n):
            B.step(0.01, 1)
    assert A.debug_launches() == [0, 0, 0, 3]
    a, b = A.read_all().astype(np.float64), B.read_all().astype(np.float64)
    # a rounding (2^-24 of 1.5) in each of some ten operations a step, 13 steps
    assert np.abs(a - b).max() <= 13 * 10 * 1.5 * 2.0 ** -24
    ta, tb = A.read_activation().astype(np.int64), B.read_activation().astype(np.int64)
    ta[ta == bbx.BBX_ACT_NONE] = tb[tb == bbx.BBX_ACT_NONE] = 14
    assert np.abs(ta - tb).max() <= 1 and (tb < 14).any()
    assert A.get_time() == B.get_time()
    assert abs(A.step_total() - a[0].sum()) <= 1e-12 * np.abs(a[0]).sum()
