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
