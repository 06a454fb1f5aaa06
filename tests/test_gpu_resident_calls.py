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
