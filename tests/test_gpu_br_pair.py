"""The Beeler-Reuter update of a pair of nodes over the whole range of V: the
removable singularities (V = -47 of the m gate, V = -23 of I_K1) and the ends
of their series, the limits beyond which the per-node formulas take over
(V = -140, V = 120, dt = 0.19), against the FP64 oracle without diffusion."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_06015_gb300 import bbx as b
    return b


@pytest.mark.parametrize("dt", [0.02, 0.19, 0.2])
def test_one_step_over_the_range_of_V(bbx, dt):
    nx, ny, nz = 66, 20, 4
    rng = np.random.default_rng(4)
    near = [c + s * e for c in (-47.0, -23.0) for s in (-1, 1) for e in (0.0, 1e-4, 0.3, 2.4999, 2.5001, 6.2499, 6.2501)]
    V = rng.uniform(-150.0, 130.0, (nz, ny, nx))
    flat = V.reshape(-1)
    flat[: len(near)] = near
    flat[100:104] = [-140.0, -139.99, 119.99, 120.0]
    st = np.empty((8, nz, ny, nx))
    st[0] = V
    st[1] = 10 ** rng.uniform(-7.2, -5.2, V.shape)
    st[2:] = rng.uniform(0.0, 1.0, (6,) + V.shape)
    st = st.astype(np.float32)
    og = oracle.Grid(nx, ny, nz, 1.0, None, None, 0.0, 0.0)
    osim = oracle.Sim(og, oracle.BR, state=st.astype(np.float64))
    osim.step(dt, 1)
    G = bbx.Grid(nx, ny, nz, 1.0)
    G.set_fibres(None, 0.0, 0.0)
    G.set_ionic_model(bbx.BBX_BR)
    G.write_all(st)
    G.step(dt, 1)
    got = G.read_all()
    # a rounding of the result, and 2e-5 of the increment: the exponentials' arguments reach 40 (a
    # relative error of 40 x 2^-24 = 2.4e-6 each, up to four in a current or a rate), the special-function
    # unit's 2^-22 each, and the currents' partial sums exceed the sum itself a few times); a gate next to
    # its steady state y_inf = alpha / (alpha + beta) moves little, but y_inf itself is uncertain by
    # y_inf (1 - y_inf) times the two rates' relative errors: 1/4 (2.4e-6 + 2.4e-6)
    for v in range(8):
        ref = osim.state[v]
        inc = np.abs(ref - st[v])
        scale = inc if v else np.maximum(inc, dt * 10.0)  # (V: currents of opposite sign)
        assert (np.abs(got[v] - ref) <= 1.2e-7 * np.maximum(np.abs(ref), np.abs(st[v])) + 2e-5 * scale + (1.2e-6 if v >= 2 else 1e-13)).all(), v
