"""Links that are not in SU(N): those of an FP32 state, which are unitary to
their rounding, and those that a caller sets off the group.  What a call
documents as products of the links holds for the links as they are."""
import numpy as np
import pytest

from oracle import glasma_oracle as O
from test_gpu_step_kernels import G, _ctx, _random_state  # noqa: F401
from test_zz_no_alloc import _device_layout

pytestmark = pytest.mark.gpu


def _off_group(st, amplitude, seed=3):
    """The links of a state moved off the group: SU(2) links (kept as real
    quaternions) by factors of their own, SU(3) links by any matrices."""
    rng = np.random.default_rng(seed)
    U, nz = st.U, st.p.nz
    if st.p.nc == 2:
        U *= 1.0 + amplitude * rng.uniform(-1.0, 1.0, U.shape[:-2])[..., None, None]
    else:
        U += amplitude * (rng.uniform(-1.0, 1.0, U.shape) + 1j * rng.uniform(-1.0, 1.0, U.shape))
    U[2][nz - 1] = np.eye(st.p.nc)
    return st


@pytest.mark.parametrize("amplitude", [0.0, 1e-5, 0.05])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nc", [2, 3])
def test_gauss_residual_holds_for_any_links(G, nc, precision, amplitude):
    """FP64 arithmetic on the stored values: 1e-13 of the largest entry."""
    import torch
    st = _off_group(_random_state(nc, 9, 7, 10, seed=nc), amplitude)
    h = _ctx(G, st, precision)
    U, E, QA, QB, n = G.glasma_get_fields(h)    # as they are stored
    ref = O.gauss_residual(O.State(st.p, U, E, QA, QB, n, U))
    got = [G.glasma_gauss_residual(h)]
    p = h.params
    u, e, qa, qb = _device_layout(G, h, torch.float64 if precision == "fp64" else torch.float32)
    got.append(G.glasma_gauss_residual_static(
        nc, precision, p.nz, p.ny, p.nx, p.a_t, p.a_z, u.data_ptr(), e.data_ptr(),
        qa.data_ptr(), 0, p.nz, qb.data_ptr(), 0, p.nz))
    for g in got:
        assert all(abs(a - b) <= 1e-13 * ref[0] for a, b in zip(g, ref)), (g, ref)
