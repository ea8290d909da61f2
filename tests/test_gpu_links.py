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


def _implicit_ctx(G, st, precision):
    p = st.p
    h = G.glasma_init_mv(dict(nc=p.nc, nz=p.nz, nx=p.nx, ny=p.ny, a_t=1.0, a_z=p.a_z, dt=p.dt,
                              sigma_l=0.05, z_offset=0.3, g2mu=0.0, m_ir=0.2, seed=0,
                              precision=precision, scheme="implicit", implicit_max_iter=80,
                              implicit_tol=1e-13 if precision == "fp64" else 1e-7), None)
    G.glasma_set_fields(h, st.U, st.E, st.QA, st.QB, st.U_prev, st.n)
    return h


def _errors(got, ref):
    return [float(np.max(np.abs(a - b)) / np.max(np.abs(b))) for a, b in zip(got, ref)]


# SU(2) takes the one-thread-per-site kernel from 3 * 2^16 sites on, SU(3) the
# staged one for rows of 64
@pytest.mark.parametrize("nc,shape,kernel", [
    (2, (9, 7, 10), "auto"), (2, (49, 64, 63), "auto"), (3, (9, 7, 10), "auto"), (3, (9, 3, 64), "auto"),
    (3, (9, 7, 10), "plaquette"), (2, (9, 7, 10), "staple_pairs"), (3, (9, 3, 64), "staple_staged")])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_steps_multiply_links_as_they_are(G, precision, nc, shape, kernel):
    """The force and the hop of links up to 5 % off the group, against the
    oracle, which multiplies matrices.  FP64: the whole state after three steps
    (1e-11).  FP32 steps put the links back on the group: the fields and charges
    after the first one (1.5e-6, the bound of the random-state tests), and T^{mu
    nu} before it (1e-5, that of the FP32 table tests)."""
    if precision == "fp64" and (kernel.startswith("staple") or shape[0] > 40):
        pytest.skip("an FP32 kernel")
    st = _off_group(_random_state(nc, *shape, seed=5 + nc), 0.05)
    h = _ctx(G, st, precision)
    G.glasma_set_step_kernel(h, kernel)
    tab, _ = G.glasma_tmunu(h)
    tol = 1e-11 if precision == "fp64" else 1e-5
    assert _errors([tab], [O.tmunu(st)[0]])[0] <= tol
    if precision == "fp64":
        G.glasma_step(h, 3)
        ref = O.step(st, 3)
        errs = _errors(G.glasma_get_fields(h)[:4], (ref.U, ref.E, ref.QA, ref.QB))
    else:
        G.glasma_step(h, 1)
        ref = O.step(st, 1)
        errs = _errors(G.glasma_get_fields(h)[1:4], (ref.E, ref.QA, ref.QB))
        tol = 1.5e-6
    assert all(e <= tol for e in errs), errs
    G.glasma_free(h)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nc", [2, 3])
def test_improved_steps_multiply_links_as_they_are(G, nc, precision):
    """The same through the improved scheme, whose U(t_{n-1}) is off the group
    too: FP64 the whole state after two steps; FP32, whose iterates are put back
    on the group, the charges after one, which see the links at t_n alone."""
    st = _off_group(_random_state(nc, 9, 6, 7, seed=8 + nc), 0.05 if precision == "fp64" else 1e-3)
    st.U_prev = st.U.copy()
    h = _implicit_ctx(G, st, precision)
    n = 2 if precision == "fp64" else 1
    G.glasma_step(h, n)
    ref = O.step_implicit(st, n, tol=1e-13)
    got = G.glasma_get_fields(h)
    if precision == "fp64":
        errs = _errors(got[:4], (ref.U, ref.E, ref.QA, ref.QB))
        assert all(e <= 1e-11 for e in errs), errs
    else:
        errs = _errors(got[2:4], (ref.QA, ref.QB))
        assert all(e <= 1.5e-6 for e in errs), errs


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nc", [2, 3])
def test_batches_and_states_keep_links_off_the_group(G, nc, precision):
    """A batch steps such an event as glasma_step does, beside one that is on
    the group, and a restored state is stepped as the state it was saved from;
    a state that an evolution has made is stepped on by the same kernel."""
    on = _random_state(nc, 9, 7, 10, seed=21)
    off = _off_group(_random_state(nc, 9, 7, 10, seed=22), 0.05)
    single = [_ctx(G, s, precision) for s in (on, off)]
    batched = [_ctx(G, s, precision) for s in (on, off)]
    saved = _ctx(G, on, precision)
    G.glasma_set_state(saved, G.glasma_get_state(single[1]))
    b = G.glasma_batch_create(batched)
    G.glasma_batch_tune(b, 1)
    G.glasma_batch_set_shape(b, "graph" if precision == "fp32" else "per_event", 32)
    G.glasma_batch_step(b, 1)
    G.glasma_batch_step(b, 2)
    for h in single:
        G.glasma_step(h, 2)
    again = _ctx(G, off, precision)
    G.glasma_set_state(again, G.glasma_get_state(single[0]))
    for h in single + [again]:
        G.glasma_step(h, 1)
    G.glasma_step(saved, 3)
    for h1, h2 in ((single[0], batched[0]), (single[1], batched[1]), (single[1], saved), (single[0], again)):
        for x, y in zip(G.glasma_get_fields(h1)[:4], G.glasma_get_fields(h2)[:4]):
            assert np.array_equal(x, y)
    b.close()
