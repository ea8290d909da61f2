"""The kernels that a context takes by its sizes and types, each at the edges
of its range and against the general path: the FP64 step in two passes (its
ring of slices wrapping, rows longer than a block, planes whose scratch holds
two slices), the FP32 SU(2) step with one thread per site (from 2^17 sites
on), T^{mu nu} of SU(2), the FP32 -> FP64 conversion of the observables, and the
kernels of a batch."""
import numpy as np
import pytest

import glasma_inputs as gi
from oracle import glasma_oracle as O
from test_gpu_slab import _compare, _run
from test_gpu_step_kernels import G, TOL64, _ctx, _random_state, rel  # noqa: F401

pytestmark = pytest.mark.gpu


def _step_both(G, st, precision, steps, tol):
    out = []
    for kernel in ("staple", "auto"):
        h = _ctx(G, st, precision)
        G.glasma_set_step_kernel(h, kernel)
        G.glasma_step(h, steps)
        out.append(G.glasma_get_fields(h)[:4])
        G.glasma_free(h)
    errs = [rel(b, a) for a, b in zip(*out)]
    assert all(e <= tol for e in errs), errs


@pytest.mark.parametrize("nc,shape", [
    (2, (40, 96, 96)), (3, (20, 96, 96)),   # 64 MB hold 32 and 12 slices: the ring wraps
    (2, (7, 3, 400)), (3, (6, 1, 513)),     # rows that the marching kernel does not take
    (3, (5, 256, 256)),                     # two slices of scratch, one per chunk
    (2, (9, 9, 7)), (3, (5, 1, 1))])        # a last block of 55, and of 5, threads
def test_fp64_two_passes_match_the_staple_form(G, nc, shape):
    """Two orders of the same FP64 sums over three steps: the FP64 target."""
    _step_both(G, _random_state(nc, *shape, seed=sum(shape) + nc), "fp64", 3, TOL64)


@pytest.mark.parametrize("shape", [
    (32, 64, 64), (140, 31, 31), (131, 1, 1001), (4099, 32, 1), (9, 121, 121)])
def test_su2_fp32_site_kernel_matches_the_staple_form(G, shape):
    """2^17 sites and a little more, with planes that end within a warp and
    planes of one row or column.  Each form stays within 1.5e-6 of the FP64
    step after three steps (the bound of the FP32 random-state test), so two
    of them within 3e-6 of one another."""
    _step_both(G, _random_state(2, *shape, seed=sum(shape)), "fp32", 3, 3e-6)


@pytest.mark.parametrize("nranks", [2, 3])
def test_su2_fp32_site_kernel_on_slabs(G, nranks):
    """The rule counts the whole lattice's sites, so slabs below 2^17 sites of
    a lattice above it take the same kernel: bitwise the whole lattice."""
    cfg = dict(gi.small_config(2, nz=47, nx=53, ny=54, sigma_l=2.0), precision="fp32")
    whole, ranks, T = _run(G, cfg, nranks, 44, "auto")
    _compare(G, cfg, whole, ranks, T)


@pytest.mark.parametrize("precision,tol", [("fp64", TOL64), ("fp32", 1e-5)])
@pytest.mark.parametrize("shape", [
    (6, 1, 1), (6, 1, 2), (7, 2, 1), (9, 17, 15), (6, 33, 67), (5, 3, 400)])
def test_su2_tmunu_matches_oracle(G, shape, precision, tol):
    """Slices below, at and above a block's 256 sites, and planes of one row
    or column.  FP32: each entry is a mean of products of at most eight
    rounded factors of O(1), 8 * 6e-8 absolute, against means of O(0.1)."""
    st = _random_state(2, *shape, seed=sum(shape))
    h = _ctx(G, st, precision)
    G.glasma_step(h, 1)
    tab, H = G.glasma_tmunu(h)
    rtab, rH = O.tmunu(O.step(st, 1))
    assert rel(tab, rtab) <= tol and abs(H - rH) <= tol * abs(rH)


@pytest.mark.parametrize("angle", [1e-4, 0.7, 3.0, 25.0])
@pytest.mark.parametrize("nc", [2, 3])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_link_update_at_any_angle(G, nc, angle, precision):
    """exp(-i dt E) by a short series for small |dt E| and by the closed form
    beyond, up to several turns.  FP32: E carries 6e-8 relative, so a link
    turns by the angle with an error of 6e-8 * angle, beside the rounding of
    the product; E itself, set by a force of O(1), is far below the angle's."""
    st = _random_state(nc, 7, 5, 9, seed=17)
    st.E *= angle / (st.p.dt * np.max(np.abs(st.E)))
    ref = O.step(st, 2)
    for kernel in ("auto", "staple"):
        h = _ctx(G, st, precision)
        G.glasma_set_step_kernel(h, kernel)
        G.glasma_step(h, 2)
        U, E = G.glasma_get_fields(h)[:2]
        tol = TOL64 if precision == "fp64" else 1.5e-6 * (1 + angle)
        assert rel(U, ref.U) <= tol and rel(E, ref.E) <= tol, kernel
        G.glasma_free(h)


@pytest.mark.parametrize("scale", [1.5e-45, 3e-40, 1.2e-38, 1.0, 1e30])
def test_fp32_fields_are_widened_exactly(G, scale):
    """The Gauss residual of FP32 fields on unit links is an FP64 sum of their
    exact values, denormals among them."""
    st = _random_state(2, 6, 5, 7, seed=3)
    st.U[:] = np.eye(2)
    rng = np.random.default_rng(5)
    st.E = (scale * rng.integers(-7, 8, st.E.shape)).astype(np.float32).astype(np.float64)
    st.E[2][st.p.nz - 1] = 0.0
    st.QA[:] = 0.0
    st.QB[:] = 0.0
    g = G.glasma_gauss_residual(_ctx(G, st, "fp32"))
    ref = O.gauss_residual(st)
    assert abs(g[0] - ref[0]) <= 1e-14 * ref[0]


@pytest.mark.parametrize("nc,precision,sizes,kernel", [
    (2, "fp64", [(48, 12, 10), (40, 16, 16)], "auto"),
    (3, "fp64", [(48, 12, 10), (56, 9, 5)], "auto"),
    (2, "fp32", [(40, 64, 64), (34, 64, 64)], "auto"),
    (2, "fp32", [(40, 64, 64), (40, 16, 16)], "staple"),
    (3, "fp32", [(48, 12, 10), (40, 64, 16)], "staple")])
def test_default_batch_takes_the_cheaper_kernel(G, nc, precision, sizes, kernel):
    """The events' own kernels where all of them do less arithmetic than the
    staple form, else the graph's staple form: bitwise the single steps."""
    cfgs = [dict(gi.small_config(nc, nz=nz, nx=nx, ny=ny, sigma_l=1.0, seed=60 + k),
                 precision=precision) for k, (nz, nx, ny) in enumerate(sizes)]
    batched = [G.glasma_init_mv(c, None) for c in cfgs]
    b = G.glasma_batch_create(batched)
    G.glasma_batch_step(b, 9)
    for c, h in zip(cfgs, batched):
        one = G.glasma_init_mv(c, None)
        G.glasma_set_step_kernel(one, kernel)
        G.glasma_step(one, 9)
        for x, y in zip(G.glasma_get_fields(one)[:4], G.glasma_get_fields(h)[:4]):
            assert np.array_equal(x, y)
    b.close()


# from 3 * 2^16 sites of FP32 SU(2) on one thread steps a site: planes of whole
# blocks, planes that end within a warp, planes of less than a block of 256, 64
# or 32 threads, and the longest lattices
SITE_SHAPES = [(48, 64, 64), (205, 31, 31), (197, 1, 1001), (6145, 32, 1), (14, 121, 121),
               (681, 17, 17), (1366, 12, 12), (65535, 1, 4)]


@pytest.mark.parametrize("shape", SITE_SHAPES)
def test_su2_fp32_site_kernel_in_blocks_of_any_size(G, shape):
    """Within 3e-6 of the staple form after three steps (each within 1.5e-6 of
    the FP64 step), and no kernel of the staple's bits."""
    st = _random_state(2, *shape, seed=sum(shape))
    out = []
    for kernel in ("staple", "auto"):
        h = _ctx(G, st, "fp32")
        G.glasma_set_step_kernel(h, kernel)
        G.glasma_step(h, 3)
        out.append(G.glasma_get_fields(h)[:4])
        G.glasma_free(h)
    assert all(rel(b, a) <= 3e-6 for a, b in zip(*out))
    assert not np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("nranks", [2, 3])
def test_su2_fp32_site_kernel_on_slabs_of_a_larger_lattice(G, nranks):
    """Slabs below the kernel's sites of a lattice above them: bitwise the
    whole lattice."""
    cfg = dict(gi.small_config(2, nz=71, nx=53, ny=54, sigma_l=2.0), precision="fp32")
    whole, ranks, T = _run(G, cfg, nranks, 44, "auto")
    _compare(G, cfg, whole, ranks, T)


@pytest.mark.parametrize("shape", [(65535, 1, 4), (6145, 32, 1), (4096, 8, 8), (768, 16, 17)])
def test_su2_fp32_site_kernel_fills_its_blocks_on_small_planes(G, shape):
    """The kernel that AUTO takes is no slower than the staple kernel where a
    plane is a part of a block of 256 (it was by up to 1.5 times)."""
    import torch
    st = _random_state(2, *shape, seed=1)
    st.QA[:] = 0.0
    st.QB[:] = 0.0
    best = {}
    for kernel in ("staple", "auto"):
        h = _ctx(G, st, "fp32")
        G.glasma_set_step_kernel(h, kernel)
        G.glasma_step(h, 100)
        times = []
        for _ in range(10):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            G.glasma_step(h, 200)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        best[kernel] = min(times)
        G.glasma_free(h)
    assert best["auto"] <= 1.1 * best["staple"], best


@pytest.mark.parametrize("nc,field", [(2, 3e18), (3, 3e18)])
def test_fp32_table_sums_beyond_the_range_of_fp32(G, nc, field):
    """T^{mu nu} adds up sites in FP64: squares of 1e38, of which an FP32 sum
    holds three, in slices of 4096 sites.  Products of two rounded factors,
    summed in FP64: 4 * 6e-8 of the entry."""
    st = _random_state(nc, 6, 64, 64, seed=1)
    st.U[:] = np.eye(nc)
    st.E[:] = field
    st.E[2][st.p.nz - 1] = 0.0
    st.QA[:] = 0.0
    st.QB[:] = 0.0
    tab, H = G.glasma_tmunu(_ctx(G, st, "fp32"))
    ref, rH = O.tmunu(st)
    assert np.max(np.abs(tab - ref)) <= 2.4e-7 * np.max(ref)
    assert abs(H - rH) <= 2.4e-7 * rH


@pytest.mark.parametrize("kernel,shape", [("staple", (40, 24, 20)), ("staple_staged", (20, 30, 32))])
def test_su3_fp32_error_of_two_steps(G, kernel, shape):
    """Two FP32 steps of generic links (exponents of 0.2, fields of 0.05) against
    the oracle's: the rms error of E is no more than with three rows of every
    product formed (2.484e-7 of the rms of E on 24 x 15 x 16, where one derived
    row alone gives 2.504e-7 and this arithmetic 2.446e-7; 19200 sites x 24
    components determine it to about a thousandth)."""
    nz, ny, nx = shape
    rng = np.random.default_rng(17)
    st = _random_state(3, *shape, seed=1)
    p = O.Params(nc=3, nz=nz, nx=nx, ny=ny, a_z=1.0, dt=0.5, sigma_l=1.0)
    st = O.State(p, st.U, st.E, 0.0 * st.QA, 0.0 * st.QB, 0, st.U)
    st.U[:] = O.expi_alg(0.2 * rng.standard_normal((3, nz, ny, nx, 8)), 1.0, 3)
    st.U[2][nz - 1] = np.eye(3)
    st.E[:] = 0.05 * rng.standard_normal(st.E.shape)
    st.E[2][nz - 1] = 0.0
    h = _ctx(G, st, "fp32")
    G.glasma_set_step_kernel(h, kernel)
    G.glasma_step(h, 2)
    E, ref = G.glasma_get_fields(h)[1], O.step(st, 2).E
    assert np.linalg.norm(E - ref) <= 2.484e-7 * np.linalg.norm(ref)


@pytest.mark.parametrize("angle", [1e-4, 0.7, 3.0, 25.0])
@pytest.mark.parametrize("nc,shape", [(2, (48, 64, 64)), (3, (9, 6, 64)), (3, (9, 6, 32))])
def test_link_update_at_any_angle_by_the_large_lattice_kernels(G, nc, shape, angle):
    """As test_link_update_at_any_angle, where AUTO is the one-thread-per-site
    kernel (its own exponential) and the staged kernel (rows of 64; of 32 it is
    asked for)."""
    st = _random_state(nc, *shape, seed=23)
    st.E *= angle / (st.p.dt * np.max(np.abs(st.E)))
    ref = O.step(st, 2)
    h = _ctx(G, st, "fp32")
    if shape[2] == 32:
        G.glasma_set_step_kernel(h, "staple_staged")
    G.glasma_step(h, 2)
    U, E = G.glasma_get_fields(h)[:2]
    tol = 1.5e-6 * (1 + angle)
    assert rel(U, ref.U) <= tol and rel(E, ref.E) <= tol


# 64 MB hold 32 (SU(2)) and 12 (SU(3)) slices of 96^2, and two of 256^2
@pytest.mark.parametrize("nc,shape", [(2, (40, 96, 96)), (3, (26, 96, 96)), (3, (5, 256, 256))])
def test_fp64_table_across_the_ring_of_the_two_passes(G, nc, shape):
    """eps, p_L, p_T and S_L of every slice from a scratch that holds a part of
    the lattice: the FP64 target."""
    st = _random_state(nc, *shape, seed=sum(shape))
    ref, rH = O.tmunu(st)
    tab, H = G.glasma_tmunu(_ctx(G, st, "fp64"))
    assert np.all(np.abs(tab - ref) <= TOL64 * np.max(np.abs(ref), axis=0))
    assert abs(H - rH) <= TOL64 * rH
