"""The scratch of the FP64 leapfrog step: an allocator that refuses a large
buffer changes no bit of a result (the step works through a shorter ring of
slices), one that refuses two slices is an OOM at creation, and planes of any
size take the two passes that the plaquette choices name."""
import numpy as np
import pytest

import glasma_inputs as gi
from test_gpu_step_kernels import G  # noqa: F401

pytestmark = pytest.mark.gpu


def _allocator(G, monkeypatch, refuse):
    """Wrap the binding's allocator: request number k of `nbytes` is refused
    where refuse(k, nbytes) holds.  Returns the list of the sizes asked for."""
    inner, sizes = G._torch_allocator, []

    def wrapped():
        a, keep = inner()

        @G._ALLOC_FN
        def alloc(nbytes, stream, user):
            sizes.append(int(nbytes))
            if refuse(len(sizes) - 1, int(nbytes)):
                return None
            return keep[0](nbytes, stream, user)
        a.alloc = alloc
        return a, keep + (alloc,)
    monkeypatch.setattr(G, "_torch_allocator", wrapped)
    return sizes


def _run(G, cfg):
    h = G.glasma_init_mv(cfg, None)
    G.glasma_step(h, 7)
    out = list(G.glasma_get_fields(h)[:4]) + [G.glasma_tmunu(h)[0]]
    G.glasma_free(h)
    return out


@pytest.mark.parametrize("nc", [2, 3])
def test_a_refused_large_scratch_changes_no_bit(G, monkeypatch, nc):
    cfg = gi.small_config(nc, nz=47, nx=9, ny=11, sigma_l=2.0)
    ref = _run(G, cfg)
    links = 47 * 9 * 11 * 3 * (4 if nc == 2 else 18) * 8
    sizes = _allocator(G, monkeypatch, lambda k, n: n > 1.05 * links)
    got = _run(G, cfg)
    assert max(sizes) > 1.05 * links        # something was refused
    for x, y in zip(ref, got):
        assert np.array_equal(x, y)


def test_no_scratch_at_all_is_an_oom_and_leaves_nothing(G, monkeypatch):
    cfg = gi.small_config(2)
    sizes = _allocator(G, monkeypatch, lambda k, n: False)
    G.glasma_free(G.glasma_init_mv(cfg, None))
    n, live = len(sizes), dict(G._live_blocks)
    two = 2 * cfg["nx"] * cfg["ny"] * (9 * 3 + 3) * 8
    monkeypatch.undo()
    sizes = _allocator(G, monkeypatch, lambda k, size: k >= n - 1)
    with pytest.raises(G.GlasmaError) as e:
        G.glasma_init_mv(cfg, None)
    assert e.value.code == "OOM"
    assert sizes[-1] == two                 # down to two slices
    assert G._live_blocks == live


def test_planes_of_any_size_take_the_two_passes(G):
    """Two slices of this plane's scratch are 540 MB."""
    cfg = dict(gi.small_config(3), nz=5, nx=150, ny=3000, a_z=0.5, dt=0.25,
               sigma_l=0.05, z_offset=0.3, g2mu=0.05)
    tabs, launches = {}, {}
    for kernel in ("plaquette", "auto", "staple"):
        h = G.glasma_init_mv(cfg, None)
        G.glasma_set_step_kernel(h, kernel)
        G.glasma_step(h, 1)
        launches[kernel] = G.glasma_get_info(h).kernel_launches
        tabs[kernel] = G.glasma_tmunu(h)[0]
        G.glasma_free(h)
    assert launches["plaquette"] == launches["auto"] >= 2 and launches["staple"] == 1
    assert np.array_equal(tabs["plaquette"], tabs["auto"])
    assert np.max(np.abs(tabs["auto"] - tabs["staple"])) <= 1e-11 * np.max(np.abs(tabs["staple"]))


def test_gradient_holds_a_checkpoint_per_recomputed_segment(G, monkeypatch):
    """Seven steps in segments of three: buffers of the links' size are the
    context's two, the checkpoints of the first two segments, four states of a
    segment, the final state and the links' adjoints."""
    cfg = dict(gi.small_config(2, nz=48, nx=5, ny=7, sigma_l=2.0))
    sizes = _allocator(G, monkeypatch, lambda k, n: False)
    G.glasma_adjoint_energy(cfg, None, 7, 4.0, checkpoint_every=3)
    assert sizes.count(96 * 48 * 5 * 7) == 2 + 2 + 4 + 1 + 1
