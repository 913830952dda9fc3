"""Overlapped-tile sweep against the plain sweep, bit for bit (the same operations on the same
operands in the same order), at the edges of its tiles: rows of one vector to several tiles, row
counts around the tile heights of the three instantiations, z chunks thinner and thicker than the
overlap, step counts with and without a remainder; and against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from tests._util import Problem, step_tol

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 5, 2), (4, 32, 7), (5, 33, 3), (124, 60, 9), (125, 61, 12), (128, 31, 40), (129, 17, 5),
          (248, 30, 11), (249, 44, 4), (252, 12, 26), (131, 13, 23), (376, 9, 8), (64, 89, 19)]
KINDS = [("7pt_const", None), ("7pt_var", None), ("7pt_var", "bf16")]


def _pair(kind, cdt, shape, T, chunks, seed=51):
    import torch
    from paper_1410_5561_gb300.stencil import Tuning
    p = Problem(kind, *shape, fdt="f32", cdt=cdt, seed=seed, halo=-0.625)
    a, b = p.make(), p.make()
    a.set_tuning("plain")
    b.set_tuning("overlap", Tuning(6, chunks, 0, 0))
    a.run(T)
    b.run(T)
    b.sync()
    assert a.parity == b.parity
    assert torch.equal(a.current, b.current)
    b.current.fill_(-0.625)  # what is left of the array is its halo, untouched
    assert bool((b.fields[b.parity] == -0.625).all())
    return p, a


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind,cdt", KINDS)
def test_overlap_is_bitwise_equal_to_plain(kind, cdt, shape):
    for chunks in (0, 1, min(3, shape[2])):
        _pair(kind, cdt, shape, 3, chunks)
    _pair(kind, cdt, shape, 7, 0)


@pytest.mark.parametrize("kind,cdt", KINDS)
def test_overlap_larger_grid_and_oracle(kind, cdt):
    T = 20
    p, a = _pair(kind, cdt, (301, 107, 75), T, 0)
    ref = p.oracle(T)
    got = a.get_field().double().cpu().numpy()
    assert oracle.step_normalised_l2(got, ref, T) <= step_tol("f32")
    assert np.max(np.abs(got - ref)) <= p.elementwise_tol(T)


def test_overlap_is_captured_in_a_graph():
    import torch
    p = Problem("7pt_var", 140, 50, 33, fdt="f32", seed=5, halo=0.25)
    a, b = p.make(), p.make()
    a.set_tuning("plain")
    b.set_tuning("overlap")
    g = b.capture(8)
    g.replay()
    g.replay()
    a.run(16)
    torch.cuda.synchronize()
    assert torch.equal(a.current, b.current)


def test_overlap_refuses_other_stencils():
    from paper_1410_5561_gb300.stencil import Stencil, Tuning
    import torch
    for kind, dt in (("25pt_var", torch.float32), ("7pt_const", torch.float64)):
        with pytest.raises(Exception):
            Stencil(kind, 20, 20, 20, dtype=dt).set_tuning("overlap")
    with pytest.raises(Exception):
        Stencil("7pt_const", 20, 20, 20).set_tuning("overlap", Tuning(6, 21, 0, 0))


@pytest.mark.parametrize("kind,cdt", KINDS)
def test_auto_grid_bound_again_without_a_workspace(kind, cdt):
    """A grid that STENCIL_AUTO gave overlapped tiles and that is then bound without a workspace runs
    what AUTO selects without one; the schedule asked for by name needs the workspace."""
    import ctypes
    from paper_1410_5561_gb300 import _lib as C
    p = Problem(kind, 45, 37, 23, fdt="f32", cdt=cdt, seed=8, halo=0.5)
    a, b, c = p.make(), p.make(), p.make()
    a.set_tuning("plain")
    b.set_tuning("auto")
    c.set_tuning("overlap")
    for s in (b, c):
        carr = (ctypes.c_void_p * 13)(*[x.data_ptr() for x in s.coefs])
        C.call("stencil_bind", s._h, ctypes.c_void_p(s.fields[0].data_ptr()), ctypes.c_void_p(s.fields[1].data_ptr()),
               carr if s.ncoef else None, None)
        s.set_field(p.torch_inputs("cuda")[0], halo=p.halo)
    a.run(7)
    b.run(7)
    assert np.array_equal(a.get_field().cpu().numpy(), b.get_field().cpu().numpy())
    with pytest.raises(C.StencilError):
        c.run(7)


@pytest.mark.parametrize("kind,cdt", KINDS)
@pytest.mark.parametrize("shape,T,launches", [
    ((70, 23, 19), 9, 1), ((70, 23, 19), 2, 2), ((70, 23, 19), 1, 1),   # no pass of three steps: plain steps
    ((1808, 30, 2), 3, 1), ((1809, 300, 2), 3, 3), ((1809, 20, 20), 3, 3), ((2000, 60, 12), 3, 1),
])
def test_auto_between_overlapped_tiles_and_plain_steps(kind, cdt, shape, T, launches):
    """AUTO runs plain steps where the overlapped tiles have nothing to share: fewer than three steps, and thin
    or small grids of long rows. The same bits either way."""
    p = Problem(kind, *shape, fdt="f32", cdt=cdt, seed=31, halo=0.25)
    a, b = p.make(), p.make()
    a.set_tuning("plain")
    b.set_tuning("auto")
    a.run(T)
    n0 = b.launches
    b.run(T)
    assert b.launches == n0 + launches
    assert a.parity == b.parity
    assert np.array_equal(a.get_field().cpu().numpy(), b.get_field().cpu().numpy())


@pytest.mark.parametrize("kind,cdt", KINDS)
def test_overlap_timeout_is_reported_not_hung(kind, cdt):
    """A tile made to wait on a flag that no tile sets, with a short wait limit, ends the launch with the
    status word set; a new field clears it and the next run is exact."""
    from paper_1410_5561_gb300._lib import STATUS, StencilError
    p = Problem(kind, 140, 64, 24, fdt="f32", cdt=cdt, seed=9)
    a, s = p.make(), p.make()
    a.set_tuning("plain")
    a.run(13)
    s.set_tuning("overlap")
    s.set_wait_limit(2000)
    s.inject_stall(5)
    s.run(13)
    assert STATUS[s.status()] == "STENCIL_ETIMEOUT"
    with pytest.raises(StencilError):
        s.sync()
    s.inject_stall(-1)
    s.set_wait_limit(1 << 24)
    s.set_field(p.torch_inputs("cuda")[0], halo=p.halo)
    s.run(13)
    assert s.status() == 0
    assert np.array_equal(s.get_field().cpu().numpy(), a.get_field().cpu().numpy())


def test_overlap_with_more_tiles_than_counters():
    """Chunks of four planes of a grid of 2^24 planes are more tiles than the workspace has counters for: the
    run is cut in two and takes plain steps."""
    import torch
    from paper_1410_5561_gb300.stencil import Stencil, Tuning
    nz = 1 << 24
    s = Stencil("7pt_const", 1, 1, nz)
    s.set_coeffs(scalars=(0.4, 0.1))
    u = torch.rand(nz, 1, 1, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    s.set_field(u, halo=0.25)
    s.run(7)
    ref = s.get_field().clone()
    s.set_field(u, halo=0.25)
    s.set_tuning("overlap", Tuning(6, nz, 0, 0))
    n0 = s.launches
    s.run(7)
    assert s.launches == n0 + 7 and s.parity == 1
    assert torch.equal(s.get_field(), ref)
