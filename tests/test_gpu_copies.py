"""Copies between dense arrays and the padded layout: rows of every length class (multiples of 16, 8,
4 and 2 bytes), dense arrays that start off a 16-byte boundary, rows longer than a warp's unrolled
pass, and zeros in every cell of a coefficient array outside the interior."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 8, 31, 130, 516, 1027])
@pytest.mark.parametrize("dt,cdt", [("float32", "float32"), ("float32", "bfloat16"), ("float64", "float64")])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_coefficients_and_field_land_in_the_padded_arrays(nx, dt, cdt, off):
    import torch
    from paper_1410_5561_gb300.stencil import Stencil
    ny, nz = 11, 3
    s = Stencil("7pt_var", nx, ny, nz, dtype=getattr(torch, dt), coef_dtype=getattr(torch, cdt))
    n = nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(nx)
    pool = torch.rand(8 * (n + 8), generator=g, device="cuda", dtype=torch.float64)
    arrs = [pool.to(s.coef_dtype)[m * (n + 8) + off:][:n].view(nz, ny, nx) for m in range(7)]
    u = pool.to(s.dtype)[7 * (n + 8) + off:][:n].view(nz, ny, nx)
    for c in s.coefs:
        c.fill_(9.0)
    n0 = s.launches
    s.set_coeffs(arrays=arrs)
    assert s.launches == n0 + 1
    s.set_field(u, halo=0.5)
    torch.cuda.synchronize()
    for m in range(7):
        assert torch.equal(s.coef_interior(m), arrs[m])
        s.coef_interior(m).zero_()
        assert not bool(s.coefs[m].any())
    assert torch.equal(s.current, u)
    out = torch.empty(n + 8, dtype=s.dtype, device="cuda")[off:][:n].view(nz, ny, nx)
    assert torch.equal(s.get_field(out), u)
    s.current.fill_(0.5)
    assert bool((s.fields[0] == 0.5).all())


@pytest.mark.parametrize("shape", [(70001, 1, 1), (40000, 2, 1), (9001, 5, 3), (130004, 8, 1)])
@pytest.mark.parametrize("dt,cdt", [("float32", "float32"), ("float32", "bfloat16"), ("float64", "float64")])
def test_long_rows_are_copied_in_segments(shape, dt, cdt):
    import torch
    from paper_1410_5561_gb300.stencil import Stencil
    nx, ny, nz = shape
    s = Stencil("7pt_var", nx, ny, nz, dtype=getattr(torch, dt), coef_dtype=getattr(torch, cdt))
    g = torch.Generator(device="cuda").manual_seed(nx)
    arrs = [torch.rand(nz, ny, nx, generator=g, device="cuda").to(s.coef_dtype) for _ in range(7)]
    u = torch.rand(nz, ny, nx, generator=g, device="cuda", dtype=s.dtype)
    for c in s.coefs:
        c.fill_(9.0)
    s.set_coeffs(arrays=arrs)
    s.set_field(u, halo=0.5)
    for m in range(7):
        assert torch.equal(s.coef_interior(m), arrs[m])
        s.coef_interior(m).zero_()
        assert not bool(s.coefs[m].any())
    assert torch.equal(s.get_field(), u)
    s.current.fill_(0.5)
    assert bool((s.fields[0] == 0.5).all())
