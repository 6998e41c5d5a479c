"""Host-side pieces of the layered-strip glue: the closed-form backward of the least-squares
solve (strip.least_squares_grads), checked on the CPU with torch's own QR standing in for the
GPU factorisation (the GPU path is tested in test_gpu_linalg.py)."""
import pytest

torch = pytest.importorskip("torch")


class _HostLeastSquares(torch.autograd.Function):
    """x = argmin ||A x - b|| by torch.linalg.qr on the CPU, backward by least_squares_grads."""

    @staticmethod
    def forward(ctx, A, b):
        Q, R = torch.linalg.qr(A)
        x = torch.linalg.solve_triangular(R, (Q.conj().transpose(0, 1) @ b)[:, None], upper=True)[:, 0]
        ctx.save_for_backward(A, b, x, R)
        return x

    @staticmethod
    def backward(ctx, g):
        from paper_2103_12172_gb300.strip import least_squares_grads
        A, b, x, R = ctx.saved_tensors
        t = torch.linalg.solve_triangular(R.conj().transpose(0, 1), g[:, None], upper=False)
        w = torch.linalg.solve_triangular(R, t, upper=True)[:, 0]
        return least_squares_grads(A, b, x, w, lambda M, v: M @ v)


def test_least_squares_closed_form_gradient_passes_gradcheck():
    g = torch.Generator().manual_seed(0)
    A = torch.randn(40, 12, dtype=torch.complex128, generator=g)
    A[:, 3] *= 1e2                                   # unequal column scales
    b = torch.randn(40, dtype=torch.complex128, generator=g)
    x = _HostLeastSquares.apply(A, b)
    xr = torch.linalg.lstsq(A, b[:, None]).solution[:, 0]
    assert (x - xr).abs().max().item() <= 1e-12 * xr.abs().max().item()
    A.requires_grad_(True)
    b.requires_grad_(True)
    assert torch.autograd.gradcheck(lambda A, b: _HostLeastSquares.apply(A, b), (A, b), eps=1e-6, atol=1e-5)


def test_least_squares_refuses_host_tensors():
    """The product path has no CPU fallback: LeastSquares takes CUDA tensors only."""
    from paper_2103_12172_gb300.strip import LeastSquares
    A = torch.randn(8, 3, dtype=torch.complex128)
    with pytest.raises(TypeError):
        LeastSquares.apply(A, torch.randn(8, dtype=torch.complex128))


def test_boundary_coefficients_keep_their_64_bits():
    """alpha and beta of the outer sides as numbers beside tensors, and as numbers alone: exactly the doubles
    that the boundary condition returned (0.3 and 0.7 have no exact 32-bit form)."""
    from paper_2103_12172_gb300.strip import LayeredStrip
    lay = LayeredStrip.__new__(LayeredStrip)
    lay._consts = {}
    vals = [0.3, 0.7 + 0.1j, 2, torch.tensor(0.1, dtype=torch.float64), torch.tensor(0.2 - 0.6j, dtype=torch.complex128)]
    want = [0.3, 0.7 + 0.1j, 2.0, 0.1, 0.2 - 0.6j]
    assert lay._scalars(vals, torch.device("cpu")).tolist() == [complex(v) for v in want]
    assert lay._scalars(vals[:3], torch.device("cpu")).tolist() == [complex(v) for v in want[:3]]


def test_a_subclass_that_overrides_the_call_alone_is_asked_side_by_side():
    from paper_2103_12172_gb300.strip import _sides_at_once, incident_impedance_bc

    class Call(incident_impedance_bc):
        def __call__(self, j, side, kj, x, y):
            return 2.0, 1.0, x

    class Both(Call):
        def sides_at_once(self, ks, side, x, y):
            return ks, [1.0] * len(side), x

    class Deeper(Both):
        pass

    assert _sides_at_once(Call(0.3)) is None and _sides_at_once(lambda j, side, kj, x, y: (1.0, 1.0, x)) is None
    for cls in (incident_impedance_bc, Both, Deeper):
        bc = cls(0.3)
        assert _sides_at_once(bc) == bc.sides_at_once


def test_sides_at_once_follow_a_change_of_direction():
    from paper_2103_12172_gb300.strip import incident_impedance_bc
    bc, other = incident_impedance_bc(0.3), incident_impedance_bc(1.1)
    ks, x, y = torch.tensor([4.0, 5.0], dtype=torch.float64), torch.rand(2, 3).double(), torch.rand(2, 3).double()
    for _ in range(2):
        _, _, phi = bc.sides_at_once(ks, [1, 4], x, y)
        for i, side in enumerate((1, 4)):
            assert torch.allclose(phi[i], bc(0, side, ks[i], x[i], y[i])[2], rtol=1e-14, atol=0)
        bc.ct, bc.sn, bc.dirs = other.ct, other.sn, other.dirs


def test_incident_data_at_a_point_given_by_numbers():
    """x, y as numbers with a tensor wavenumber: as at a point given by tensors."""
    from paper_2103_12172_gb300.strip import incident_impedance_bc
    bc, k = incident_impedance_bc(0.3), torch.tensor(5.0, dtype=torch.float64)
    t = torch.tensor([0.25, 0.75], dtype=torch.float64)
    assert torch.allclose(bc(0, 2, k, 0.25, 0.75)[2], bc(0, 2, k, t[0], t[1])[2], rtol=1e-14, atol=0)
