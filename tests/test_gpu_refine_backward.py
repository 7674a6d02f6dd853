"""dP/dX of P(r, z) where the backward pass changes its quadrature rule (|z| about
33 and 111), at the widest window and at the ends of the spectrum.

P = |F|^2 with F = sum_k X_k conj(rho(r - k, z)), so its gradient is 2 F rho(r - k, z)
in FP64, rho being the sum over 512 quadrature nodes that fdas.h defines (the
integral itself up to |z| = 268; past it the two differ).  Tolerance: every rho in FP32 is off by at most 4e-6 (phases rounded to
2^-24 of a few turns, products of up to 16 steps), so F is by 4e-6 sum |X_k| and
an element by 2 (4e-6 sum |X_k| |rho_k| + 4e-6 |F|).
"""
import ctypes

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 1 << 13   # 4096 bins
POINTS = [(r, s * z) for z in (0.0, 32.9, 33.0, 33.1, 34.0, 110.9, 111.0, 111.1, 112.0, 267.0, 446.0)
          for s in (1, -1) for r in (2000.0, 2000.49, 2000.51)]
ENDS = [(r, z) for r in (0.0, 0.3, 40.7, 4054.2, 4095.0) for z in (0.0, -33.2, 90.5, -200.1)]


@pytest.mark.parametrize("points", [POINTS, ENDS])
def test_spectrum_gradient(points):
    import paper_2211_13517_gb300 as pkg
    pkg.build()
    from paper_2211_13517_gb300 import capi
    plan = capi.Plan(N, 64e-6, 16.0, 1.0, 1024, 4)
    n_r = N // 2
    rng = np.random.RandomState(3)
    X = (rng.standard_normal(n_r) + 1j * rng.standard_normal(n_r)).astype(np.complex64)
    spec = torch.view_as_real(torch.from_numpy(X).cuda())
    X = X.astype(np.complex128)
    for r, z in points:
        grad = torch.zeros((n_r, 2), dtype=torch.float32, device="cuda")
        grz = torch.empty((1, 2), dtype=torch.float64, device="cuda")
        rz = torch.tensor([[r, z]], dtype=torch.float64, device="cuda")
        g = torch.ones(1, dtype=torch.float32, device="cuda")
        capi.fdas_fourier_power_backward(
            plan.handle, ctypes.c_void_p(spec.data_ptr()), ctypes.c_void_p(rz.data_ptr()), 1,
            ctypes.c_void_p(g.data_ptr()), ctypes.c_void_p(grad.data_ptr()),
            ctypes.c_void_p(grz.data_ptr()))
        got = torch.view_as_complex(grad).cpu().numpy().astype(np.complex128)
        k = O.refine_window(r, z, n_r)
        rho = O.rho(r - k, z, n_nodes=512)
        F = np.sum(X[k] * np.conj(rho))
        size = 4e-6 * np.sum(np.abs(X[k]))
        bound = 2.0 * (size * np.abs(rho) + 4e-6 * abs(F) + 4e-6 * size)
        assert np.all(np.abs(got[k] - 2.0 * F * rho) <= bound), (r, z)
        got[k] = 0.0
        assert np.all(got == 0.0), (r, z)
    plan.close()
