"""The 3D energy with all of it in the last stored mode of every row of the sum
(largest kx, kz index nz - 1), on shapes whose nx/2 nz is no power of two and whose
Me nx/2 nz indices times it pass 2^32: each row must take its own quadrature weight.

Expected: E = (1/2) sum over modes (twice, for +-kx) of (1/2) int |u_m(y)|^2 dy with
int T_a T_b dy in closed form; FP64 sums of a few hundred terms, 1e-12 relative (the
mixed form transforms in FP32: 1e-5)."""
import numpy as np
import pytest

import ptt_inputs as I

pytestmark = pytest.mark.gpu


def _overlap(a, b):
    """int_{-1}^{1} T_a T_b dy."""
    return sum(1.0 / (1.0 - n * n) for n in (a + b, abs(a - b))) if (a + b) % 2 == 0 else 0.0


@pytest.mark.parametrize("form,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("nx,ny,nz", [(32, 33, 504), (150, 129, 90), (250, 65, 182)])
def test_energy_of_the_last_mode(nx, ny, nz, form, tol):
    import paper_2606_09468_gb300 as P
    P.load_library()
    spec = np.zeros((9, ny, nx // 2, nz, 2))
    deg = [0, 3, 10, ny - 1]
    coef = np.array([[0.7, -0.2], [0.3, 0.5], [-0.4, 0.1], [0.05, 0.02]])
    for f, s in enumerate((1.0, 0.5, -0.25)):
        spec[f, deg, nx // 2 - 1, nz - 1] = s * coef
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, lz=5.0, dt=I.DT, precision=getattr(P, "PTT_" + form.upper()),
                                   **I.PAPER)])
    ctx.set_spectral(0, spec)
    c = coef[:, 0] + 1j * coef[:, 1]
    q = sum((c[i] * np.conj(c[j])).real * _overlap(deg[i], deg[j]) for i in range(4) for j in range(4))
    ref = 0.5 * 2.0 * 0.5 * q * (1.0 + 0.25 + 0.0625)
    got = ctx.diagnostics(0)[-1]["energy"]
    assert abs(got - ref) <= tol * ref, (got, ref)
