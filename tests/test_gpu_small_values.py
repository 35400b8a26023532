"""Fields far below one: modes of 2^-790 to 2^-915 (10^-238 to 10^-275), alone in a
field and beside modes of ordinary size, with real coefficients, so that many of a
transform's results are exactly zero.  A fixed-point line keeps its own scale at
any size down to 2^-927: values, coefficients and a few steps come out finite and
as accurate as at ordinary sizes.

Tolerances: round trips 1e-13 of the field's largest value (lines of at most 64
points: three transforms each way of at most 2^-60 64^1.5 = 2^-51 of it); right-hand
sides 1e-12 of their largest products and steps 1e-11 per step of the field's
largest coefficient, as elsewhere."""
import numpy as np
import pytest

import ptt_inputs as I
from oracle import ptt2d as O2
from oracle import ptt3d as O3

pytestmark = pytest.mark.gpu

EXPONENTS = [-790, -815, -840, -846, -860, -915]
KW = dict(I.PAPER, dt=I.DT)


def _P():
    import paper_2606_09468_gb300 as P
    P.load_library()
    return P


def _tiny2(nx, ny, seed, e):
    a = I.random_spectral(nx, ny, seed=seed, decay=0.1).real.astype(complex)
    a[0] = 0.0
    return a * 2.0 ** e


@pytest.mark.parametrize("e", EXPONENTS)
def test_state_round_trip_2d(e):
    P, (nx, ny) = _P(), (32, 33)
    ora = O2.Channel2D(O2.Params(nx=nx, ny=ny, **KW))
    big = I.random_spectral(nx, ny, seed=2, decay=0.1)
    spec = [_tiny2(nx, ny, 3, e), _tiny2(nx, ny, 4, e), big + _tiny2(nx, ny, 5, e), _tiny2(nx, ny, 6, e),
            np.zeros_like(big)]
    spec[0][0] = big[0]                  # an ordinary mean over tiny modes
    ctx = P.Context([P.make_params(nx=nx, ny=ny, **KW)])
    ctx.set_spectral(0, I.spectral_to_abi(spec))
    assert ctx.diagnostics(0)[-1]["status"] == 0
    phys = I.abi_to_phys(ctx.get_state(0))
    for f in range(5):
        ref = ora.unpadded_phys(spec[f])
        assert np.max(np.abs(phys[f] - ref)) <= 1e-13 * np.max(np.abs(ref)), f
    ctx.set_state(0, I.phys_to_abi(phys))
    back = I.abi_to_spectral(ctx.get_spectral(0))
    for f in range(5):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-13 * np.max(np.abs(phys[f])), f


@pytest.mark.parametrize("e", EXPONENTS)
def test_state_round_trip_3d(e):
    P, (nx, ny, nz) = _P(), (16, 17, 8)
    kw = dict(KW, lz=5.0)
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    spec = []
    for f in range(9):
        a = I.random_spectral3(nx, ny, nz, seed=20 + f, decay=0.2).real.astype(complex)
        a[0] = 0.0                       # the mx = 0 plane is Hermitian in z: left out
        spec.append(a * (2.0 ** e if f % 2 else 1.0))
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, **kw)])
    ctx.set_spectral(0, I.spectral3_to_abi(spec))
    phys = I.abi_to_phys3(ctx.get_state(0))
    for f in range(9):
        ref = ora.unpadded_phys(spec[f])
        assert np.max(np.abs(phys[f] - ref)) <= 1e-13 * np.max(np.abs(ref)), f
    ctx.set_state(0, I.phys3_to_abi(phys))
    back = I.abi_to_spectral3(ctx.get_spectral(0))
    for f in range(9):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-13 * np.max(np.abs(phys[f])), f


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("e", EXPONENTS)
def test_steps_2d(e, form):
    """The laminar channel with tiny modes of v and c_xy: the right-hand side and
    three steps against the oracle (mixed: finite and not blown up)."""
    P, (nx, ny) = _P(), (32, 33)
    ora = O2.Channel2D(O2.Params(nx=nx, ny=ny, **KW))
    ora.init_state(0, 0.0)
    ora.state.v = ora.state.v + _tiny2(nx, ny, 4, e)
    ora.state.cxy = ora.state.cxy + _tiny2(nx, ny, 6, e)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, precision=getattr(P, "PTT_" + form.upper()), **KW)])
    ctx.set_spectral(0, I.spectral_to_abi(ora.state.as_list()))
    got = I.abi_to_spectral(ctx.explicit_rhs(0))
    assert all(np.all(np.isfinite(a)) for a in got)
    if form == "fp64":
        # the laminar products nearly cancel: measured by the relaxation term c rw
        phys = ora.get_physical()
        rw = (1.0 + KW["eps"] * np.max(phys[2])) / KW["wi"]
        ref = ora.explicit_terms(ora.state)
        scale = [np.max(np.abs(c)) * rw for c in phys[2:]] + [np.max(np.abs(ref[3]))]
        for f in range(4):               # H_y has no mean part to measure by
            assert np.max(np.abs(got[f] - ref[f])) <= 1e-12 * scale[f], f
    ctx.step(3)
    assert ctx.synchronize() == 0
    out = I.abi_to_spectral(ctx.get_spectral(0))
    assert all(np.all(np.isfinite(a)) for a in out)
    if form == "fp64":
        for _ in range(3):
            ora.step()
        for f, a in enumerate(ora.state.as_list()):
            if f != 1:
                assert np.max(np.abs(out[f] - a)) <= 3e-11 * np.max(np.abs(a)), f


@pytest.mark.parametrize("e", EXPONENTS)
def test_steps_3d(e):
    P, (nx, ny, nz) = _P(), (16, 17, 8)
    kw = dict(KW, lz=5.0)
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    ora.init_state(0, 0.0)
    for name, seed in (("v", 24), ("w", 25), ("cxz", 26)):
        a = I.random_spectral3(nx, ny, nz, seed=seed, decay=0.2).real.astype(complex)
        a[0] = 0.0
        setattr(ora.state, name, getattr(ora.state, name) + a * 2.0 ** e)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, **kw)])
    ctx.set_spectral(0, I.spectral3_to_abi(ora.state.as_list()))
    assert np.all(np.isfinite(ctx.explicit_rhs(0)))
    ctx.step(3)
    assert ctx.synchronize() == 0
    out = I.abi_to_spectral3(ctx.get_spectral(0))
    assert all(np.all(np.isfinite(a)) for a in out)
    for _ in range(3):
        ora.step()
    ref = ora.state.as_list()
    for f in (0, 3, 4, 6, 8):            # u, c_xx, c_xy, c_yy, c_zz: the laminar fields
        assert np.max(np.abs(out[f] - ref[f])) <= 3e-11 * np.max(np.abs(ref[f])), f
