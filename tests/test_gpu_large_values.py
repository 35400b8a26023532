"""Fields far above one: sizes of 2^985 to 2^1005 (10^296 to 10^302), where the sums of
a line's moduli stay below 2^1018, go through the state round trips like ordinary ones;
a line beyond the range, or with an infinity, is NaN and nothing else is.

Tolerances: 1e-13 of the field's largest value (see test_gpu_small_values.py)."""
import numpy as np
import pytest

import ptt_inputs as I
from oracle import ptt2d as O2
from oracle import ptt3d as O3

pytestmark = pytest.mark.gpu

KW = dict(I.PAPER, dt=I.DT)


def _P():
    import paper_2606_09468_gb300 as P
    P.load_library()
    return P


@pytest.mark.parametrize("e", [985, 992, 1005])
def test_state_round_trip_2d(e):
    P, (nx, ny) = _P(), (32, 33)
    ora = O2.Channel2D(O2.Params(nx=nx, ny=ny, **KW))
    spec = [I.random_spectral(nx, ny, seed=40 + f, decay=0.2) * (2.0 ** e if f in (1, 3) else 1.0) for f in range(5)]
    ctx = P.Context([P.make_params(nx=nx, ny=ny, **KW)])
    ctx.set_spectral(0, I.spectral_to_abi(spec))
    phys = I.abi_to_phys(ctx.get_state(0))
    for f in range(5):
        ref = ora.unpadded_phys(spec[f])
        assert np.max(np.abs(phys[f] - ref)) <= 1e-13 * np.max(np.abs(ref)), f
    ctx.set_state(0, I.phys_to_abi(phys))
    back = I.abi_to_spectral(ctx.get_spectral(0))
    for f in range(5):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-13 * np.max(np.abs(phys[f])), f


@pytest.mark.parametrize("e", [985, 992, 1005])
def test_state_round_trip_3d(e):
    P, (nx, ny, nz) = _P(), (16, 17, 8)
    kw = dict(KW, lz=5.0)
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    spec = [I.random_spectral3(nx, ny, nz, seed=40 + f, decay=0.3) * (2.0 ** e if f % 2 else 1.0) for f in range(9)]
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


@pytest.mark.parametrize("value", [1.5e308, np.inf, -np.inf, np.nan])
def test_beyond_the_range_is_nan(value):
    """u at one point beyond the range: the member's u is NaN and the run is blown
    up; v, beside u in the same lines, keeps its values."""
    P, (nx, ny) = _P(), (32, 33)
    ora = O2.Channel2D(O2.Params(nx=nx, ny=ny, **KW))
    spec = [I.random_spectral(nx, ny, seed=40 + f, decay=0.2) for f in range(5)]
    phys = [ora.unpadded_phys(a) for a in spec]
    phys[0][3, 5] = value
    ctx = P.Context([P.make_params(nx=nx, ny=ny, **KW)])
    ctx.set_state(0, I.phys_to_abi(phys))
    assert ctx.diagnostics(0)[-1]["status"] == P.PTT_BLOWUP
    back = I.abi_to_spectral(ctx.get_spectral(0))
    assert not np.any(np.isfinite(back[0]))
    for f in range(1, 5):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-13 * np.max(np.abs(phys[f])), f
