"""State transforms and diagnostics where the y transforms are longest: ny whose
unpadded (2 (ny - 1)) or energy-grid (Me) FFT length takes radix-3 passes of more
than 256 butterflies (810, 882, 972, 990: ny = 401 to 496), and the largest, 513.

Tolerances are those of the shorter sizes: values and coefficients to 1e-12 of a
field's maximum (the oracle sums 500 terms per value with FP64 matrices, about
500 2^-53 = 6e-14, the library's transforms stay below 2^-45 = 3e-14), averages
and extrema to 1e-11, counts to the points in the tie bands."""
import numpy as np
import pytest

import ptt_inputs as I
from oracle import ptt2d as O2
from oracle import ptt3d as O3

pytestmark = pytest.mark.gpu

NY = [401, 406, 442, 481, 485, 487, 496, 513]


def _P():
    import paper_2606_09468_gb300 as P
    P.load_library()
    return P


def _check(g, o, energy):
    for k in (("energy", "mean_trc") if energy else ("mean_trc",)):
        assert abs(g[k] - o[k]) <= 1e-11 * abs(o[k]), (k, g[k], o[k])
    sc = max(abs(o["max_trc"]), abs(o["min_trc"]))
    for k in ("min_trc", "max_trc"):
        assert abs(g[k] - o[k]) <= 1e-11 * sc, (k, g[k], o[k])
    for k, band in (("n_lt3", "n_band3"), ("n_lt0", "n_band0")):
        assert abs(g[k] - o[k]) <= o[band], (k, g[k], o[k])


@pytest.mark.parametrize("form", ["fp64", "mixed", "fp64_ds"])
@pytest.mark.parametrize("ny", NY)
def test_2d(ny, form):
    P, nx = _P(), 8
    kw = dict(I.PAPER, dt=I.DT)
    prec = {"fp64": P.PTT_FP64, "mixed": P.PTT_MIXED, "fp64_ds": P.PTT_FP64_DS}[form]
    ora = O2.Channel2D(O2.Params(nx=nx, ny=ny, **kw))
    ora.init_state(3, 0.01)
    spec = [a + I.random_spectral(nx, ny, seed=50 + f, decay=0.05, scale=0.1)
            for f, a in enumerate(ora.state.as_list())]
    ora.state = O2.State(*spec)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, precision=prec, **kw)])
    ctx.set_spectral(0, I.spectral_to_abi(spec))
    _check(ctx.diagnostics(0)[-1], ora.diagnostics(), form != "mixed")   # the mixed form's energy is FP32
    ref = ora.get_physical()
    got = I.abi_to_phys(ctx.get_state(0))
    for f in range(5):
        assert np.max(np.abs(got[f] - ref[f])) <= 1e-12 * np.max(np.abs(ref[f])), f
    ctx.set_state(0, I.phys_to_abi(ref))
    back = I.abi_to_spectral(ctx.get_spectral(0))
    for f in range(5):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-12 * np.max(np.abs(ref[f])), f
    ctx.init_state(0, 3, 0.01)
    ora.init_state(3, 0.01)
    back = I.abi_to_spectral(ctx.get_spectral(0))
    for f, a in enumerate(ora.state.as_list()):
        assert np.max(np.abs(back[f] - a)) <= 1e-12 * np.max(np.abs(a)), f


@pytest.mark.parametrize("ny", [406, 481])
def test_3d(ny):
    P, nx, nz = _P(), 8, 4
    kw = dict(I.PAPER, lz=5.0, dt=I.DT)
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    ora.init_state(3, 0.01)
    spec = [a + I.random_spectral3(nx, ny, nz, seed=50 + f, decay=0.05, scale=0.1)
            for f, a in enumerate(ora.state.as_list())]
    ora.state = O3.State3(*spec)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, **kw)])
    ctx.set_spectral(0, I.spectral3_to_abi(spec))
    _check(ctx.diagnostics(0)[-1], ora.diagnostics(), True)
    ref = ora.get_physical()
    got = I.abi_to_phys3(ctx.get_state(0))
    for f in range(9):
        assert np.max(np.abs(got[f] - ref[f])) <= 1e-12 * np.max(np.abs(ref[f])), f
    ctx.set_state(0, I.phys3_to_abi(ref))
    back = I.abi_to_spectral3(ctx.get_spectral(0))
    for f in range(9):
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-12 * np.max(np.abs(ref[f])), f
