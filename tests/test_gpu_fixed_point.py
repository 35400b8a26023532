"""The fixed-point transforms of the FP64 form at the sizes and values where
they could go wrong: plans of every radix and of one to four passes, lines that
do not fill a block's groups, fields packed in one line that differ by twenty
orders of magnitude, lines of zeros.

Round trips: the DFT of a line of N values has an error of a few units of
2^-60 times the line's sum of moduli per value, at most 2^-60 N max|x| sqrt(N);
for N <= 1024 (2 (ny - 1), nx, nz) that is below 2^-45 = 2.9e-14 of the
field's maximum per transform, three transforms each way: 1e-13 is asked, as
of FP64 it would be.  Right-hand sides are held to the FP64 form's 1e-12."""
import numpy as np
import pytest

import ptt_inputs as I

pytestmark = pytest.mark.gpu


def _P():
    import paper_2606_09468_gb300 as P
    P.load_library()
    return P


# padded lengths (Mx, M): 10, 14 -> 5 2, 5 3; ... 6 8 4 4, 5 5 8 2, 6 6 10, one-pass and ragged
@pytest.mark.parametrize("nx,ny", [(8, 9), (14, 23), (18, 33), (50, 27), (54, 46), (84, 45), (112, 61), (250, 34)])
def test_explicit_rhs_2d(nx, ny):
    from oracle.ptt2d import Channel2D, Params, State
    P = _P()
    kw = dict(I.PAPER, dt=I.DT)
    ora = Channel2D(Params(nx=nx, ny=ny, **kw))
    ora.init_state(7, 0.05)
    extra = [I.random_spectral(nx, ny, seed=90 + f, decay=0.3, scale=0.01) for f in range(5)]
    st = State(*[a + e for a, e in zip(ora.state.as_list(), extra)])
    ctx = P.Context([P.make_params(nx=nx, ny=ny, **kw)])
    ctx.set_spectral(0, I.spectral_to_abi(st.as_list()))
    got, ref = I.abi_to_spectral(ctx.explicit_rhs(0)), ora.explicit_terms(st)
    for f in range(5):
        err = np.max(np.abs(got[f] - ref[f])) / np.max(np.abs(ref[f]))
        assert err <= 1e-12, (f, err)


@pytest.mark.parametrize("nx,ny,nz", [(8, 9, 4), (14, 11, 10), (30, 13, 18), (22, 26, 6)])
def test_explicit_rhs_3d(nx, ny, nz):
    from oracle import ptt3d as O3
    P = _P()
    kw = dict(I.PAPER, lz=5.0, dt=I.DT)
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    ora.init_state(7, 0.05)
    extra = [I.random_spectral3(nx, ny, nz, seed=90 + f, decay=0.3, scale=0.01) for f in range(9)]
    st = O3.State3(*(a + e for a, e in zip(ora.state.as_list(), extra)))
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, **kw)])
    ctx.set_spectral(0, I.spectral3_to_abi(st.as_list()))
    Nc, H = ora.explicit_terms(st)
    got, ref = I.abi_to_spectral3(ctx.explicit_rhs(0)), Nc + H
    for f in range(9):
        err = np.max(np.abs(got[f] - ref[f])) / np.max(np.abs(ref[f]))
        assert err <= 1e-12, (f, err)


@pytest.mark.parametrize("nx,ny", [(18, 33), (64, 65), (512, 257), (26, 14)])
def test_packed_fields_keep_their_own_size(nx, ny):
    """Physical values and back with (u, v), (c_xx, c_xy) of sizes 1e8 and
    1e-12 and c_yy zero: each field to 1e-13 of its own maximum."""
    P = _P()
    ctx = P.Context([P.make_params(nx=nx, ny=ny, dt=I.DT, **I.PAPER)])
    size = (1e8, 1e-12, 1e-12, 1e8, 0.0)
    spec = [I.random_spectral(nx, ny, seed=30 + f, decay=0.05, scale=s) for f, s in enumerate(size)]
    ctx.set_spectral(0, I.spectral_to_abi(spec))
    phys = I.abi_to_phys(ctx.get_state(0))
    K = nx // 2
    j, l = np.arange(nx), np.arange(ny)
    T = np.cos(np.pi * ((l[:, None] * l[None, :]) % (2 * (ny - 1))) / (ny - 1))
    E = np.exp(2j * np.pi * ((j[:, None] * np.arange(K)[None, :]) % nx) / nx)
    for f in range(5):
        ref = (E[:, :1] @ (spec[f][:1] @ T.T)).real + 2 * (E[:, 1:] @ (spec[f][1:] @ T.T)).real
        assert np.max(np.abs(phys[f] - ref)) <= 1e-13 * max(np.max(np.abs(ref)), 1e-300), f
    ctx.set_state(0, I.phys_to_abi(phys))
    back = I.abi_to_spectral(ctx.get_spectral(0))
    for f in range(5):
        # coefficients: to 1e-13 of the field's values
        assert np.max(np.abs(back[f] - spec[f])) <= 1e-13 * max(np.max(np.abs(phys[f])), 1e-300), f
