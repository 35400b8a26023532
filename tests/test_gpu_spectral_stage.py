"""The lane-sequential per-mode stage at the sizes where it can go wrong: mode
counts that are no multiple of a block's 16, both parities of ny, the fewest
Chebyshev rows, no diffusion, every order of the start-up steps.  Six steps
against the oracle: each step's error is that of FP64 sums and of the tau
systems (1e-11 per step is the one-step bar of the parity tests); the steps
are far below the flow's own time scale, so six of them are given 6e-11."""
import numpy as np
import pytest

import ptt_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,kappa", [(12, 9, 6, 5e-5), (10, 10, 6, 5e-5), (14, 13, 10, 0.0),
                                            (22, 26, 18, 5e-5), (8, 129, 4, 5e-5)])
def test_steps_3d(nx, ny, nz, kappa):
    import paper_2606_09468_gb300 as P
    from oracle import ptt3d as O3
    P.load_library()
    kw = dict(I.PAPER, lz=5.0, dt=I.DT)
    kw["kappa"] = kappa
    ora = O3.Channel3D(O3.Params3(nx=nx, ny=ny, nz=nz, **kw))
    ora.init_state(5, 0.02)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, nz=nz, **kw)])
    ctx.init_state(0, 5, 0.02)
    for _ in range(6):
        ora.step()
    ctx.step(6)
    assert ctx.synchronize() == P.PTT_OK
    got, ref = I.abi_to_phys3(ctx.get_state(0)), ora.get_physical()
    for f in range(9):
        scale = max(np.max(np.abs(r)) for r in (ref[:3] if f < 3 else ref[3:]))
        assert np.max(np.abs(got[f] - ref[f])) <= 6e-11 * scale, f


@pytest.mark.parametrize("nx,ny,kappa", [(8, 9, 5e-5), (10, 10, 5e-5), (14, 13, 0.0), (22, 34, 5e-5),
                                         (16, 513, 5e-5), (512, 9, 5e-5)])
def test_steps_2d(nx, ny, kappa):
    import paper_2606_09468_gb300 as P
    from oracle.ptt2d import Channel2D, Params
    P.load_library()
    kw = dict(I.PAPER, dt=I.DT)
    kw["kappa"] = kappa
    ora = Channel2D(Params(nx=nx, ny=ny, **kw))
    ora.init_state(5, 0.02)
    ctx = P.Context([P.make_params(nx=nx, ny=ny, **kw)])
    ctx.init_state(0, 5, 0.02)
    for _ in range(6):
        ora.step()
    ctx.step(6)
    assert ctx.synchronize() == P.PTT_OK
    got, ref = I.abi_to_phys(ctx.get_state(0)), ora.get_physical()
    for f in range(5):
        scale = max(np.max(np.abs(r)) for r in (ref[:2] if f < 2 else ref[2:]))
        assert np.max(np.abs(got[f] - ref[f])) <= 6e-11 * scale, f
