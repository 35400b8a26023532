"""Performance cases of the sPTT channel library.

Each case is a piece of work that a program using the library asks of it, through
the calls such a program makes: runs advanced by a number of time steps, with the
diagnostics records and the state read back at the end; the explicit right-hand
side on its own (the workspace-free call on device buffers, and the call of a
context); a snapshot re-interpolated onto another grid and read out in physical
space.  Shapes are those of the configurations, tests and benchmark of this
repository, or generic ones of the same range.

Initial states are the laminar sPTT channel plus a seeded, broad-band,
divergence-free no-slip velocity perturbation and a perturbation of every
conformation component, built directly as spectral coefficients.

`exact` is a plain 64-bit restatement of the method in torch (FFTs in x and z,
dense Chebyshev matrices in y, the tau systems solved through an eigen-basis of
the second-derivative operator); it uses nothing of the library."""
import functools
import math

import numpy as np
import torch

import paper_2606_09468_gb300 as P
import ptt_inputs as I

FORMS = {"fp64": P.PTT_FP64, "mixed": P.PTT_MIXED, "mixed_tc": P.PTT_MIXED_TC,
         "fp64_ds": P.PTT_FP64_DS}
FLUID = dict(I.PAPER, dt=I.DT)      # the paper's fluid, the benchmark's time step
LZ = I.LZ3
U_AMPLITUDE, C_AMPLITUDE = 1e-3, 0.03


def _shapes(case):
    """The (nx, ny, nz) of every run of a case, from "128x97x64 64x65"."""
    out = []
    for word in case["shapes"].split():
        s = [int(v) for v in word.split("x")]
        out.append(tuple(s + [1]) if len(s) == 2 else tuple(s))
    return [s for s in out for _ in range(case.get("copies", 1))]


def _wi(case, i):
    """Wi of run i: the fluid's, or spread evenly over [50, 200] (the ragged ensemble)."""
    return 50.0 + 150.0 * ((i * 29) % 64) / 63.0 if case.get("spread_wi") else FLUID["wi"]


# ---------------------------------------------------------------- the cases --
def listed():
    sweep = " ".join("%dx%d" % (nx, ny) for nx in I.SWEEP_NX for ny in I.SWEEP_NY)
    ragged = " ".join("%dx%d" % (nx, ny) for nx, ny, _, _ in I.ensemble_members())
    return [
        # one small run followed step by step (a monitored or steered run): launches and latency
        {"name": "step_2d_64x65_fp64", "kind": "steps", "shapes": "64x65", "form": "fp64", "steps": 1},
        # the right-hand side inside someone else's integrator, device buffers in and out
        {"name": "rhs_noalloc_2d_256x129", "kind": "rhs_noalloc", "shapes": "256x129", "form": "fp64"},
        # one 2D run at an odd size (factors 7 and 11)
        {"name": "run_2d_350x155_fp64", "kind": "steps", "shapes": "350x155", "form": "fp64", "steps": 20},
        # the 2D resolution scan: 27 runs of nine shapes, the benchmark's headline workload
        {"name": "sweep_2d_27_fp64", "kind": "steps", "shapes": sweep, "copies": 3, "form": "fp64", "steps": 20},
        # the ragged ensemble: 64 runs of uneven shape and Wi, mixed precision
        {"name": "ensemble_2d_64_mixed", "kind": "steps", "shapes": ragged, "form": "mixed", "steps": 20,
         "spread_wi": True},
        # the 3D channel of the benchmark in its arithmetic forms
        {"name": "run_3d_128x97x64_fp64", "kind": "steps", "shapes": "128x97x64", "form": "fp64", "steps": 10},
        {"name": "run_3d_128x97x64_mixed", "kind": "steps", "shapes": "128x97x64", "form": "mixed", "steps": 10},
        {"name": "run_3d_128x97x64_ds", "kind": "steps", "shapes": "128x97x64", "form": "fp64_ds", "steps": 10},
        # an odd 3D size (factors 5, 9, 11, 13) with the tensor-core Chebyshev transforms
        {"name": "run_3d_90x79x44_mixed_tc", "kind": "steps", "shapes": "90x79x44", "form": "mixed_tc", "steps": 10},
        # the largest production run of the benchmark's default list that a session waits for
        {"name": "run_3d_256x129x128_mixed", "kind": "steps", "shapes": "256x129x128", "form": "mixed", "steps": 5},
        # the explicit right-hand side of a 3D context, to the host
        {"name": "rhs_3d_64x65x32_fp64", "kind": "rhs", "shapes": "64x65x32", "form": "fp64"},
        # a snapshot re-interpolated onto a finer grid and read out in physical space
        {"name": "snapshot_3d_to_128x97x64", "kind": "snapshot", "shapes": "64x65x32 128x97x64", "form": "fp64"},
    ]


def _smooth(n, primes=(2, 3, 5, 7, 11, 13)):
    for p in primes:
        while n % p == 0:
            n //= p
    return n == 1


def _between(rng, lo, hi, ok):
    """A size of the library's range between lo and hi, spread over its logarithm."""
    while True:
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        if lo <= n <= hi and ok(n):
            return n


def _nx(rng, lo, hi):
    return _between(rng, lo, hi, lambda n: n % 2 == 0 and _smooth(n))


def _ny(rng, lo, hi):
    return _between(rng, lo, hi, lambda n: _smooth(n - 1))


def draw(rng):
    kind = rng.choice(["steps2", "steps2", "many2", "many2", "steps3", "steps3", "steps3", "rhs_noalloc",
                       "rhs", "snapshot"])
    form = rng.choice(["fp64", "mixed", "fp64_ds"])
    if kind == "steps2":
        return {"kind": "steps", "shapes": "%dx%d" % (_nx(rng, 64, 512), _ny(rng, 65, 257)), "form": form,
                "steps": rng.choice([1, 5, 20])}
    if kind == "many2":
        shapes = " ".join("%dx%d" % (_nx(rng, 64, 512), _ny(rng, 65, 257)) for _ in range(rng.randint(2, 12)))
        return {"kind": "steps", "shapes": shapes, "copies": rng.choice([1, 2, 3]), "form": form,
                "steps": rng.choice([5, 20]), "spread_wi": True}
    if kind == "steps3":
        form = rng.choice(["fp64", "mixed", "mixed_tc", "fp64_ds"])
        while True:
            nx, ny, nz = _nx(rng, 32, 256), _ny(rng, 33, 129), _nx(rng, 16, 128)
            if nx * ny * nz <= 900000:
                return {"kind": "steps", "shapes": "%dx%dx%d" % (nx, ny, nz), "form": form,
                        "steps": rng.choice([1, 5])}
    if kind == "rhs_noalloc":
        return {"kind": "rhs_noalloc", "shapes": "%dx%d" % (_nx(rng, 64, 512), _ny(rng, 65, 257)), "form": "fp64"}
    if kind == "rhs":
        return {"kind": "rhs", "shapes": "%dx%dx%d" % (_nx(rng, 32, 96), _ny(rng, 33, 97), _nx(rng, 16, 64)),
                "form": rng.choice(["fp64", "fp64_ds"])}
    a = (_nx(rng, 32, 96), _ny(rng, 33, 97), _nx(rng, 16, 64))
    b = (_nx(rng, 64, 160), _ny(rng, 65, 129), _nx(rng, 32, 64))
    return {"kind": "snapshot", "shapes": "%dx%dx%d %dx%dx%d" % (a + b), "form": "fp64"}


# -------------------------------------------------------------------- work --
def _fft(n):
    return 5.0 * n * math.log2(n)


def _step_work(nx, ny, nz):
    """Bytes (state and history, each array read and written once) and operations of one step."""
    K, nf, ne = nx // 2, (9 if nz > 1 else 5), (8 if nz > 1 else 4)
    NK = K * nz * ny
    M, Mx, Mz = 1.5 * ny, 1.5 * nx, (1.5 * nz if nz > 1 else 1)
    by = 16.0 * NK * (2 * nf + 8 * ne)
    if nz > 1:
        fl = 26 * K * nz * _fft(M) + 35 * M * K * _fft(Mz) + M * Mz * (23 * _fft(Mx) + 200 * Mx) + 480 * NK
    else:
        fl = 14 * K * _fft(M) + M * (10 * _fft(Mx) + 42 * Mx) + 250 * NK
    return by, fl


def work(case):
    by = fl = 0.0
    if case["kind"] == "steps":
        for s in _shapes(case):
            b, f = _step_work(*s)
            by, fl = by + b * case["steps"], fl + f * case["steps"]
    elif case["kind"] in ("rhs", "rhs_noalloc"):
        nx, ny, nz = _shapes(case)[0]
        by = 32.0 * (9 if nz > 1 else 5) * (nx // 2) * nz * ny
        fl = _step_work(nx, ny, nz)[1]
    else:
        (ax, ay, az), (bx, b_y, bz) = _shapes(case)
        by = 9.0 * (16 * (ax // 2) * ay * az + 8 * bx * b_y * bz)
        fl = 9.0 * ((bx // 2) * bz * _fft(2 * b_y) + b_y * (bx // 2) * _fft(bz) + b_y * bz * _fft(bx) / 2)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ inputs --
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


@functools.lru_cache(maxsize=64)
def _cheb(N):
    """(derivative matrix, matrix of the product with 1 - y^2), N x N, on the device."""
    n = np.arange(N)
    D = np.where((n[None, :] > n[:, None]) & ((n[None, :] + n[:, None]) % 2 == 1), 2.0 * n[None, :], 0.0)
    D[0] *= 0.5
    W = 0.5 * np.eye(N)
    for k in range(N):                       # (1 - y^2) T_k = T_k/2 - (T_{k+2} + T_{|k-2|})/4
        if k + 2 < N:
            W[k + 2, k] -= 0.25
        W[abs(k - 2), k] -= 0.25
    return tuple(torch.tensor(a, dtype=torch.float64, device=_device()) for a in (D, W))


def _laminar(N, wi):
    """Chebyshev coefficients of the laminar U, c_xx, c_xy (closed form with kappa = 0)."""
    beta, eps = FLUID["beta"], FLUID["eps"]
    y = np.cos(np.pi * np.arange(N) / (N - 1))
    y[N // 2] = 0.0 if N % 2 else y[N // 2]
    s = -2.0 * wi * y
    a = 2.0 * beta * eps
    for _ in range(60):
        s = s - (a * s ** 3 + s + 2.0 * wi * y) / (3.0 * a * s * s + 1.0)
    F = 0.5 * s ** 2 + 0.5 * eps * (1 + 3 * beta) * s ** 4 + 2 * beta * eps ** 2 * s ** 6
    U = -(F - F[0]) / (2.0 * wi * wi)
    n = np.arange(N)
    E = np.cos(np.pi * ((n[:, None] * n[None, :]) % (2 * (N - 1))) / (N - 1))   # DCT-I
    w = np.where((n == 0) | (n == N - 1), 0.5, 1.0)
    A = (2.0 / (N - 1)) * w[:, None] * E * w[None, :]
    return [A @ f for f in (U, 1.0 + 2.0 * s * s, s)]


def _signed(nz):
    s = torch.arange(nz, device=_device())
    return torch.where(s < (nz + 1) // 2, s, s - nz)


def _state(shape, wi, seed):
    """Initial coefficients, complex (9, ny, nx/2, nz): u, v, w, c_xx, c_xy, c_xz, c_yy, c_yz, c_zz
    (in 2D nz = 1, w = c_xz = c_yz = 0 and c_zz = 1)."""
    nx, N, nz = shape
    K, dev = nx // 2, _device()
    g = torch.Generator(device=dev).manual_seed(seed)
    D, W = _cheb(N)
    m, s, n = torch.arange(K, device=dev).double(), _signed(nz).double(), torch.arange(N, device=dev).double()
    decay = (torch.exp(-n / 6.0) * (n < N - 6))[:, None, None] / (1.0 + m[:, None] ** 2 + s[None, :] ** 2) ** 1.5

    def field():
        a = torch.randn((N, K, nz, 2), generator=g, dtype=torch.float64, device=dev)
        a = torch.view_as_complex(a) * decay
        if nz > 1:
            a[:, :, nz // 2] = 0
            a[:, 0, nz // 2 + 1:] = torch.flip(a[:, 0, 1:nz // 2], (-1,)).conj()
        a[:, 0, 0] = a[:, 0, 0].real + 0j
        return a

    def mat(A, a):
        return (A @ torch.view_as_real(a.reshape(N, -1).contiguous()).reshape(N, -1)).reshape(N, -1, 2) \
            .contiguous().view(torch.complex128).reshape(a.shape)

    def scaled(fields, amplitude):
        rms = math.sqrt(sum(float((2 * f[:, 1:].abs() ** 2).sum() + (f[:, 0].abs() ** 2).sum()) for f in fields))
        return [f * (amplitude / rms) for f in fields]

    ikx = (2j * math.pi / FLUID["lx"]) * m[:, None]
    ikz = (2j * math.pi / LZ) * s[None, :] * (s[None, :] != -(nz // 2) if nz > 1 else 1)
    p1 = mat(W, mat(W, field()))
    p1[:, 0, 0] = 0
    vel = [mat(D, p1), -ikx * p1, torch.zeros_like(p1)]
    if nz > 1:
        p2 = mat(W, mat(W, field()))
        p2[:, 0, 0] = 0
        vel[1], vel[2] = vel[1] - ikz * p2, mat(D, p2)
    vel = scaled(vel, U_AMPLITUDE)
    keep = (0, 1, 2, 3, 4, 5) if nz > 1 else (0, 1, 3)
    c = [mat(W, field()) if i in keep else torch.zeros_like(p1) for i in range(6)]
    c = scaled(c, C_AMPLITUDE)
    X = torch.stack(vel + c)
    for f, a in zip((0, 3, 4), _laminar(N, wi)):
        X[f, :, 0, 0] += torch.tensor(a, device=dev)
    X[6, 0, 0, 0] += 1.0
    X[8, 0, 0, 0] += 1.0
    return X


FIELDS2 = [0, 1, 3, 4, 6]


def _abi(X):
    """Coefficients as the library lays them out: double [nf][ny][nx/2](2D: [2], 3D: [nz][2])."""
    Y = X[FIELDS2][..., 0] if X.shape[-1] == 1 else X
    return torch.view_as_real(Y.contiguous())


def _pinned(n, dtype=torch.float64):
    return torch.empty(n, dtype=dtype, pin_memory=torch.cuda.is_available())


def _params(case, shape, i, form):
    return P.make_params(nx=shape[0], ny=shape[1], nz=shape[2], precision=FORMS[form],
                         **dict(FLUID, wi=_wi(case, i), **({"lz": LZ} if shape[2] > 1 else {})))


def _context(case, shapes, seed):
    ctx = P.Context([_params(case, s, i, case["form"]) for i, s in enumerate(shapes)])
    for i, s in enumerate(shapes):
        ctx.set_spectral(i, _abi(_state(s, _wi(case, i), 1000 * seed + i)).cpu().numpy())
        ctx.diagnostics(i)
    return ctx


def prepare(case, seed):
    shapes = _shapes(case)
    if case["kind"] == "rhs_noalloc":
        spec = _abi(_state(shapes[0], _wi(case, 0), 1000 * seed)).contiguous()
        return {"kind": case["kind"], "params": _params(case, shapes[0], 0, "fp64"), "in": spec,
                "out": torch.empty_like(spec)}
    if case["kind"] == "snapshot":
        src, dst = _context(case, shapes[:1], seed), P.Context([_params(case, shapes[1], 0, case["form"])])
        nx, ny, nz = shapes[1]
        out = _pinned(9 * nx * ny * nz)
        return {"kind": case["kind"], "src": src, "dst": dst, "out": out, "view": out.numpy()}
    ctx = _context(case, shapes, seed)
    sizes = [(9 if s[2] > 1 else 5) * s[1] * (s[0] // 2) * s[2] * 2 for s in shapes]
    out = _pinned(sum(sizes))
    at = np.concatenate([[0], np.cumsum(sizes)])
    views = [out.numpy()[a:b] for a, b in zip(at[:-1], at[1:])]
    return {"kind": case["kind"], "ctx": ctx, "steps": case.get("steps", 0), "out": out, "views": views}


RECORD = np.dtype([("step", "i8"), ("t", "f8"), ("real", "f8", 4), ("count", "i8", 8), ("mid", "f8", 32),
                   ("status", "i4"), ("reserved", "i4")])


def run(state):
    if state["kind"] == "rhs_noalloc":
        P.ptt_explicit_rhs_noalloc(state["params"], state["in"].data_ptr(), state["out"].data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if state["kind"] == "snapshot":
        state["dst"].resample_from(0, state["src"], 0)
        P.ptt_get_state(state["dst"].ctx, 0, state["view"])
        return state["out"]
    ctx = state["ctx"]
    if state["kind"] == "rhs":
        P.ptt_explicit_rhs(ctx.ctx, 0, state["views"][0])
        return state["out"]
    n = state["steps"]
    ctx.step(n)
    records = []
    for i, view in enumerate(state["views"]):
        records += P.ptt_diagnostics(ctx.ctx, i, n)
        P.ptt_get_spectral(ctx.ctx, i, view)
    r = np.frombuffer(b"".join(bytes(x) for x in records), dtype=RECORD).reshape(len(state["views"]), n)
    return {"state": state["out"], "records": np.concatenate([r["real"], r["mid"]], axis=-1), "counts": r["count"]}


# -------------------------------------------------- the method in 64 bits --
def _pad(n):
    while not _smooth(n, (2, 3, 5)):
        n += 1
    return n


def _pad_y(N):
    M = (3 * N - 1) // 2
    while M % 2 or not _smooth(M, (2, 3, 5)):
        M += 1
    return M


@functools.lru_cache(maxsize=64)
def _solver(N):
    """Per parity p of the Chebyshev index: rows n = p, p+2, .. <= N-3, unknowns a_n, n = p+2, .., with
    a_p = g - sum of the others: (alpha E - beta D2) b = R - alpha g e_p, through E^-1 D2 = V diag(lam) V^-1."""
    dev = _device()
    D = _cheb(N)[0].cpu().numpy()
    D2 = D @ D
    out = []
    for p in (0, 1):
        rows, cols = np.arange(p, N - 2, 2), np.arange(p + 2, N, 2)
        E = (rows[:, None] == cols[None, :]).astype(float)
        E[0] = -1.0
        Ei = np.linalg.inv(E)
        lam, V = np.linalg.eig(Ei @ D2[np.ix_(rows, cols)])
        W = np.linalg.inv(V) @ Ei
        out.append([torch.tensor(np.ascontiguousarray(x.real), device=dev) for x in (lam, V, W)]
                   + [torch.tensor(x, device=dev) for x in (rows, cols)])
        assert np.max(np.abs(lam.imag)) < 1e-6 * np.max(np.abs(lam.real))
    return out


class _Channel:
    """One run, in 64 bits.  Fields complex (9, ny, K nz) with the modes flattened."""

    def __init__(self, shape, wi):
        self.nx, self.N, self.nz = shape
        dev, N, nz = _device(), self.N, self.nz
        self.K = K = self.nx // 2
        f = FLUID
        self.dt, self.eps, self.iwi, self.kappa = f["dt"], f["eps"], 1.0 / wi, f["kappa"]
        self.gam, self.nu, self.force = (1 - f["beta"]) / (f["re"] * wi), f["beta"] / f["re"], 2.0 / f["re"]
        s = _signed(nz).double()
        self.live = (s != -(nz // 2)) if nz > 1 else torch.ones(1, dtype=torch.bool, device=dev)
        kx = (2 * math.pi / f["lx"]) * torch.arange(K, dtype=torch.float64, device=dev)
        kz = (2 * math.pi / LZ) * s * self.live
        self.kx, self.kz = [a.reshape(-1) for a in torch.broadcast_tensors(kx[:, None], kz[None, :])]
        self.k2 = self.kx ** 2 + self.kz ** 2
        self.on = self.live[None, :].expand(K, nz).reshape(-1)
        self.Mx, self.Mz, self.M = _pad(3 * self.nx // 2 - 2), (_pad(3 * nz // 2 - 2) if nz > 1 else 1), _pad_y(N)
        self.D = _cheb(N)[0]
        j, n = torch.arange(self.M, device=dev), torch.arange(N, device=dev)
        arg = ((2 * j[:, None] + 1) * n[None, :]) % (4 * self.M)
        self.T = torch.cos(math.pi / (2.0 * self.M) * arg.double())
        self.A = (2.0 / self.M) * self.T.T.contiguous()
        self.A[0] *= 0.5
        self.old = []

    def mat(self, A, a):
        """A times the Chebyshev (second to last) axis."""
        r = torch.view_as_real(a.contiguous()).flatten(-2)
        return torch.view_as_complex((A @ r).unflatten(-1, (-1, 2)).contiguous())

    def grid(self, a, Mx, Mz):
        """Modes (.., rows, K nz) -> values (.., rows, Mz, Mx)."""
        K, nz = self.K, self.nz
        b = a.unflatten(-1, (K, nz))
        if nz > 1:
            h = nz // 2
            z = torch.zeros(b.shape[:-1] + (Mz,), dtype=b.dtype, device=b.device)
            z[..., :h], z[..., Mz - h + 1:] = b[..., :h], b[..., h + 1:]
            b = torch.fft.ifft(z, dim=-1, norm="forward")
        return torch.fft.irfft(b.transpose(-1, -2), n=Mx, dim=-1, norm="forward")

    def modes(self, f):
        """Values on the padded (Mz, Mx) grid -> modes (.., rows, K nz)."""
        K, nz = self.K, self.nz
        b = torch.fft.rfft(f, dim=-1, norm="forward")[..., :K].transpose(-1, -2)
        if nz > 1:
            h = nz // 2
            z = torch.fft.fft(b, dim=-1, norm="forward")
            b = torch.zeros(b.shape[:-1] + (nz,), dtype=b.dtype, device=b.device)
            b[..., :h], b[..., h + 1:] = z[..., :h], z[..., self.Mz - h + 1:]
        return b.flatten(-2)

    def products(self, X):
        """Dealiased N_c (6) and -u.grad u (3), spectral."""
        step = 16 if X[0].numel() > 1 << 18 else self.M      # y rows at a time
        out = []
        dX = self.mat(self.D, X)
        ikx, ikz = 1j * self.kx, 1j * self.kz
        for j in range(0, self.M, step):
            T = self.T[j:j + step]
            Y, dY = self.mat(T, X), self.mat(T, dX)
            q = self.grid(Y, self.Mx, self.Mz)
            qx, qz = self.grid(ikx * Y, self.Mx, self.Mz), self.grid(ikz * Y, self.Mx, self.Mz)
            qy = self.grid(dY, self.Mx, self.Mz)
            u, c = q[:3], q[3:]
            C = [[c[0], c[1], c[2]], [c[1], c[3], c[4]], [c[2], c[4], c[5]]]
            L = [[qx[i], qy[i], qz[i]] for i in range(3)]
            rw = (1.0 + self.eps * (c[0] + c[3] + c[5] - 3.0)) * self.iwi
            o = []
            for a, (i, k) in enumerate([(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]):
                t = -(u[0] * qx[3 + a] + u[1] * qy[3 + a] + u[2] * qz[3 + a])
                for b in range(3):
                    t = t + L[i][b] * C[b][k] + C[i][b] * L[k][b]
                o.append(t - (C[i][k] - (1.0 if i == k else 0.0)) * rw)
            for i in range(3):
                o.append(-(u[0] * L[i][0] + u[1] * L[i][1] + u[2] * L[i][2]))
            out.append(self.modes(torch.stack(o)))
        return self.mat(self.A, torch.cat(out, dim=1))

    def explicit(self, X):
        """N_c and H."""
        R = self.products(X)
        dc = self.mat(self.D, X[[4, 6, 7]])
        ikx, ikz = 1j * self.kx, 1j * self.kz
        for t, (a, b) in enumerate([(3, 5), (4, 7), (5, 8)]):
            R[6 + t] += self.gam * (ikx * X[a] + dc[t] + ikz * X[b])
        R[6, 0, 0] += self.force
        return R * self.on

    def solve(self, R, alpha, beta, g):
        """(alpha - beta D^2) a = R on the tau rows, the sum over each parity = g[parity]."""
        a = torch.zeros_like(R)
        for p, (lam, V, W, rows, cols) in enumerate(_solver(self.N)):
            r = R[..., rows, :].clone()
            r[..., 0, :] -= alpha * g[p]
            b = self.mat(V, self.mat(W, r) / (alpha - beta * lam[:, None]))
            a[..., cols, :] = b
            a[..., p, :] = g[p] - b.sum(dim=-2)
        return a

    def step(self, X):
        o = min(len(self.old), 3)
        sa = [[1, -1, 0, 0, 0], [1.5, -2, 0.5, 0, 0], [11 / 6, -3, 1.5, -1 / 3, 0], [25 / 12, -4, 3, -4 / 3, 0.25]][o]
        sb = [[1, 0, 0, 0], [2, -1, 0, 0], [3, -3, 1, 0], [4, -6, 4, -1]][o]
        ikx, ikz, k2 = 1j * self.kx, 1j * self.kz, self.k2
        R = self.explicit(X)
        H = R[6:]
        q1 = self.mat(self.D, self.mat(self.D, X[1])) - k2 * X[1]
        q2 = ikz * X[0] - ikx * X[2]
        f1 = -self.mat(self.D, ikx * H[0] + ikz * H[2]) - k2 * H[1]
        f2 = ikz * H[0] - ikx * H[2]
        q1[:, 0], q2[:, 0], f1[:, 0], f2[:, 0] = X[0][:, 0], X[2][:, 0], H[0][:, 0], H[2][:, 0]
        self.old.insert(0, (torch.cat([X[3:], q1[None], q2[None]]), torch.cat([R[:6], f1[None], f2[None]])))
        self.old = self.old[:4]
        S = sum(-sa[j + 1] / self.dt * x + sb[j] * n for j, (x, n) in enumerate(self.old[:o + 1]))
        a0 = sa[0] / self.dt
        Y = torch.empty_like(X)
        walls = [S[:6, p::2].sum(dim=1) / a0 for p in (0, 1)]
        Y[3:] = self.solve(S[:6], a0 + self.kappa * k2, self.kappa, walls)
        z = [torch.zeros_like(k2), torch.zeros_like(k2)]
        phi, eta = self.solve(S[6:], a0 + self.nu * k2, self.nu, z)
        kk = torch.where(k2 > 0, k2, torch.ones_like(k2))
        v = self.solve(-phi, kk, 1.0, z)
        n2 = (torch.arange(self.N, device=k2.device, dtype=torch.float64) ** 2)[:, None]
        for p in (0, 1):       # influence correction: v'(+-1) = 0, parity by parity
            one = [torch.full_like(k2, float(p == q)) + 0j for q in (0, 1)]
            ph = self.solve(torch.zeros_like(v), a0 + self.nu * k2, self.nu, one)
            vh = self.solve(-ph, kk, 1.0, z)
            v = v - vh * ((n2 * v)[p::2].sum(dim=0) / (n2 * vh)[p::2].sum(dim=0))
        dv = self.mat(self.D, v)
        Y[0] = 1j * (self.kx * dv - self.kz * eta) / kk
        Y[2] = 1j * (self.kz * dv + self.kx * eta) / kk
        Y[1] = v
        Y[0][:, 0], Y[1][:, 0], Y[2][:, 0] = phi[:, 0], 0, eta[:, 0]
        return Y * self.on

    def record(self, X):
        """Energy, <Tr c>, extrema of Tr c, mid-plane power sums (8 x 4)."""
        N, nx, nz, dev = self.N, self.nx, self.nz, X.device
        n = torch.arange(N, device=dev)
        tr = X[3] + X[6] + X[8]
        even = n[::2].double()
        mean = 0.5 * (tr[::2, 0].real * (2.0 / (1.0 - even ** 2))).sum()
        y, w = np.polynomial.legendre.leggauss(N + 2)
        G = torch.tensor(np.cos(np.arange(N)[None, :] * np.arccos(y)[:, None]), device=dev)
        e = self.mat(G, X[:3])
        e = e.real ** 2 + e.imag ** 2
        twice = torch.where(self.kx > 0, 2.0, 1.0)
        energy = 0.25 * ((e * twice).sum(dim=(0, 2)) * torch.tensor(w, device=dev)).sum()
        l = torch.arange(N, device=dev)
        G = torch.cos(math.pi / (N - 1) * ((l[:, None] * n[None, :]) % (2 * (N - 1))).double())
        t = self.grid(self.mat(G, tr), nx, nz)
        mid = torch.tensor([1.0, 0.0, -1.0, 0.0], device=dev, dtype=torch.float64)[n % 4]
        dmid = torch.tensor([0.0, 1.0, 0.0, -1.0], device=dev, dtype=torch.float64)[n % 4] * n
        at = lambda a, row: self.mat(row[None], a)                  # noqa: E731
        u, v, w3 = at(X[0], mid), at(X[1], mid), at(X[2], mid)
        up, wp = u.clone(), w3.clone()
        up[:, 0] = 0
        wp[:, 0] = 0
        ikx, ikz = 1j * self.kx, 1j * self.kz
        if nz > 1:
            q = [at(tr, mid), up, wp, ikx * u, ikz * u, ikx * w3, ikz * w3, v]
        else:
            q = [at(tr, mid), up, v, ikx * u, ikx * v, at(X[0], dmid)]
        q = self.grid(torch.stack(q), nx, nz).flatten(1)
        sums = torch.zeros(8, 4, dtype=torch.float64, device=dev)
        for p in range(4):
            sums[:len(q), p] = (q ** (p + 1)).sum(dim=1)
        return torch.cat([torch.stack([energy, mean, t.min(), t.max()]), sums.flatten()])


def _flat(X, nz):
    """(9, ny, K nz) -> the library's spectral layout, flat."""
    return _abi(X.unflatten(-1, (-1, nz))).flatten().cpu()


def exact(case, seed):
    shapes = _shapes(case)
    state = lambda i: _state(shapes[i], _wi(case, i), 1000 * seed + i).flatten(-2)   # noqa: E731
    if case["kind"] in ("rhs", "rhs_noalloc"):
        ch = _Channel(shapes[0], _wi(case, 0))
        R = ch.explicit(state(0))                       # N_c (6), H (3)
        if case["kind"] == "rhs":
            return _flat(R, shapes[0][2])
        return torch.view_as_real(R[[0, 1, 3, 6, 7]].contiguous())
    if case["kind"] == "snapshot":
        (_, N, nz), (bx, b_y, bz) = shapes
        a, ch, b = state(0).unflatten(-1, (-1, nz)), _Channel(shapes[1], FLUID["wi"]), None
        K, h = min(a.shape[2], bx // 2), min(nz, bz) // 2
        b = torch.zeros((9, b_y, bx // 2, bz), dtype=a.dtype, device=a.device)
        n = min(N, b_y)
        b[:, :n, :K, :h], b[:, :n, :K, bz - h + 1:] = a[:, :n, :K, :h], a[:, :n, :K, nz - h + 1:]
        l = torch.arange(b_y, device=a.device)
        G = torch.cos(math.pi / (b_y - 1) * ((l[:, None] * l[None, :]) % (2 * (b_y - 1))).double())
        return ch.grid(ch.mat(G, b.flatten(-2)), bx, bz).transpose(1, 2).flatten().cpu()
    flats, records = [], []
    for i, s in enumerate(shapes):
        X, ch, rec = state(i), _Channel(s, _wi(case, i)), []
        for _ in range(case["steps"]):
            X = ch.step(X)
            rec.append(ch.record(X))
        flats.append(_flat(X, s[2]))
        records.append(torch.stack(rec))
    return {"state": torch.cat(flats), "records": torch.stack(records).cpu(), "counts": None}
