"""The work that users of the library have it do, as cases to time and compare.

A case is one pass through the public entry points on data that the caller
holds: time steps of one trajectory or of an ensemble (a start state goes in,
the state n steps later comes out), one evaluation of the nonlinear term, one
forward or gradient pass of the proposal network.  `exact` restates each of
them in plain 64-bit torch.

Fields of a case: "kind" (step, host, ens, noalloc, forward, gradients); the
resolution N, K, M, m_p (ensembles: "shapes", "count x N x K x M" separated by
blanks); alpha, Re, dt; "precision" 0 (FP64) or 1 (mixed); "steps" per pass.
"""
import ctypes
import functools
import math

import numpy as np
import torch

from paper_1705_03838_gb300 import opf


def listed():
    return [
        # A saturated helical wave of rotating pipe flow at the resolution its
        # orbit search uses: the smallest grid in use, all launch latency.
        dict(name="tiny_fp64", kind="step", N=20, K=4, M=5, m_p=2, alpha=1.0, Re=140.0, dt=0.01, precision=0, steps=10,
             rot=1.0, force=0.0, cfl=0.0),
        # The plain FP64 run at the smallest published-size resolution.
        dict(name="small_fp64", kind="step", N=32, K=16, M=16, m_p=1, alpha=1.25, Re=2000.0, dt=0.01, precision=0,
             steps=10, rot=0.0, force=0.0, cfl=0.0),
        # The usual single run (a puff at Re = 2400), in both precisions.
        dict(name="medium_mixed", kind="step", N=48, K=32, M=24, m_p=2, alpha=1.25, Re=2400.0, dt=0.005, precision=1,
             steps=5, rot=0.0, force=0.0, cfl=0.0),
        dict(name="medium_fp64", kind="step", N=48, K=32, M=24, m_p=2, alpha=1.25, Re=2400.0, dt=0.005, precision=0,
             steps=5, rot=0.0, force=0.0, cfl=0.0),
        # Sizes that fit no table: odd N, 3K = 81, 3M = 60, with a body force
        # and a frame rotation.
        dict(name="ragged_mixed", kind="step", N=41, K=27, M=20, m_p=1, alpha=1.1, Re=1900.0, dt=0.004, precision=1,
             steps=3, rot=0.3, force=0.05, cfl=0.0),
        # Driving the solver from a host program, one step at a time: the
        # state goes in from pinned memory, the new state and the energy
        # budget come back.
        dict(name="medium_host", kind="host", N=48, K=32, M=24, m_p=2, alpha=1.25, Re=2400.0, dt=0.005, precision=0,
             steps=1),
        # A sweep over Re at mixed resolutions (training data, transition
        # statistics): every trajectory has operators of its own.
        dict(name="ensemble_mixed", kind="ens", shapes="8x32x16x16 8x48x24x24 6x64x32x32", m_p=1, alpha=1.25, Re=1800.0,
             Re2=2600.0, dt=0.005, dt2=0.005, precision=1, steps=4),
        # The integrations of a Newton-Krylov iteration: many guesses of one
        # resolution in FP64, each with the time step of its own period.
        dict(name="orbits_fp64", kind="ens", shapes="64x32x16x16", m_p=2, alpha=1.25, Re=2250.0, Re2=2250.0, dt=0.005,
             dt2=0.0049, precision=0, steps=4),
        # A large turbulent run under CFL control (dt already at its bound).
        dict(name="large_mixed", kind="step", N=128, K=128, M=128, m_p=1, alpha=0.4, Re=5300.0, dt=5e-5, precision=1,
             steps=2, rot=0.0, force=0.0, cfl=0.5),
        # The nonlinear term alone for a caller that owns the device memory.
        dict(name="noalloc_fp64", kind="noalloc", N=32, K=16, M=16, m_p=1, alpha=1.25, Re=2000.0),
        # Proposals for one batch of search starts, and one gradient of the
        # training loss at the training batch size.
        dict(name="net_forward", kind="forward", cin=720, hidden=384, L=48, B=12),
        dict(name="net_gradients", kind="gradients", cin=720, hidden=384, L=48, B=64),
    ]


def _smooth(rng, lo, hi):
    """A size in lo..hi, spread over its logarithm, with no prime factor above 5."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    sizes = {2 ** a * 3 ** b * 5 ** c for a in range(8) for b in range(5) for c in range(4)}
    return min((k for k in sizes if lo <= k <= hi), key=lambda k: (abs(math.log(k / x)), k))


def _dt(N, M):
    """A time step that the near-axis spacing of the resolution allows."""
    return min(0.01, 0.01 * (16 / M) * (32 / N) ** 2)


def _cost(case):
    """Grid points times steps, FP64 counted three times."""
    if "shapes" in case:
        points = sum(math.prod(int(x) for x in g.split("x")) for g in case["shapes"].split())
    else:
        points = case.get("N", 0) * case.get("K", 0) * case.get("M", 0)
    return points * case.get("steps", 1) * (1 if case.get("precision", 0) else 3)


def draw(rng):
    while True:  # no more work than the large run
        case = _draw(rng)
        if _cost(case) <= 4_000_000:
            return case


def _draw(rng):
    kind = rng.choice(["step"] * 5 + ["ens"] * 2 + ["host", "noalloc", "forward", "gradients"])
    if kind in ("forward", "gradients"):
        return dict(kind=kind, cin=8 * rng.randint(30, 90), hidden=8 * rng.randint(16, 64), L=rng.randint(24, 64),
                    B=int(math.exp(rng.uniform(math.log(4), math.log(96)))))
    alpha = round(rng.uniform(0.4, 1.7), 3)
    if kind == "noalloc":
        N, K, M = rng.randint(16, 40), _smooth(rng, 4, 18), _smooth(rng, 4, 16)
        return dict(kind=kind, N=N, K=K, M=M, m_p=rng.randint(1, 3), alpha=alpha, Re=round(rng.uniform(300, 4000), 1))
    if kind == "ens":
        groups = []
        for _ in range(rng.randint(1, 3)):
            N = int(math.exp(rng.uniform(math.log(20), math.log(64))))
            groups.append((rng.randint(2, 12), N, _smooth(rng, 6, 32), _smooth(rng, 6, 32)))
        groups = [g for i, g in enumerate(groups) if g[1:] not in [h[1:] for h in groups[:i]]]
        dt = round(min(_dt(g[1], g[3]) for g in groups), 7)
        return dict(kind=kind, shapes=" ".join("%dx%dx%dx%d" % g for g in groups), m_p=rng.randint(1, 2), alpha=alpha,
                    Re=1800.0, Re2=rng.choice([1800.0, 2600.0]), dt=dt, dt2=dt, precision=rng.randint(0, 1),
                    steps=rng.randint(2, 4))
    N = int(math.exp(rng.uniform(math.log(16), math.log(112))))
    K, M = _smooth(rng, 4, 100), _smooth(rng, 4, 100)
    m_p = rng.choice([1, 1, 2, 3, 4])
    c = dict(kind=kind, N=N, K=K, M=M, m_p=m_p, alpha=alpha, Re=round(rng.uniform(500, 6000), 1),
             dt=round(_dt(N, M * m_p), 7), precision=rng.randint(0, 1))
    if kind == "host":
        return dict(c, precision=0, steps=1)
    return dict(c, steps=2 if N * K * M > 60000 else rng.randint(2, 4) * (2 - c["precision"]), rot=rng.choice([0.0, 0.0, 0.5]),
                force=rng.choice([0.0, 0.0, 0.05]), cfl=0.0)


# ------------------------------------------------------------------ inputs


def _gen(seed, salt=0):
    g = torch.Generator()
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _points(N):
    n = torch.arange(1, N + 1, dtype=torch.float64)
    r = torch.cos(math.pi * (N - n) / (2 * N - 1))
    r[-1] = 1.0
    return r


def _perturbation(N, K, M, m_p, alpha, gen):
    """A divergence-free broadband perturbation (3, M, 2K-1, N) of rms about 1
    that vanishes at the wall and is regular on the axis: per mode
    u+ = a r^(m~+1) s, u- = b r^|m~-1| s, s = (1 - r^2)^2, u_z from
    continuity; for k = 0 a streamfunction."""
    dev = _dev()
    nk = 2 * K - 1
    draws = torch.randn(4, M, nk, 2, dtype=torch.float64, generator=gen).to(dev)
    a, b, c, e = (torch.view_as_complex(draws[i].contiguous())[..., None] for i in range(4))
    r = _points(N).to(dev)
    s, ds = (1 - r * r) ** 2, -4 * r * (1 - r * r)
    k = torch.arange(-(K - 1), K, dtype=torch.float64, device=dev)[None, :, None]
    mt = (m_p * torch.arange(M, dtype=torch.float64, device=dev))[:, None, None]
    q = (mt - 1).abs()
    up, um = a * r ** (mt + 1) * s, b * r ** q * s
    pp = a * ((2 * mt + 2) * r ** (mt + 1) * s + r ** (mt + 2) * ds)
    pm = b * ((q + 1 - mt) * r ** q * s + r ** (q + 1) * ds)
    kz = torch.where(k == 0, torch.ones_like(k), k)
    U = torch.stack([0.5 * (up + um), -0.5j * (up - um), 0.5j / (alpha * kz * r) * (pp + pm)])
    psi, dpsi = c * r ** mt * s, c * (mt * r ** (mt - 1) * s + r ** mt * ds)
    flat = torch.stack([1j * mt * psi / r, -dpsi, e * r ** mt * s])
    U[:, :, K - 1] = flat[:, :, K - 1]
    mean = torch.stack([0 * r, e[0, K - 1].real * r * (1 - r * r), c[0, K - 1].real * (1 - r * r) * (1 - 3 * r * r)])
    U[:, 0, K - 1] = mean.to(U.dtype)
    U = U * torch.exp(-6 * (k.abs() / K + (mt / m_p) / M))
    U[:, 0, :K - 1] = torch.conj(torch.flip(U[:, 0, K:], [1]))
    w = torch.full((M, 1, 1), 2.0, dtype=torch.float64, device=dev)
    w[0] = 1.0
    f = torch.cat([torch.zeros(1, dtype=torch.float64, device=dev), (U.abs() ** 2 * w).sum((0, 1, 2)) * r])
    x = torch.cat([torch.zeros(1, dtype=torch.float64, device=dev), r])
    return U / torch.sqrt(2 * torch.trapezoid(f, x))


def _state(N, K, M, m_p, alpha, amplitude, gen):
    """Hagen-Poiseuille flow plus a perturbation of the given rms."""
    U = amplitude * _perturbation(N, K, M, m_p, alpha, gen)
    r = _points(N).to(U.device)
    U[2, 0, K - 1] += 1 - r * r
    return U.contiguous()


def _force(case, N, K, M):
    """A steady axial body force (1 - r^2) r cos(alpha z + m_p theta) / 2."""
    f = torch.zeros(3, M, 2 * K - 1, N, dtype=torch.complex128)
    r = _points(N)
    f[2, 1, K] = 0.5 * case["force"] * (1 - r * r) * r
    return f


def _members(case):
    """(N, K, M, Re, dt) of every trajectory of an ensemble."""
    shapes = [tuple(int(x) for x in g.split("x")) for g in case["shapes"].split()]
    out = [g[1:] for g in shapes for _ in range(g[0])]
    n = max(1, len(out) - 1)
    return [(N, K, M, case["Re"] + (case["Re2"] - case["Re"]) * i / n, case["dt"] + (case["dt2"] - case["dt"]) * i / n)
            for i, (N, K, M) in enumerate(out)]


def _ens_states(case, seed):
    """Start states, stacked per shape in the members' order."""
    gen = _gen(seed)
    groups = {}
    for N, K, M, _, _ in _members(case):
        amp = 10.0 ** (-3 + 2 * float(torch.rand(1, generator=gen)))
        groups.setdefault((N, K, M), []).append(_state(N, K, M, case["m_p"], case["alpha"], amp, gen))
    return [torch.stack(v) for v in groups.values()]


def _net_inputs(case, seed):
    """Parameters (flat, the library's order), features and targets of the proposal network."""
    gen = _gen(seed)
    cin, H, L, B, O = case["cin"], case["hidden"], case["L"], case["B"], 3
    sizes = [(H * 3 * cin, 3 * cin), (H, 0), (H * 3 * H, 3 * H), (H, 0), (cin * 3 * H, 3 * H), (cin, 0), (O * H, H), (O, 0)]
    flat = [(2 * torch.rand(n, generator=gen) - 1) / math.sqrt(fan) if fan else 0.02 * torch.randn(n, generator=gen)
            for n, fan in sizes]
    rows = torch.exp(-0.01 * torch.arange(cin))
    x = torch.randn(B, L, cin, generator=gen) * rows
    ty = 0.3 * torch.randn(B, L, cin, generator=gen) * rows
    tz = torch.rand(B, O, generator=gen)
    return torch.cat(flat).numpy(), x.to(_dev()), ty.to(_dev()), tz.to(_dev())


# ------------------------------------------------------------------ the cases


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind in ("forward", "gradients"):
        params, s.x, s.ty, s.tz = _net_inputs(case, seed)
        s.net = opf.opf_net_create(case["cin"], case["hidden"], case["L"], 3, seed=1)
        opf.opf_net_set_params(s.net, params)
        s.y, s.z = torch.empty_like(s.x), torch.empty_like(s.tz)
    elif kind == "ens":
        mem = _members(case)
        n = len(mem)
        s.states = _ens_states(case, seed)
        s.out = [torch.empty_like(v) for v in s.states]
        s.inp = [v[i].data_ptr() for v in s.states for i in range(len(v))]
        s.outp = [v[i].data_ptr() for v in s.out for i in range(len(v))]
        s.ens = opf.opf_ens_create([m[0] for m in mem], [m[1] for m in mem], [m[2] for m in mem], [case["m_p"]] * n,
                                   [case["alpha"]] * n, [m[3] for m in mem], [m[4] for m in mem])
        opf.opf_ens_set_option(s.ens, "precision", case["precision"])
    else:
        dims = (case["N"], case["K"], case["M"], case["m_p"], case["alpha"])
        s.state = _state(*dims, 0.1, _gen(seed))
        s.out = torch.empty_like(s.state)
        if kind != "noalloc":
            s.h = opf.opf_create(*dims, case["Re"], case["dt"])
            opf.opf_set_option(s.h, "precision", case["precision"])
        if kind == "host":
            s.pin = [v.cpu().pin_memory() for v in (s.state, s.out)]
            s.host = [v.numpy() for v in s.pin]
            del s.state, s.out
        if kind == "step":
            if case["rot"]:
                opf.opf_set_option(s.h, "rot_z", case["rot"])
            if case["force"]:
                opf.opf_set_forcing(s.h, _force(case, *dims[:3]).numpy())
            if case["cfl"]:
                opf.opf_set_option(s.h, "cfl", case["cfl"])
                opf.opf_set_option(s.h, "dt_max", case["dt"])
    if torch.cuda.is_available():
        torch.cuda.synchronize()  # the library works on streams of its own
    return s


def _device(call, ens, i, ptr):
    """The C entry points that move one trajectory's state within the GPU."""
    if call(ctypes.c_void_p(ens.ptr), i, ctypes.c_void_p(ptr)):
        raise RuntimeError(opf.lib().opf_last_error().decode())


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "step":
        opf.opf_set_state_device(s.h, s.state.data_ptr())
        opf.opf_step(s.h, case["steps"])
        opf.opf_get_state_device(s.h, s.out.data_ptr())
        return s.out
    if kind == "host":
        opf.opf_set_state(s.h, s.host[0])
        opf.opf_step(s.h, case["steps"])
        return opf.opf_get_state(s.h, s.host[1]), opf.opf_energy(s.h)
    if kind == "ens":
        for i, p in enumerate(s.inp):
            _device(opf.lib().opf_ens_set_state_device, s.ens, i, p)
        opf.opf_ens_step(s.ens, case["steps"])
        for i, p in enumerate(s.outp):
            _device(opf.lib().opf_ens_get_state_device, s.ens, i, p)
        return s.out
    if kind == "noalloc":
        opf.opf_nonlinear_noalloc(case["N"], case["K"], case["M"], case["m_p"], case["alpha"], case["Re"],
                                  s.state.data_ptr(), s.out.data_ptr())
        return s.out
    if kind == "forward":
        opf.opf_net_forward(s.net, s.x.data_ptr(), case["B"], s.y.data_ptr(), s.z.data_ptr())
        return s.y, s.z
    loss = opf.opf_net_gradients(s.net, s.x.data_ptr(), s.ty.data_ptr(), s.tz.data_ptr(), case["B"], 1.0)
    return loss, opf.opf_net_get_params(s.net, grads=True)


def _step_work(N, K, M, m_p, steps):
    """One pass of n steps: the state in and out and the radial factors once;
    two nonlinear evaluations and two solves a step."""
    nk, nz, nth = 2 * K - 1, 3 * K, 3 * M
    F, n = M * N * nk, nz * nth
    transforms = 9 * N * 2.5 * n * (math.log2(nz) + math.log2(nth)) + 9 * N * n
    solve = nk * M * N * (48 + 36 + 30 + 36 + 8 * 17)
    return {"bytes": 96 * F + K * M * N * 8 * (4 * 9 + 6), "flops": 2 * steps * (102 * F + transforms + solve)}


def work(case):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        cin, H, L, B = case["cin"], case["hidden"], case["L"], case["B"]
        w = 3 * (2 * cin * H + H * H)
        fwd = 2 * B * L * w
        if kind == "forward":
            return {"bytes": 4 * w + 8 * B * L * cin, "flops": fwd}
        return {"bytes": 8 * w + 8 * B * L * cin, "flops": 3 * fwd - 2 * B * L * 3 * cin * H}
    if kind == "ens":
        each = [_step_work(m[0], m[1], m[2], case["m_p"], case["steps"]) for m in _members(case)]
        return {q: sum(e[q] for e in each) for q in ("bytes", "flops")}
    N, K, M = case["N"], case["K"], case["M"]
    if kind == "noalloc":
        nk, n = 2 * K - 1, 9 * K * M
        F = M * N * nk
        return {"bytes": 96 * F, "flops": 102 * F + 9 * N * 2.5 * n * math.log2(n) + 9 * N * n}
    return _step_work(N, K, M, case["m_p"], case["steps"])


# ------------------------------------------------------------------ exact: plain 64-bit torch


@functools.lru_cache(maxsize=None)
def _radial(N):
    """Points, 9-point first / second derivative matrices per axis parity
    (even, odd) and the weights of int f r dr, in long double, then double."""
    L = np.longdouble
    r = np.cos(np.pi * (N - np.arange(1, N + 1)) / (2 * N - 1)).astype(L)
    r[-1] = 1
    ext = np.concatenate([-r[::-1], r])
    D = np.zeros((2, 2, N, N), dtype=L)
    wq = np.zeros(N, dtype=L)
    gx, gw = np.polynomial.legendre.leggauss(10)
    for n in range(N):
        first = min(N + n - 4, 2 * N - 9)
        x = ext[first:first + 9]
        # monomial coefficients of the Lagrange basis about r_n, scaled to the stencil's width
        h = np.max(np.abs(x - r[n]))
        t = (x - r[n]) / h
        lo, hi = (L(0) if n == 0 else r[n - 1]), r[n]
        g = ((hi - lo) / 2 * gx + (hi + lo) / 2 - r[n]) / h
        for i in range(9):
            p = np.ones(1, dtype=L)
            for j in range(9):
                if j != i:
                    p = np.convolve(p, np.array([-t[j], 1], dtype=L)) / (t[i] - t[j])
            col = first + i - N if first + i >= N else N - 1 - first - i
            for par, sign in enumerate((1, -1)):
                f = 1 if first + i >= N else sign
                D[par, 0, n, col] += f * p[1] / h
                D[par, 1, n, col] += f * 2 * p[2] / h ** 2
            wq[col] += np.sum((hi - lo) / 2 * gw * sum(p[q] * g ** q for q in range(9))) * x[i]
    dev = _dev()
    to = lambda v: torch.from_numpy(v.astype(np.float64)).to(dev)
    return to(r), to(D), to(wq)


class _Exact:
    """The time step in plain 64-bit torch: torch.fft on the 3K x 3M grid,
    dense LU per Fourier mode."""

    def __init__(self, N, K, M, m_p, alpha, Re, dt=None, rot=0.0, force=None):
        self.N, self.K, self.M, self.Re, self.dt, self.rot, self.force = N, K, M, Re, dt, rot, force
        self.r, self.D, self.wq = _radial(N)
        dev = self.r.device
        self.mt = m_p * torch.arange(M, device=dev)
        self.ak = (alpha * torch.arange(-(K - 1), K, dtype=torch.float64, device=dev))[None, :, None]
        self.mr = self.mt.to(torch.float64)[:, None, None] / self.r
        self.par = self.mt % 2  # of u_z and p; the others have the opposite one
        if dt is not None:
            self.factor()

    def d1(self, A, par):
        D = self.D[par, 0].to(A.dtype)  # (M, N, N)
        return A @ D.transpose(1, 2)

    def curl(self, U):
        ur, ut, uz = U
        return torch.stack([1j * (self.mr * uz - self.ak * ut), 1j * self.ak * ur - self.d1(uz, self.par),
                            self.d1(ut, 1 - self.par) + ut / self.r - 1j * self.mr * ur])

    def synth(self, A):  # (3, M, 2K-1, N) -> (3, 3M, 3K, N)
        Z = torch.zeros(A.shape[:2] + (3 * self.K, self.N), dtype=A.dtype, device=A.device)
        Z[:, :, :self.K] = A[:, :, self.K - 1:]
        Z[:, :, 2 * self.K + 1:] = A[:, :, :self.K - 1]
        return torch.fft.irfft(torch.fft.ifft(Z, dim=2, norm="forward"), n=3 * self.M, dim=1, norm="forward")

    def nonlinear(self, U):
        u, w = self.synth(U), self.synth(self.curl(U))
        n = torch.linalg.cross(u, w, dim=0)
        if self.rot:
            n[0] += 2 * self.rot * u[1]
            n[1] -= 2 * self.rot * u[0]
        A = torch.fft.fft(torch.fft.rfft(n, dim=1, norm="forward")[:, :self.M], dim=2, norm="forward")
        A = torch.cat([A[:, :, 2 * self.K + 1:], A[:, :, :self.K]], dim=2)
        A[2, 0, self.K - 1] += 4.0 / self.Re
        return A if self.force is None else A + self.force

    def factor(self):
        N, K, M, dev = self.N, self.K, self.M, self.r.device
        eye = torch.eye(N, dtype=torch.float64, device=dev)
        ak2 = (self.ak[0, K - 1:, 0] ** 2)[:, None, None, None]  # (K, 1, 1, 1)

        def op(j, par, diag, coef, wall):
            lap = self.D[par, 1] + self.D[par, 0] / self.r[:, None]  # (M, N, N)
            d = diag + coef * (-(j.to(torch.float64)[:, None] ** 2) / self.r ** 2 - ak2[..., 0])  # (K, M, N)
            A = coef * lap + d[..., None] * eye
            A[:, :, -1] = wall
            return A

        c = 0.5
        H = [op(j, j.abs() % 2, 1.0 / self.dt, -c / self.Re, eye[-1]) for j in (self.mt + 1, self.mt - 1, self.mt)]
        P = op(self.mt, self.par, 0.0, 1.0, self.D[self.par, 0][:, -1])
        P[0, 0, -1] = eye[-1]
        self.H = [torch.linalg.lu_factor(A) for A in H]
        del H
        self.P = torch.linalg.lu_factor(P)
        del P
        e = torch.zeros(K, M, N, 1, dtype=torch.float64, device=dev)
        e[:, :, -1] = 1.0
        self.p1 = self.spread(torch.linalg.lu_solve(*self.P, e))
        self.B = torch.stack(self.velocities([-g for g in self.grad(self.p1)], 0.0))
        self.B[:, 0, K - 1] = 0.0
        one = torch.ones(M, 2 * K - 1, N, dtype=torch.complex128, device=dev)
        self.G = self.solve(self.H[2], self.walled(one, 0.0))[0, K - 1].real
        self.sumG = (self.wq * self.G).sum()

    def spread(self, x):  # (K, M, N, 1) -> complex (M, 2K-1, N)
        x = x[..., 0].permute(1, 0, 2)
        return torch.cat([torch.flip(x[:, 1:], [1]), x], 1).to(torch.complex128)

    def solve(self, lu, b):  # b: (M, 2K-1, N) complex
        K = self.K
        pos, neg = b[:, K - 1:], torch.flip(b[:, :K], [1])
        cols = torch.stack([pos.real, pos.imag, neg.real, neg.imag], -1).permute(1, 0, 2, 3).contiguous()
        x = torch.linalg.lu_solve(*lu, cols).permute(1, 0, 2, 3)
        return torch.cat([torch.flip(torch.complex(x[..., 2], x[..., 3])[:, 1:], [1]), torch.complex(x[..., 0], x[..., 1])], 1)

    def walled(self, b, wall):
        b = b.clone()
        b[..., -1] = wall
        return b

    def velocities(self, b, walls):
        walls = [walls] * 3 if isinstance(walls, float) else walls
        return [self.solve(self.H[f], self.walled(b[f], walls[f])) for f in range(3)]

    def grad(self, p):  # +- form
        d = self.d1(p, self.par)
        return [d - self.mr * p, d + self.mr * p, 1j * self.ak * p]

    def div(self, a):  # +- form
        m = self.mt.to(torch.float64)[:, None, None]
        return (0.5 * self.d1(a[0] + a[1], 1 - self.par) + 0.5 * ((1 + m) * a[0] + (1 - m) * a[1]) / self.r
                + 1j * self.ak * a[2])

    def solve_pass(self, U, Nl):
        """(1/dt - cL) u = (1/dt + (1-c)L) u_j + N - grad p with no slip, zero
        wall divergence and fixed flux, c = 1/2."""
        pm = lambda A: [A[0] + 1j * A[1], A[0] - 1j * A[1], A[2]]
        u, n, K = pm(U), pm(Nl), self.K
        p = self.solve(self.P, self.walled(self.div(n), 0.0))
        g = self.grad(p)
        walls = [u[f][..., -1].clone() for f in range(3)]
        for w in walls:
            w[0, K - 1] = 0.0
        v = self.velocities([2.0 / self.dt * u[f] + n[f] - g[f] for f in range(3)], walls)
        v = [v[f] - u[f] for f in range(3)]
        ref = self.div(self.B)[..., -1].clone()
        ref[0, K - 1] = 1.0
        a = (self.div(v)[..., -1] / ref)[..., None]
        a[0, K - 1] = 0.0
        v = [v[f] - a * self.B[f] for f in range(3)]
        self.beta = (0.25 - (self.wq * v[2][0, K - 1].real).sum()) / self.sumG
        v[2][0, K - 1] += self.beta * self.G
        return torch.stack([0.5 * (v[0] + v[1]), -0.5j * (v[0] - v[1]), v[2]])

    def energy(self, U):
        """E, I and D over their laminar values."""
        w = self.wq * torch.where(torch.arange(self.M, device=U.device) == 0, 1.0, 2.0)[:, None, None]
        E, D = (float((w * A.abs() ** 2).sum()) for A in (U, self.curl(U)))
        flux = (self.wq * U[2, 0, self.K - 1].real).sum()
        return np.array([6 * E, float(4 * (1 + self.beta * self.Re / 4) * flux), D])

    def steps(self, U, n):
        for _ in range(n):
            Nj = self.nonlinear(U)
            U1 = self.solve_pass(U, Nj)
            U = self.solve_pass(U, 0.5 * (self.nonlinear(U1) + Nj))
        return U


def _exact_net(case, seed):
    params, x, ty, tz = _net_inputs(case, seed)
    cin, H, O = case["cin"], case["hidden"], 3
    p = torch.from_numpy(params).to(x.device).double().requires_grad_(True)
    parts = torch.split(p, [H * 3 * cin, H, H * 3 * H, H, cin * 3 * H, cin, O * H, O])
    conv = lambda v, w, b, ci: torch.nn.functional.conv1d(v, w.view(-1, 3, ci).permute(0, 2, 1), b, padding=1)
    gelu = torch.nn.functional.gelu
    h = gelu(conv(x.double().transpose(1, 2), parts[0], parts[1], cin))
    h = gelu(conv(h, parts[2], parts[3], H))
    y = conv(h, parts[4], parts[5], H).transpose(1, 2)
    z = h.mean(2) @ parts[6].view(O, H).T + parts[7]
    if case["kind"] == "forward":
        return y.detach(), z.detach()
    loss = ((y - ty) ** 2).mean() + ((z - tz) ** 2).mean()
    loss.backward()
    return float(loss), p.grad


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        return _exact_net(case, seed)
    if kind == "ens":
        mem, out, i = _members(case), [], 0
        for stack in _ens_states(case, seed):
            got = []
            for U in stack:
                N, K, M, Re, dt = mem[i]
                got.append(_Exact(N, K, M, case["m_p"], case["alpha"], Re, dt).steps(U, case["steps"]))
                i += 1
            out.append(torch.stack(got))
        return out
    dims = (case["N"], case["K"], case["M"], case["m_p"], case["alpha"])
    U = _state(*dims, 0.1, _gen(seed))
    if kind == "noalloc":
        return _Exact(*dims, case["Re"]).nonlinear(U)
    force = _force(case, *dims[:3]).to(U.device) if case.get("force") else None
    e = _Exact(*dims, case["Re"], case["dt"], case.get("rot", 0.0), force)
    U = e.steps(U, case["steps"])
    return U if kind == "step" else (U.cpu().numpy(), e.energy(U))
