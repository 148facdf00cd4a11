"""Errors of the fused Burgers step and its adjoint element by element, each over the element's own
largest value, on rough fields whose patches of four elements differ in size and on waves
through zero: the steps hold an element in integers at a scale of its neighbourhood, which must
not cost a small element the accuracy that FP64 stages give it. Both are measured against the
same scheme in extended precision."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2404_03399_gb300 as adg  # noqa: E402

pytestmark = pytest.mark.gpu
X = np.longdouble   # 64 bits of significand or more
K, STEPS, SEEDS = 104, 20, 4
SHU_OSHER = ((X(0), X(1)), (X(3) / 4, X(1) / 4), (X(1) / 3, X(2) / 3))
TWO_N = {"rk2": ((0, 1), (-1, X(1) / 2)), "lsrk3": ((0, X(1) / 3), (X(-5) / 9, X(15) / 16), (X(-153) / 128, X(8) / 15))}


def _operators(p):
    """D and M^-1 on the Legendre-Gauss-Lobatto nodes."""
    s = {1: [], 2: [X(0)], 3: [-1 / np.sqrt(X(5)), 1 / np.sqrt(X(5))],
         4: [-np.sqrt(X(3) / 7), X(0), np.sqrt(X(3) / 7)]}[p]
    x = np.array([X(-1)] + s + [X(1)])
    L = [np.ones_like(x), x.copy()]
    dL = [np.zeros_like(x), np.ones_like(x)]
    for n in range(1, p):
        L.append(((2 * n + 1) * x * L[n] - n * L[n - 1]) / (n + 1))
        dL.append(dL[n - 1] + (2 * n + 1) * L[n])
    V = np.stack([L[n] * np.sqrt(X(2 * n + 1) / 2) for n in range(p + 1)], axis=1)
    dV = np.stack([dL[n] * np.sqrt(X(2 * n + 1) / 2) for n in range(p + 1)], axis=1)
    Mi = V @ V.T   # the modes are orthonormal: M^-1 = V V^T, and V^-1 = V^T M
    M = np.array([[_entry(x, i, j) for j in range(p + 1)] for i in range(p + 1)])
    return dV @ V.T @ M, M, Mi


def _entry(x, i, j):
    """The integral of l_i l_j over [-1, 1], from their coefficients."""
    def basis(m):
        c = np.array([X(1)])
        for k in range(len(x)):
            if k != m:
                c = np.convolve(c, np.array([X(1), -x[k]])) / (x[m] - x[k])
        return c
    c = np.convolve(basis(i), basis(j))[::-1]
    return sum(2 * c[n] / (n + 1) for n in range(0, len(c), 2))


class Scheme:
    """Synchronous inviscid Burgers in the arithmetic of `T`, with folded stage constants."""

    def __init__(self, T, p, dt, dx):
        D, self.M, Mi = _operators(p)
        c2 = -2 * X(dt) / X(dx)
        self.T, self.Np = T, p + 1
        self.A, self.l0, self.lp = c2 * D / 2, c2 * Mi[:, 0], -c2 * Mi[:, -1]

    def const(self, b):
        return [np.array(b * c, dtype=self.T) for c in (self.A, self.l0, self.lp)]

    def dtL(self, v, acc, b=X(1)):
        """acc + b dt L(v)."""
        A, l0, lp = self.const(b)
        h = self.T(0.5)
        um, up = np.roll(v[:, -1], 1), v[:, 0]
        F = h * (h * (um * um) + h * (up * up)) - h * np.maximum(abs(um), abs(up)) * (up - um)
        jl, jr = h * (up * up) - F, h * (v[:, -1] * v[:, -1]) - np.roll(F, -1)
        g = v * v
        for k in range(self.Np):
            acc = acc + A[None, :, k] * g[:, k, None]
        return acc + l0[None] * jl[:, None] + lp[None] * jr[:, None]

    def step(self, u, rk, rec=None):
        T = self.T
        if rk == "ssprk3":
            v = u
            for al, be in SHU_OSHER:
                if rec is not None:
                    rec.append(v)
                v = self.dtL(v, T(al) * u + T(be) * v, be)
            return v
        d, v = np.zeros_like(u), u
        for a, b in TWO_N[rk]:
            d = self.dtL(v, T(a) * d)
            v = v + T(b) * d
        return v


    def reverse(self, w, y):
        """The adjoint of an SSP-RK3 step's result to that of its input; y: its stage inputs."""
        T, acc = self.T, 0
        h = T(0.5)
        for s in (2, 1, 0):
            al, be = SHU_OSHER[s]
            (A, l0, lp), v = self.const(be), y[s]
            sl = sum(l0[i] * w[:, i] for i in range(self.Np))
            sr = sum(lp[i] * w[:, i] for i in range(self.Np))
            lv = T(be) * w + 2 * v * sum(A[i][None, :] * w[:, i, None] for i in range(self.Np))
            lv[:, 0] += v[:, 0] * sl
            lv[:, -1] += v[:, -1] * sr
            mu = -sl - np.roll(sr, 1)
            a, b = np.roll(v[:, -1], 1), v[:, 0]
            left = abs(a) >= abs(b)
            lam = np.where(left, abs(a), abs(b))
            gl = np.where(left, np.where(a >= 0, T(1), T(-1)), T(0))
            gr = np.where(left, T(0), np.where(b >= 0, T(1), T(-1)))
            lv[:, 0] += mu * (h * b - h * lam - h * gr * (b - a))
            lv[:, -1] += np.roll(mu * (h * a + h * lam - h * gl * (b - a)), -1)
            acc = acc + T(al) * w
            w = lv
        return acc + w


def _patches(rng, p, ratio):
    u = 0.7 + 0.28 * rng.uniform(-1.0, 1.0, (K, p + 1))
    return u * np.where((np.arange(K) // 4) % 2 == 0, 1.0, 1.0 / ratio)[:, None]


def _rms(got, ref):
    e = np.max(np.abs(got - ref), axis=1) / np.max(np.abs(ref), axis=1)
    return float(np.sqrt(np.mean((e * e).astype(np.float64))))


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("rk,ratio", [("ssprk3", 1.0), ("ssprk3", 8.0), ("ssprk3", 60.0), ("rk2", 1.0),
                                      ("rk2", 4.0), ("rk2", 25.0), ("lsrk3", 25.0)])
def test_elements_keep_the_accuracy_of_fp64_stages(rk, ratio, p):
    _compare(rk, ratio, p, 0.01, STEPS)


@pytest.mark.parametrize("rk,ratio,p", [("rk2", 4.0, 1), ("lsrk3", 4.0, 1), ("rk2", 1.0, 3), ("ssprk3", 4.0, 1)])
def test_roundings_do_not_add_up(rk, ratio, p):
    _compare(rk, ratio, p, 0.05 if p == 1 else 0.01, 200)


def _compare(rk, ratio, p, cfl, steps):
    # 1.25: the two errors are averages over some 400 elements each, equal where the step takes
    # FP64 itself, and the FP64 arithmetic here differs from the kernels' in its order
    dx = 2.0 * math.pi / K
    dt = cfl * dx
    got = ref = 0.0
    for seed in range(SEEDS):
        u0 = _patches(np.random.default_rng(seed), p, ratio)
        s = adg.Solver(adg.Config(pde="burgers", K=K, p=p, dt=dt, rk=rk), torch.tensor(u0, device="cuda"))
        s.step(steps)
        g = s.state().cpu().numpy()
        s.close()
        f, x = u0, u0.astype(X)
        fs, xs = Scheme(np.float64, p, dt, dx), Scheme(X, p, dt, dx)
        for _ in range(steps):
            f, x = fs.step(f, rk), xs.step(x, rk)
        got, ref = got + _rms(g.astype(X), x), ref + _rms(f.astype(X), x)
    assert got <= 1.25 * ref


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("field", [1.0, 8.0, 60.0, "wave"])
def test_gradient_elements_keep_the_accuracy_of_fp64_stages(field, p):
    # misfits of the final state in patches, or a wave through zero; 1.25 as above
    dx = 2.0 * math.pi / K
    dt = 0.01 * dx
    x = (np.arange(K)[:, None] + np.linspace(0.0, 1.0, p + 1)[None]) * dx
    got = ref = 0.0
    for seed in range(SEEDS):
        u0 = 0.5 + np.sin(x + seed)
        d = np.sin(3.0 * x + seed) if field == "wave" else _patches(np.random.default_rng(seed), p, field)
        s = adg.Solver(adg.Config(pde="burgers", K=K, p=p, dt=dt), torch.tensor(u0, device="cuda"))
        s.step(STEPS)
        end = s.state().cpu().numpy()
        s.close()
        target = end - d
        s = adg.Solver(adg.Config(pde="burgers", K=K, p=p, dt=dt), torch.tensor(u0, device="cuda"))
        g = s.grad(torch.tensor(target, device="cuda"), STEPS, STEPS)[1].cpu().numpy()
        s.close()
        fs, xs = Scheme(np.float64, p, dt, dx), Scheme(X, p, dt, dx)
        rec, u = [], u0.astype(X)
        for _ in range(STEPS):
            u = xs.step(u, "ssprk3", rec)
        w = ((end.astype(X) - target.astype(X)) @ xs.M) * (X(dx) / 2)
        f = w.astype(np.float64)
        for n in range(STEPS - 1, -1, -1):
            y = rec[3 * n:3 * n + 3]
            w, f = xs.reverse(w, y), fs.reverse(f, [v.astype(np.float64) for v in y])
        got, ref = got + _rms(g.astype(X), w), ref + _rms(f.astype(X), w)
    assert got <= 1.25 * ref
