"""What rounding alone does to plain FP64 CG with a varying R, and to CG preconditioned by R: the same solve with
every entry of HA moved by half a unit in its last place. Plain CG takes some 90 steps here, its recurrences lose
their orthogonality, and where they stop (||r|| <= 1e-8 ||d||) depends on the last bits: the analyses
differ by up to what that tolerance leaves, whichever form evaluates them. Preconditioned CG, with some tens of
rows per member, ends before rounding matters. (The GPU library keeps one evaluation order for the former and chooses freely for the latter.)"""
import numpy as np

import synth


def _cg(HA, D, r, tol, precondition):
    N = HA.shape[1]
    minv = (1.0 / r if precondition else np.ones_like(r))[:, None]
    x, q = np.zeros_like(D), D.copy()
    z = minv * q
    p, g = z.copy(), (q * z).sum(0)
    stop = tol * np.linalg.norm(D, axis=0)
    act = np.ones(N, bool)
    steps = 0
    while act.any() and steps < 500:
        Sp = HA @ (HA.T @ p) / (N - 1) + r[:, None] * p
        a = np.where(act, g / (p * Sp).sum(0), 0.0)
        x += a * p
        q -= a * Sp
        act &= np.linalg.norm(q, axis=0) > stop
        z = minv * q
        g2 = (q * z).sum(0)
        p = z + np.where(act, g2 / g, 0.0) * p
        g = g2
        steps += 1
    return x, steps


def _increments(precondition):
    m, N = 4096, 64
    p = synth.grf_problem(128, 4.0, N, m, 0.5, 1.5, 11, dtype=np.float64)
    HA = p.Xf[p.col] - p.Xf[p.col].mean(1, keepdims=True)
    rng = np.random.default_rng(3)
    D = p.y[:, None] - p.Xf[p.col] + np.sqrt(p.r)[:, None] * rng.standard_normal((m, N))
    A = p.Xf - p.Xf.mean(1, keepdims=True)
    out = []
    for H in (HA, HA * (1.0 + 2.0 ** -53 * rng.choice([-1.0, 1.0], HA.shape)), HA * (1.0 + 2.0 ** -52 * (rng.random(HA.shape) < 0.5))):
        Z, steps = _cg(H, D, p.r, 1e-8, precondition)
        out.append(A @ (HA.T @ Z) / (N - 1))
    d = [np.linalg.norm(o - out[0]) / np.linalg.norm(out[0]) for o in out[1:]]
    return max(d), steps


def test_plain_cg_with_a_varying_r_depends_on_the_last_bits():
    d, steps = _increments(False)
    assert steps > 64 and 1e-10 < d < 1e-6, (d, steps)


def test_preconditioned_cg_does_not():
    d, steps = _increments(True)
    assert steps < 64 and d < 1e-12, (d, steps)
