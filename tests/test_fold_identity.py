"""The folded sums that the tensor-core operators evaluate equal Eq. (1) and its
adjoint: about the point half a pixel below pixel N/2 the grid is symmetric,
mirror pixels share |cos| and |sin| of their phases, and V is a rotation of four
real contractions over N/2 rows.  Plain numpy in FP64 against the oracle's
direct sums, at ordinary, degenerate and aliased frequencies."""
import numpy as np
import pytest

import oracle


def _freqs(N, dx, dy, seed):
    r = np.random.default_rng(seed)
    g = 1.0 / (N * dx)
    u = np.concatenate([[0, 0, 0.5 / dx, -0.5 / dx, 0.7 / dx, 3 * g, 1 / dx], r.uniform(-0.6, 0.6, 20) / dx])
    v = np.concatenate([[0, 0.5 / dy, 0, 3 * g, -0.7 / dy, 0, 1 / dy], r.uniform(-0.6, 0.6, 20) / dy])
    return u, v


def _half_tables(f, d, N):
    t = f * d
    t = t - np.rint(t)
    ph = -2 * np.pi * t[:, None] * (np.arange(N // 2) + 0.5)
    return np.cos(ph), np.sin(ph), np.exp(1j * np.pi * t)


@pytest.mark.parametrize("N", [2, 16, 64])
def test_folded_forward_and_adjoint(N):
    dx, dy = 3e-7, 4e-7
    u, v = _freqs(N, dx, dy, N)
    rng = np.random.default_rng(N + 1)
    B = rng.standard_normal((N, N))
    M = N // 2
    # mirror quadrants (first sign rows, second columns), from the centre outwards
    pp, pm = B[M:, M:], B[M:, :M][:, ::-1]
    mp, mm = B[:M, M:][::-1], B[:M, :M][::-1, ::-1]
    cx, sx, ex = _half_tables(u, dx, N)   # c + i y of the half-pixel grid, y = -sin
    cy, sy, ey = _half_tables(v, dy, N)
    Tss, Tsa = cy @ (pp + pm + mp + mm), cy @ (pp - pm + mp - mm)
    Tas, Taa = sy @ (pp + pm - mp - mm), sy @ (pp - pm - mp + mm)
    V = ex * ey * ((cx * Tss - sx * Taa).sum(1) + 1j * (sx * Tsa + cx * Tas).sum(1))
    ref = oracle.forward(N, dx, dy, u, v, B)
    assert np.max(np.abs(V - ref)) <= 1e-12 * np.max(np.abs(ref)) * N
    # adjoint: two real contractions D0, D1 over the half rows and all columns
    y = rng.standard_normal(u.size) + 1j * rng.standard_normal(u.size)
    t = u * dx
    P = (y / ey)[:, None] * np.exp(2j * np.pi * (t - np.rint(t))[:, None] * (np.arange(N) - M))
    D0, D1 = cy.T @ P.real, sy.T @ P.imag
    G = np.empty((N, N))
    G[M:], G[:M] = D0 + D1, (D0 - D1)[::-1]
    assert np.max(np.abs(G - oracle.adjoint(N, dx, dy, u, v, y))) <= 1e-11 * np.max(np.abs(G)) * N
