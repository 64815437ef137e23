"""The scaled Newton-Schulz steps of the global path's inverse square root, in FP64 on the host: with
eigenvalues x^2 of P a step maps x -> x (a - b x^2), a = 3 rho / 2, b = rho^3 / 2,
rho^2 = min(2.5, 3 / (1 + l + l^2)) while the lower bound l of x is below 0.94, else rho = 1.

Checked: every step keeps [l, 1] inside [l', 1]; an eigenvalue above 1 by 1e-3 (rounding) stays positive;
from any conditioning up to 1e6 one plain step behind the scaled ones leaves 1 - x^2 < 1e-2; and the
iteration on matrices gives A^(-1/2)."""

import numpy as np
import pytest


def first(s):
    l2 = 2.5 / s
    return min(0.5 * np.sqrt(l2) * (3 - l2), 0.395)


def step(l):
    if l >= 0.94:
        return 1.5, 0.5, l * (1.5 - 0.5 * l * l), True
    r2 = min(2.5, 3 / (1 + l + l * l))
    a, b = 1.5 * np.sqrt(r2), 0.5 * r2 ** 1.5
    return a, b, min(l * (a - b * l * l), a - b), False


@pytest.mark.parametrize("s", [16.0, 25.0, 40.0, 300.0, 1e4, 1e6])
def test_bounds_hold_and_converge(s):
    x = np.sqrt(np.linspace(2.5 / s, 2.5, 20001))
    x = x * (1.5 - 0.5 * x * x)
    l, plain = first(s), False
    while not plain:
        assert x.min() >= l * (1 - 1e-12) and x.max() <= 1 + 1e-12
        a, b, l, plain = step(l)
        assert a - b * (1 + 1e-3) > 0
        x = x * (a - b * x * x)
    assert (1 - x * x).max() < 1e-2


@pytest.mark.parametrize("m,scale", [(60, 4.0), (200, 20.0)])
def test_matrix_iteration(m, scale):
    rng = np.random.default_rng(m)
    Y = scale * rng.standard_normal((3 * m, m)) * np.geomspace(1, 0.05, m)
    Y -= Y.mean(axis=1, keepdims=True)
    A = np.eye(m) + Y.T @ Y / (m - 1)
    s = 1 + np.linalg.norm(Y.T @ Y) / (m - 1)
    B = A * 2.5 / s
    Z = 1.5 * np.eye(m) - 0.5 * B
    Yk, l = B @ Z, first(s)
    for _ in range(40):
        P = Z @ Yk
        a, b, l, plain = step(l)
        T = a * np.eye(m) - b * P
        Yk, Z = Yk @ T, T @ Z
        if plain and np.abs(P - np.eye(m)).max() < 1e-12:
            break
    w, V = np.linalg.eigh(B)
    ref = (V / np.sqrt(w)) @ V.T
    assert np.abs(Z - ref).max() < 1e-9 * np.abs(ref).max()
