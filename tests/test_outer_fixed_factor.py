"""B^T p of the fixed-point outer Stokes kernel (csrc/outer.cuh) carries no rounding of a whole cell: its factor
112.5 h / mu and the last scaling mu h / 97200 are rounded numbers, but their product is h^2 / 864 (fix_factor). Host
runs of the kernel's phases with u = 0 and one viscosity, against exact sums (p are integers, so B^T p over h^2 / 216 is
one); measured is the part of the error along the result, sum(e y) / sum(y y), which a wrong factor shifts as a whole.

Tolerance 2^-53: each cell's share is rounded twice (53 bits, the scaling) and up to 3 partial sums are, each by at most
2^-53 of its value and with either sign: about 2^-53 a row (sqrt(5/3) 2^-53 for results near a power of two), averaged
over the 81 or 375 rows of the free nodes, of which at least 30 have a share, 0.2 x 2^-53; 5 of those standard deviations.
Two roundings of the factor and three of the scaling shift it by up to 4 x 2^-53 for some viscosities."""
from fractions import Fraction

import numpy as np
import pytest

import sinker_inputs as si
from oracle import mesh
from test_outer_fixed import apply_host  # noqa: F401  (fixture)

VP = [[1, 0], [2, 2], [0, 1]]        # 6 int l_m psi_v and 6 int l_m' psi_v on [0,1]
DP = [[-5, -1], [4, -4], [1, 5]]


def bt_integers(n, p):
    """-216 / h^2 B^T p on the free nodes, [3][M][M][M] (0 on the walls), for integers p [n+1]^3."""
    M = 2 * n + 1
    out = np.zeros((3, M, M, M), dtype=np.int64)
    for c in range(3):
        T = [np.array(DP if d == c else VP, dtype=np.int64) for d in range(3)]
        for k in range(n):
            for j in range(n):
                for i in range(n):
                    cell = np.einsum("ak,bj,ci,kji->abc", T[2], T[1], T[0], p[k:k + 2, j:j + 2, i:i + 2])
                    out[c, 2 * k:2 * k + 3, 2 * j:2 * j + 3, 2 * i:2 * i + 3] += cell
    free = np.zeros((M, M, M), dtype=bool)
    free[1:-1, 1:-1, 1:-1] = True
    return out * free


@pytest.mark.parametrize("n", [2, 3])
def test_pressure_gradient_has_no_error_of_the_factor(apply_host, n):  # noqa: F811
    m = mesh.Mesh(n)
    p = np.floor(si.uniform(91, m.n_p) * 2.0 ** 30).astype(np.int64)
    scale = -Fraction(1.0 / n) ** 2 / 216
    ref = bt_integers(n, p.reshape((n + 1,) * 3)).ravel()
    rows = np.flatnonzero(ref)
    exact = [scale * int(v) for v in ref[rows]]
    y = np.array([float(v) for v in exact])
    for mu in 10.0 ** si.uniform(92, 24, -3.0, 3.0):
        x = np.concatenate([np.zeros(m.n_u), p.astype(np.float64)])
        du, _ = apply_host(n, np.full(n ** 3, mu), x)
        e = np.array([float(Fraction(float(a)) - b) for a, b in zip(du[rows], exact)])
        assert abs(e @ y) <= 2.0 ** -53 * (y @ y), mu
