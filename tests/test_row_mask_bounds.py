"""The y-interval of a plane section clipped by a brick's nearer x face (the adjoint's row mask),
checked by brute force in 64 bits (CPU only): in section coordinates y = yc + hw s and x = xc +
hw (c1 s -+ beta sqrt(1 - s^2)), beta^2 = Pyy / a, the part with |x| <= X on the section's side of the
brick centre spans s in [s0, s1], s0 and s1 being +-1 or (A c -+ beta sqrt(lam^2 - A^2)) / lam^2 with
A = (X - |xc|) / hw, c = sign(xc) c1, lam^2 = beta^2 + c1^2."""
import numpy as np

from test_cull_bounds import HALF_LOG2E, T, _random_sigma, _row_form


def _interval(xc, hw, c1, beta, X):
    lam2 = beta * beta + c1 * c1
    A, c = (X - abs(xc)) / hw, np.copysign(1.0, xc) * c1
    t = beta * np.sqrt(max(lam2 - A * A, 0.0)) / lam2
    e = A * c / lam2
    s1 = e + t if c > A and e + t < 1.0 else 1.0
    s0 = e - t if -c > A and e - t > -1.0 else -1.0
    return s0, s1


def test_clipped_section_interval():
    rng = np.random.default_rng(5)
    clipped = 0
    for _ in range(400):
        sigma = _random_sigma(rng)
        a, c1, c2, pyy, p2yz, pzz = _row_form(HALF_LOG2E * np.linalg.inv(sigma))
        kappa = pzz - p2yz ** 2 / (4 * pyy)
        dz = rng.uniform(-0.99, 0.99) * np.sqrt(T / kappa)
        hw, beta = np.sqrt((T - kappa * dz * dz) / pyy), np.sqrt(pyy / a)
        lam = np.hypot(beta, c1)
        X = rng.uniform(0.5, 8.0)
        # centres from the middle of the brick to where the section only just reaches it
        xc = rng.uniform(-1.0, 1.0) * (X + 0.999 * hw * lam)
        s0, s1 = _interval(xc, hw, c1, beta, X)
        s = np.linspace(-1.0, 1.0, 20001)
        r = beta * np.sqrt(1.0 - s * s)
        lo, hi = xc + hw * (c1 * s - r), xc + hw * (c1 * s + r)
        # the nearer face alone, on which the interval is exact
        near = lo <= X if xc >= 0 else hi >= -X
        assert near.any()
        assert s[near].min() >= s0 - 1e-9 and s[near].max() <= s1 + 1e-9
        assert s[near].min() <= s0 + 2e-3 and s[near].max() >= s1 - 2e-3  # attained
        # and a superset of the rows that meet the brick
        both = (lo <= X) & (hi >= -X)
        assert not both.any() or (s[both].min() >= s0 - 1e-9 and s[both].max() <= s1 + 1e-9)
        clipped += s0 > -1.0 or s1 < 1.0
    assert clipped > 100
