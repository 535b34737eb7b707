"""The walk test's one rounding bound for the three weights: whenever it decides, the exact orientation
of the FP32 point agrees, and every decision it takes the three separate bounds take as well. Emulated
in numpy float32 like test_walk_bound, on thin and ordinary elements and points within ulps of edges."""
import numpy as np

from paper_1006_0549_gb300 import workloads as wl
from tests.test_walk_bound import coefficients, exact_signs, fast


def single(coef, px, py, fma):
    f = np.float32
    x0, y0, b1, g1, b2, g2 = coef
    dx, dy = f(f(px) - x0), f(f(py) - y0)
    t1, s1, t2, s2 = f(b1 * dx), f(g1 * dy), f(b2 * dx), f(g2 * dy)
    l1 = f(float(b1) * float(dx) + float(s1)) if fma else f(t1 + s1)
    l2 = f(float(b2) * float(dx) + float(s2)) if fma else f(t2 + s2)
    l0 = f(f(f(1.0) - l1) - l2)
    T = f(f(abs(t1) + abs(s1)) + f(abs(t2) + abs(s2)))
    E = f(float(f(4.6e-7)) * float(T) + float(f(1.55e-7)))
    lam = [l0, l1, l2]
    a = int(np.argmin(lam))
    if lam[a] > E:
        return "in", None
    return ("out", a) if lam[a] < -E else ("undecided", None)


def test_single_bound_decisions_are_certified():
    rng = np.random.default_rng(8)
    checked = decided = 0
    for mesh in (wl.channel_mesh(250, 100, 1006054902), wl.cavity_mesh(316, 316, 1006054903), wl.bump_channel_mesh(60, 24, 5)):
        for e in rng.choice(mesh.n_tri, 200, replace=False):
            xy = mesh.node_xy[mesh.tri[e]].astype(np.float64)
            coef = coefficients(xy)
            for _ in range(12):
                k = rng.integers(3)
                t = rng.choice([0.0, 1.0, rng.random(), rng.normal() * 3.0])     # on the edge, or along its line
                p = xy[k] + t * (xy[(k + 1) % 3] - xy[k])
                px, py = np.float32(p[0]), np.float32(p[1])
                for _ in range(int(rng.integers(0, 4))):
                    px = np.nextafter(px, np.float32(rng.choice([-1e9, 1e9])), dtype=np.float32)
                    py = np.nextafter(py, np.float32(rng.choice([-1e9, 1e9])), dtype=np.float32)
                signs = exact_signs(xy, px, py)
                for fma in (False, True):
                    decision, a = single(coef, px, py, fma)
                    checked += 1
                    if decision == "undecided":
                        continue
                    decided += 1
                    assert (decision, a) == fast(coef, px, py, fma)
                    if decision == "in":
                        assert min(signs) > 0, (e, px, py, signs)
                    else:
                        assert signs[a] < 0, (e, px, py, signs, a)
            px, py = np.float32(xy.mean(0)[0]), np.float32(xy.mean(0)[1])
            assert single(coef, px, py, False)[0] == "in"
    assert decided > checked // 5
