"""The FP64 evaluation's three forms of the closed form (general, middle distances, far) at the
distances where they meet, against the oracle: one element of each kind with unit density.

The forms change where the largest x = len / (R_a + R_b) over the edges reaches 1/2 and 1/8.
Tolerance (derived before the first run): the oracle's corner terms (magnitude up to about 10 r,
rounded to 2^-53) cancel down to A / r, so its relative error grows like 1e-15 (r / l)^2 with l
the shortest edge; a hundred times that, plus 1e-13, bounds the difference."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 1e-4
SHAPES = {
    "square": (I.KIND_RECT, [[0, 0, 0], [U, 0, 0], [U, 0, U], [0, 0, U]]),
    "strip": (I.KIND_RECT, [[0, 0, 0], [U, 0, 0], [U, 0, 0.1 * U], [0, 0, 0.1 * U]]),
    "triangle": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [0.3 * U, 0, 0.8 * U]]),
    "obtuse": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [1.6 * U, 0, 0.3 * U]]),
    "quad": (I.KIND_QUAD, [[0, 0, 0], [U, 0, 0], [0.8 * U, 0, 0.9 * U], [0.1 * U, 0, 0.6 * U]]),
}


def _points(verts, target, gen):
    """Points whose largest x lies on both sides of `target` (1/2 or 1/8), in random directions,
    some of them in the element's plane or within 1e-6 of it."""
    v = np.array(verts, float)
    c, n = v.mean(axis=0), len(v)
    d = gen.normal(size=(40, 3))
    d[:8, 1] = 0.0
    d[8:14, 1] *= 1e-6
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    lens = [np.linalg.norm(v[(i + 1) % n] - v[i]) for i in range(n)]

    def worst(r, k):
        R = np.linalg.norm(v - (c + r * d[k]), axis=1)
        return max(lens[i] / (R[i] + R[(i + 1) % n]) for i in range(n))

    out = []
    for k in range(d.shape[0]):
        lo, hi = 0.0, 100 * U  # worst() falls through the target between them
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if worst(mid, k) > target else (lo, mid)
        out += [c + f * hi * d[k] for f in (0.9, 1 - 1e-9, 1 + 1e-9, 1.1)]
    return np.array(out)


@pytest.mark.parametrize("target", [0.5, 0.125])
@pytest.mark.parametrize("name", list(SHAPES))
def test_forms_meet(name, target):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    kind, verts = SHAPES[name]
    el = np.zeros(1, dtype=I.ELEMENT_DTYPE)
    el["kind"], el["eps_a"], el["eps_b"] = kind, 1.0, 1.0
    v = np.zeros((4, 3))
    v[: len(verts)] = verts
    el["v"] = v
    pts = _points(verts, target, np.random.default_rng(7))
    pts = np.concatenate([pts, pts.mean(axis=0) + 50 * U * np.random.default_rng(8).normal(size=(20, 3))])
    ctx = N.Context()
    N.nebem_set_geometry(ctx.h, el)
    ctx.n = 1
    ctx.set_sigma(np.ones(1))
    phi, E = ctx.eval(pts, N.NEBEM_FP64)
    ctx.close()
    ke = 1.0 / (4.0 * np.pi * 8.8541878128e-12)
    rphi, rE = O.influence(el, pts)
    rphi, rE = ke * rphi, ke * rE
    n = len(verts)
    short = min(np.linalg.norm(np.subtract(verts[(i + 1) % n], verts[i])) for i in range(n))
    r = np.linalg.norm(pts - np.mean(verts, axis=0), axis=1)
    tol = 1e-13 + 1e-13 * (r / short) ** 2
    assert (np.abs(phi - rphi) <= tol * np.abs(rphi)).all()
    assert (np.linalg.norm(E - rE, axis=1) <= tol * np.linalg.norm(rE, axis=1)).all()
