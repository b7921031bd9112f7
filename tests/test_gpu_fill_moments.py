"""Mixed fill: pairs from 32 (conductor rows) and 52 radii on (interface rows) by the source's moments, nearer
ones by Gauss nodes, against a 256-node rule; every kind of element as source, of 20 um, and scaled by
1e-5 and 1e5, rows of both kinds at the edges of the ranges, one copy, and 9 and 121 (an odd count leaves
half of the last packed step empty).  (The FP64 closed forms lose digits with the distance: 1.2e-11 of the
pair for the sliver at 1000 radii, so they are no reference here.)

Tolerance (derived before the first run), relative to the pair's own A / d or A / d^2: terms left
out 3e-13 at 32 radii and 8 x 3e-13 (32 / 52)^7 = 8e-14 at 52, falling; the FP32 terms 1.5e-6 x 1e-7 and
six times that; nodes 3e-12 and six times that; two-float sums 44 bits.  With copies the entries are
sums of pairs, of one sign for the potential, and the field's errors count to the sum of the pairs' A / d^2."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2e-5
SHAPES = {
    "triangle": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [0.3 * U, 0.1 * U, 0.8 * U]]),
    "sliver": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [0.1 * U, 0, 0.05 * U]]),
    "strip": (I.KIND_RECT, [[0, 0, 0], [U, 0, 0], [U, 0, 0.1 * U], [0, 0, 0.1 * U]]),
    "quad": (I.KIND_QUAD, [[0, 0, 0], [U, 0, 0], [0.8 * U, 0, 0.9 * U], [0.1 * U, 0, 0.6 * U]]),
}


def rule(v):
    """256 nodes and weights of a triangle (collapsed) or quadrilateral (bilinear)."""
    x, w = np.polynomial.legendre.leggauss(16)
    s, t = np.meshgrid(0.5 * (x + 1), 0.5 * (x + 1), indexing="ij")
    w = 0.25 * np.outer(w, w)
    s, t = s[..., None], t[..., None]
    if len(v) == 3:
        p, ds, dt = v[0] + s * (v[1] - v[0]) + t * (1 - s) * (v[2] - v[0]), v[1] - v[0], (1 - s) * (v[2] - v[0])
    else:
        e1, e3, tw = v[1] - v[0], v[3] - v[0], v[2] - v[1] - v[3] + v[0]
        p, ds, dt = v[0] + s * e1 + t * e3 + s * t * tw, e1 + t * tw, e3 + s * tw
    return p.reshape(-1, 3), (w * np.linalg.norm(np.cross(ds + 0 * s, dt + 0 * s), axis=-1)).ravel()


@pytest.mark.parametrize("half, scale", [(0, 1.0), (1, 1.0), (5, 1.0), (0, 1e-5), (0, 1e5)])
@pytest.mark.parametrize("name", list(SHAPES))
def test_fill_moments_against_fp64(name, half, scale):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    kind, verts = SHAPES[name][0], scale * np.array(SHAPES[name][1], float)
    cen = verts.mean(axis=0)
    rho = np.linalg.norm(verts - cen, axis=1).max()
    gen = np.random.default_rng(half)
    radii = np.repeat([20.0, 31.9, 32.1, 51.9, 52.1, 100.0, 1000.0], 20)
    d = gen.normal(size=(radii.size, 3))
    d[::5, 1] = 0.0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    at = cen + (radii * rho)[:, None] * d
    # element 0 is the source; small triangles elsewhere are the rows, every second one an interface
    el = np.zeros(1 + radii.size, dtype=I.ELEMENT_DTYPE)
    el["eps_a"], el["eps_b"] = 1.0, 1.0
    el["kind"] = I.KIND_TRI
    el["kind"][0] = kind
    el["v"][0, : len(verts)] = verts
    for i, p in enumerate(at):
        a, b = np.linalg.qr(gen.normal(size=(3, 3)))[0][:2] * 0.3 * rho
        el["v"][1 + i, :3] = [p, p + a, p + b] - (a + b) / 3
    el["bc"][1::2] = I.BC_DIELECTRIC
    el["eps_b"][1::2] = 4.0
    ctx = N.Context()
    lattice = scale * np.array([3000.0 * U, 0, 0, 0, 3000.0 * U, 0]) if half else None
    N.nebem_set_geometry(ctx.h, el, lattice, -half, half)
    ctx.n = el.size
    mixed = ctx.fill(N.NEBEM_MIXED)[1:, 0].copy()
    ctx.close()
    ke = 1.0 / (4 * np.pi * 8.8541878128e-12)
    k = np.arange(-half, half + 1) * 3000.0 * U * scale
    copies = np.array([[a, b, 0.0] for a in k for b in k])
    tri = el["v"][1:, :3]
    rows = tri.mean(axis=1)
    normal = np.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    normal /= np.linalg.norm(normal, axis=1, keepdims=True)
    iface = el["bc"][1:] == I.BC_DIELECTRIC
    nodes, weights = rule(verts)
    phi, field, size = np.zeros((3, radii.size))
    for t in copies:
        dist = rows[:, None] - t - nodes
        r = np.linalg.norm(dist, axis=-1)
        phi += ke * (weights / r).sum(1)
        field += ke * (weights * (dist * normal[:, None]).sum(-1) / r**3).sum(1)
        dc = np.linalg.norm(rows - t - cen, axis=1)
        size += ke * weights.sum() * np.where(iface, dc**-2.0, 1 / dc)
    near = radii < np.where(iface, 52, 32)
    tol = np.where(near, 3e-12, 1e-12) * np.where(iface, 6, 1)
    err = np.minimum(np.abs(mixed - field), np.abs(mixed + field))  # the normal's sign is the library's choice
    err = np.where(iface, err, np.abs(mixed - phi))
    assert (err <= tol * size).all()
