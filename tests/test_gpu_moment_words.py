"""Stored words of the moment-space formats after one pass of two or three steps, against the same
pass taken level by level in NumPy: populations rebuilt once, FP32 node updates, moments stored once.
Every operation is a single FP32 rounding, so the words are equal (0 and -0 count as equal)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
F = np.float32
SIGN = np.array([-1, -1, 1, 1, 1], F)[:, None, None]


def fma(a, b, c):
    """a b + c rounded once to FP32: the FP64 sum rounded to odd, then to FP32."""
    p = np.asarray(a, np.float64) * np.asarray(b, np.float64)          # exact
    p, c = np.broadcast_arrays(p, np.asarray(c, np.float64))
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)                                        # s + e = p + c exactly
    bits = s.view(np.int64)
    odd = np.where((e != 0) & (bits & 1 == 0), np.where((e > 0) == (s > 0), 1, -1), 0)
    return (bits + odd).view(np.float64).astype(F)


def collide(x, a, b):
    """Node update: x the four pulled populations [5][ny][nx], returns the four new ones."""
    rx, ry = x[1] + x[3], x[0] + x[2]
    U = rx + ry
    h = F(0.5)
    t0 = [fma(a, U[2], fma(b, U[3], -x[0][0])), fma(b, U[4], -x[0][1]), fma(a, U[0], -x[0][2]),
          fma(b, U[0], -x[0][3]), fma(b, U[1], -x[0][4])]
    t1 = [fma(b, U[4], -x[1][0]), fma(a, U[2], fma(-b, U[3], -x[1][1])), fma(a, U[1], -x[1][2]),
          fma(-b, U[1], -x[1][3]), fma(b, U[0], -x[1][4])]
    o0 = np.stack([fma(h, U[k], t0[k]) for k in range(5)])
    o1 = np.stack([fma(h, U[k], t1[k]) for k in range(5)])
    return [o0, o1, rx - o0, ry - o1]


def pull(f, dirichlet):
    """Populations that stream into each node; on a wall the opposite one, reflected."""
    x = [np.roll(f[0], 1, 2), np.roll(f[1], 1, 1), np.roll(f[2], -1, 2), np.roll(f[3], -1, 1)]
    if dirichlet:
        x[0][:, :, 0], x[2][:, :, -1] = SIGN[:, 0] * f[2][:, :, 0], SIGN[:, 0] * f[0][:, :, -1]
        x[1][:, 0], x[3][:, -1] = SIGN[:, 0] * f[3][:, 0], SIGN[:, 0] * f[1][:, -1]
    return x


def one_pass(m0, dx, dy, dd, a, b, steps, dirichlet, split):
    q, two = F(0.25), F(2)
    tx = [fma(a, m0[2], b * m0[3]) + dx[0], fma(b, m0[4], dx[1]), fma(a, m0[0], dx[2]), fma(b, m0[0], dx[3]),
          fma(b, m0[1], dx[4])]
    ty = [fma(b, m0[4], dy[0]), fma(a, m0[2], -(b * m0[3])) + dy[1], fma(a, m0[1], dy[2]), fma(-b, m0[1], dy[3]),
          fma(b, m0[0], dy[4])]
    seam = {0: q * (fma(two, tx[4], m0[4]) + dd[4]), 2: q * (fma(-two, tx[4], m0[4]) + dd[4])}
    if split:
        tx[4], ty[3] = b * m0[1] + dx[4], dy[3] - b * m0[1]
    tx, ty = np.stack(tx), np.stack(ty)
    f = [q * (fma(two, tx, m0) + dd), q * (fma(two, ty, m0) - dd), q * (fma(-two, tx, m0) + dd),
         q * (fma(-two, ty, m0) - dd)]
    # the seams: at columns c that are multiples of `period`, direction 0 into c and direction 2 into c - 1
    alt = {d: {4: seam[d]} for d in (0, 2)}
    period = {3: 28, 2: 30}[steps]
    nx = m0.shape[2]
    c = np.arange(0, nx + 1, period)
    into = {0: c[c < nx], 2: c[c > 0] - 1}
    if dirichlet:
        into = {0: into[0][into[0] > 0], 2: into[2][into[2] < nx - 1]}
    for level in range(steps):
        x = pull(f, dirichlet)
        nxt = {}
        for d, shift, wall in ((0, 1, 0), (2, -1, nx - 1)):
            y = [v.copy() for v in x]
            for k, v in alt[d].items():
                v = np.roll(v, shift, 1)
                if dirichlet:
                    v[:, wall] = x[d][k][:, wall]
                y[d][k] = v
            if level < steps - 1:
                o = collide(y, a, b)[d]
                nxt[d] = {1: o[1], 4: o[4]}
            elif split:
                x[d][:, :, into[d]] = y[d][:, :, into[d]]
        alt = nxt
        f = collide(x, a, b)
    sx, sy = f[0] + f[2], f[1] + f[3]
    m = sx + sy
    ex, ey = f[0] - f[2], f[1] - f[3]
    ex = np.stack([ex[0] - fma(a, m[2], b * m[3]), fma(-b, m[4], ex[1]), fma(-a, m[0], ex[2]), fma(-b, m[0], ex[3]),
                   fma(-b, m[1], ex[4])])
    ey = np.stack([fma(-b, m[4], ey[0]), ey[1] - fma(a, m[2], -(b * m[3])), fma(-a, m[1], ey[2]), fma(b, m[1], ey[3]),
                   fma(-b, m[0], ey[4])])
    return m, ex, ey, sx - sy


def decode(storage, w, inv):
    if storage == "ms_bfp":
        e = sum((w[i] & 1).astype(np.int32) << i for i in range(3))
        return [(w[i].astype(np.int16) >> 1).astype(F) * (np.ldexp(F(1), e - 7).astype(F) * inv) for i in range(3)]
    if storage == "ms_f16":
        return [v.view(np.float16).astype(F) * inv for v in w]
    return [(v.astype(np.uint32) << 16).view(F) * inv for v in w]


def encode(storage, v):
    if storage == "ms_f16":
        return [x.astype(np.float16).view(np.uint16) for x in v]
    if storage == "ms_bf16":
        u = [x.view(np.uint32) for x in v]
        return [((x + 0x7FFF + ((x >> 16) & 1)) >> 16).astype(np.uint16) for x in u]
    big = np.maximum(np.maximum(np.abs(v[0]), np.abs(v[1])), np.abs(v[2]))
    e = np.clip((big.view(np.uint32) >> 23).astype(np.int32) - 127 - 6, 0, 7)
    m = [np.clip(np.rint(x * np.ldexp(F(1), 7 - e).astype(F)), -16383, 16383).astype(np.int32) for x in v]
    return [((m[i] << 1) & 0xFFFE | (e >> i) & 1).astype(np.uint16) for i in range(3)]


def state(lat, lbm, nx, ny):
    lat.synchronize()
    pitch = (nx + 63) // 64 * 64
    plane = pitch * ny
    buf = np.zeros(50 * plane, np.uint8)
    lbm.lbm_save_state(lat.ctx, buf)
    m0 = buf[:20 * plane].view(F).reshape(5, ny, pitch)[:, :, :nx].copy()
    w = buf[20 * plane:].view(np.uint16).reshape(3, 5, ny, pitch)[..., :nx].copy()
    return m0, [w[0], w[1], w[2]]


@pytest.mark.parametrize("steps", [2, 3])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("storage", ["ms_bf16", "ms_f16", "ms_bfp"])
@pytest.mark.parametrize("nx,ny", [(3, 4), (28, 6), (30, 5), (57, 9), (169, 7), (361, 11)])
def test_words_of_one_pass(lbm, nx, ny, storage, dirichlet, steps):
    cK, cmu, dx, dt = 1.0, 0.6, 0.1, 0.1 / 3.2
    a, b = F(cK / (dx / dt)), F(cmu / (dx / dt))
    rng = np.random.default_rng(nx + 100 * ny)
    pop = rng.standard_normal((4, 5, ny, nx)) * 1e-3
    lat = lbm.Lattice(nx, ny, dx, dt, cK, cmu, dirichlet=dirichlet, storage=storage, track_displacement=False)
    lat.set_populations(pop, None)
    # the scale puts the largest deviation of the state set into [1024, 2048)
    o = pop.astype(F).astype(np.float64)
    m = o.sum(0)
    px = np.stack([a * m[2] + b * m[3], b * m[4], a * m[0], b * m[0], b * m[1]])
    py = np.stack([b * m[4], a * m[2] - b * m[3], a * m[1], -b * m[1], b * m[0]])
    big = max(np.abs(o[0] - o[2] - px).max(), np.abs(o[1] - o[3] - py).max(), np.abs(o[0] + o[2] - o[1] - o[3]).max())
    scale = F(2.0 ** math.floor(math.log2(2048.0 / big)))
    m0, w = state(lat, lbm, nx, ny)
    lat.step(steps)
    got_m, got_w = state(lat, lbm, nx, ny)
    lat.close()
    split = not (storage == "ms_bfp" and not dirichlet)
    want_m, *dev = one_pass(m0, *decode(storage, w, F(1) / scale), a, b, steps, dirichlet, split)
    want_w = encode(storage, [v * scale for v in dev])
    np.testing.assert_array_equal(got_m, want_m)
    for g, v in zip(got_w, want_w):
        if storage != "ms_bfp":
            g, v = (np.where(t == 0x8000, 0, t) for t in (g, v))
        np.testing.assert_array_equal(g, v)
