"""The work that a user of the library has it do, as cases that can be timed and compared.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a user's program
holds before the call, run() is one pass through the public entry points, work() the bytes and
operations that the pass cannot do without, exact() the pass in 64-bit torch without the library.

Tables that a case only reads are made here in 64 bits and stored in the library's record layouts, so
that they do not depend on the library's own bakes; the cases that bake do so in run().
"""
from __future__ import annotations

import math

import torch

import paper_2602_20063_gb300 as S

DEV = "cuda"
F64 = torch.float64
DT = {"f32": S.SHM_F32, "f16": S.SHM_F16, "bf16": S.SHM_BF16}
LY = {"texel": S.SHM_LAYOUT_TEXEL, "cell": S.SHM_LAYOUT_CELL}
REC = {"f32": 16, "f16": 8, "bf16": 8}


# ------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one small glyph under the mouse: the smallest call, outputs allocated by the library (latency)
        dict(name="glyph_preview", kind="query", G=1, N=10, L=4, per=65536, select="one", dtype="f32", layout="texel"),
        # a close-up: a few dozen 16-bit glyphs, each covering much of the screen, queries grouped by glyph
        dict(name="dense_glyphs", kind="query", G=37, N=32, L=8, per=60000, select="seg", dtype="f16", layout="texel"),
        # a 4K orbit view of one large 16-bit terrain table in pixel order (screen-coherent queries)
        dict(name="planet_view", kind="view", N=2048, W=3840, H=2160, dtype="f16", layout="cell"),
        # random directions on the same planet (scatter, physics, sampling): the partitioned query
        dict(name="planet_random", kind="random", N=2048, Q=1 << 26, dtype="f32", layout="texel"),
        # a new procedural planet: fBm bake and its mip levels
        dict(name="planet_bake", kind="bake", N=2048, octaves=8, levels=6),
        # a field of SH glyphs, new coefficients each step: bake and query (the largest)
        dict(name="glyph_field", kind="field", G=16384, N=32, L=8, per=4096),
        # SH coefficients trained through bake and query under autograd, uneven query counts per glyph
        dict(name="sh_training", kind="train", G=4096, N=32, L=8, per=2048),
        # reproducible table gradients (deterministic reverse pass), uneven query counts per glyph
        dict(name="reproducible_grad", kind="repro", G=4096, N=32, L=6, per=1500),
        # one step of fitting tables to targets: fused loss and adjoint, then Adam
        dict(name="table_fit", kind="fit", G=1024, N=64, per=16384),
        # ground-truth targets by direct SH evaluation at high degree
        dict(name="sh_targets", kind="targets", G=1024, L=16, per=4096),
        # a frame of bump impostors of mixed resolution: bake, bounds, ray cast at 1080p
        dict(name="impostor_frame", kind="impostors", n=512, W=1920, H=1080),
        # the value-only bicubic baseline on the same glyphs (quality comparisons)
        dict(name="bicubic_baseline", kind="recon", G=2048, N=32, L=8, per=4096, method=S.SHM_RECON_BICUBIC,
             dtype="f32"),
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm; most are odd or not a multiple of a tile."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["query", "query", "view", "random", "bake", "field", "train", "repro", "fit", "targets",
                       "impostors", "recon"])
    if kind == "query":
        select = rng.choice(["one", "seg", "seg", "ids"])
        G = 1 if select == "one" else _log(rng, 2, 4000)
        per = _log(rng, 4000, 4000000) if select == "one" else _log(rng, 64, max(65, 16000000 // G))
        N = _log(rng, 8, 64)
        return dict(kind=kind, G=G, N=N, L=rng.randint(2, 8), per=per, select=select,
                    dtype=rng.choice(["f32", "f32", "f16", "bf16"]), layout=rng.choice(["texel", "texel", "cell"]))
    if kind == "view":
        H = _log(rng, 480, 2160)
        return dict(kind=kind, N=_log(rng, 256, 2048), W=H * 16 // 9, H=H, dtype=rng.choice(["f32", "f16"]),
                    layout=rng.choice(["texel", "cell"]))
    if kind == "random":
        return dict(kind=kind, N=_log(rng, 512, 2048), Q=_log(rng, 1 << 20, 1 << 26), dtype=rng.choice(["f32", "f16"]),
                    layout="texel")
    if kind == "bake":
        return dict(kind=kind, N=64 * _log(rng, 4, 32), octaves=rng.randint(4, 10), levels=rng.randint(1, 4))
    if kind == "field":
        N, G = _log(rng, 8, 64), _log(rng, 300, 16384)
        G = min(G, 1500000000 // (96 * (N + 2) ** 2))
        return dict(kind=kind, G=G, N=N, L=rng.randint(3, 10), per=_log(rng, 200, min(8192, 40000000 // G)))
    if kind == "train":
        N, G = _log(rng, 10, 40), _log(rng, 100, 4096)
        return dict(kind=kind, G=G, N=N, L=rng.randint(3, 10), per=_log(rng, 300, min(20000, 8000000 // G)))
    if kind == "repro":
        N, G = _log(rng, 10, 64), _log(rng, 100, 4096)
        return dict(kind=kind, G=G, N=N, L=rng.randint(2, 6), per=_log(rng, 300, min(20000, 8000000 // G)))
    if kind == "fit":
        N, G = _log(rng, 24, 96), _log(rng, 60, 1024)
        return dict(kind=kind, G=G, N=N, per=_log(rng, 2000, 16384))
    if kind == "targets":
        G = _log(rng, 1, 2000)
        return dict(kind=kind, G=G, L=rng.randint(4, 20), per=_log(rng, 100, max(101, 4000000 // G)))
    if kind == "impostors":
        H = _log(rng, 360, 1080)
        return dict(kind=kind, n=_log(rng, 20, 512), W=H * 16 // 9, H=H)
    N, G = _log(rng, 8, 48), _log(rng, 100, 2048)
    return dict(kind=kind, G=G, N=N, L=rng.randint(3, 8), per=_log(rng, 500, min(8192, 12000000 // G)),
                method=rng.randint(0, 3), dtype=rng.choice(["f32", "f16"]))


# ------------------------------------------------------------------------------------------ inputs
def _gen(seed, tag=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFFFFFF)
    return g


def _dirs(n, g):
    """[n][3] float32 directions uniform on the sphere."""
    d = torch.randn((n, 3), generator=g, device=DEV)
    return torch.nn.functional.normalize(d, dim=1)


def _coeffs(G, L, g):
    """c_lm ~ N(0, 1)/(l+1)^2, mean radius added to c_00."""
    l = torch.tensor([math.isqrt(k) for k in range((L + 1) ** 2)], device=DEV, dtype=torch.float32)
    c = torch.randn((G, (L + 1) ** 2), generator=g, device=DEV) / (l + 1.0) ** 2
    c[:, 0] += 2.5
    return c.contiguous()


def _even_seg(G, per):
    return torch.arange(0, G * per + 1, per, device=DEV, dtype=torch.int64)


def _ragged_seg(G, per, g):
    """Uneven segments of G * per queries in all (random cuts: some are empty, some several times the mean)."""
    Q = G * per
    cuts = torch.randint(0, Q + 1, (G - 1,), generator=g, device=DEV).sort().values
    ends = torch.tensor([0], device=DEV), cuts, torch.tensor([Q], device=DEV)
    return torch.cat(ends).to(torch.int64)


def _glyph_of(seg, lo, hi):
    q = torch.arange(lo, hi, device=DEV)
    return torch.searchsorted(seg, q, right=True) - 1


def _store(records, N, dtype, layout, r0=None):
    """Lut of [G][6][N+2][N+2][4] records (any float type) in the library's layout and storage type."""
    G = records.shape[0]
    lut = S.alloc_lut(G, N, DT[dtype], LY[layout], r0=r0)
    if layout == "cell":
        n = N + 1
        r = records.view(G, 6, N + 2, N + 2, 4)
        out = lut.data.view(G, 6, n, n, 4, 4)
        for c in range(4):
            out[..., c, :] = r[:, :, c >> 1:(c >> 1) + n, c & 1:(c & 1) + n, :]
    else:
        lut.data.copy_(records.reshape(-1))
    return lut


# ------------------------------------------------------------------------------------------ 64-bit mathematics
def _legendre(z, L):
    """Normalised associated Legendre functions without their (1 - z^2)^(m/2) factor, [l][m]."""
    one = torch.ones_like(z)
    P = [[None] * (L + 3) for _ in range(L + 1)]
    for m in range(L + 1):
        P[m][m] = one * math.sqrt(1 / (4 * math.pi)) if m == 0 else P[m - 1][m - 1] * math.sqrt((2 * m + 1) / (2 * m))
        for l in range(m + 1, L + 1):
            a = math.sqrt((4 * l * l - 1) / (l * l - m * m))
            v = z * P[l - 1][m]
            if l > m + 1:
                v = v - math.sqrt(((l - 1) ** 2 - m * m) / (4 * (l - 1) ** 2 - 1)) * P[l - 2][m]
            P[l][m] = a * v
    return P


def _sh_terms(w, L, second=False):
    """Yields (k, Y, dY, d2Y) of the real SH in polynomial form at unit vectors w [n][3] (64 bits)."""
    x, y, z = w.unbind(1)
    P = _legendre(z, L)
    zero = torch.zeros_like(z)
    c, s = [torch.ones_like(z)], [zero]
    for m in range(1, L + 1):
        c.append(x * c[-1] - y * s[-1])
        s.append(x * s[-1] + y * c[m - 1])
    for l in range(L + 1):
        for m in range(l + 1):
            q0 = P[l][m]
            f1 = math.sqrt((l - m) * (l + m + 1))
            q1 = f1 * P[l][m + 1] if m + 1 <= l else zero
            q2 = f1 * math.sqrt((l - m - 1) * (l + m + 2)) * P[l][m + 2] if m + 2 <= l else zero
            n = 1.0 if m == 0 else math.sqrt(2.0)
            for sine in ([False] if m == 0 else [False, True]):
                A = s[m] if sine else c[m]
                Ax = m * (s[m - 1] if sine else c[m - 1]) if m else zero
                Ay = m * (c[m - 1] if sine else -s[m - 1]) if m else zero
                H = None
                if second:
                    mm = m * (m - 1)
                    Axx = mm * (s[m - 2] if sine else c[m - 2]) if m > 1 else zero
                    Axy = mm * (c[m - 2] if sine else -s[m - 2]) if m > 1 else zero
                    H = [n * v for v in (q0 * Axx, q0 * Axy, -q0 * Axx, q1 * Ax, q1 * Ay, q2 * A)]
                yield l * l + l + (-m if sine else m), n * q0 * A, [n * q0 * Ax, n * q0 * Ay, n * q1 * A], H


def _grid(N, pad):
    """Chart coordinates 2u - 1 of texels 1 - pad .. N + pad, and per face the unit vectors of all of them."""
    i = torch.arange(1 - pad, N + pad + 1, device=DEV, dtype=F64)
    X = (2 * i - 1 - N) / N
    faces = []
    for f in range(6):
        k, sg = f >> 1, (-1.0 if f & 1 else 1.0)
        v = torch.empty((len(X), len(X), 3), device=DEV, dtype=F64)
        v[..., k] = sg
        v[..., (k + 1) % 3] = X[None, :]
        v[..., (k + 2) % 3] = X[:, None]
        faces.append(v)
    return X, torch.stack(faces)


def _sh_records(N, L):
    """[K][6 (N+2)^2 4]: the records (Y, Y_u h, Y_v h, Y_uv h^2) of every SH function at every texel."""
    X, wt = _grid(N, 1)
    P = N + 2
    wt = wt.reshape(-1, 3)
    f = torch.arange(6, device=DEV).repeat_interleave(P * P)
    xx = X[None, None, :].expand(6, P, P).reshape(-1)
    yy = X[None, :, None].expand(6, P, P).reshape(-1)
    rho = wt.norm(dim=1)
    eye = torch.eye(3, device=DEV, dtype=F64)
    b, c = eye[(f // 2 + 1) % 3], eye[(f // 2 + 2) % 3]
    w = wt / rho[:, None]
    r1 = rho[:, None]
    e1 = 2 / r1 * (b - w * (xx / rho)[:, None])
    e2 = 2 / r1 * (c - w * (yy / rho)[:, None])
    W = 4 / r1 ** 3 * (-yy[:, None] * b - xx[:, None] * c) + 12 * (xx * yy)[:, None] / r1 ** 5 * wt
    out = torch.empty(((L + 1) ** 2, 6 * P * P, 4), device=DEV, dtype=F64)
    for k, Y, g, H in _sh_terms(w, L, second=True):
        out[k, :, 0] = Y
        out[k, :, 1] = sum(g[a] * e1[:, a] for a in range(3)) / N
        out[k, :, 2] = sum(g[a] * e2[:, a] for a in range(3)) / N
        hxx, hxy, hyy, hxz, hyz, hzz = H
        q = (hxx * e1[:, 0] * e2[:, 0] + hyy * e1[:, 1] * e2[:, 1] + hzz * e1[:, 2] * e2[:, 2]
             + hxy * (e1[:, 0] * e2[:, 1] + e1[:, 1] * e2[:, 0]) + hxz * (e1[:, 0] * e2[:, 2] + e1[:, 2] * e2[:, 0])
             + hyz * (e1[:, 1] * e2[:, 2] + e1[:, 2] * e2[:, 1]))
        out[k, :, 3] = (q + sum(g[a] * W[:, a] for a in range(3))) / N ** 2
    return out.reshape((L + 1) ** 2, -1)


def _sh_tables(coeffs, N, L):
    """[G][6 (N+2)^2][4] records of SH glyphs in 64 bits."""
    return (coeffs.to(F64) @ _sh_records(N, L)).view(coeffs.shape[0], -1, 4)


def _sh_values(coeffs, N, L):
    """[G][6][N+4][N+4] values of SH glyphs in 64 bits (the value-only tables)."""
    _, w = _grid(N, 2)
    w = torch.nn.functional.normalize(w.reshape(-1, 3), dim=1)
    B = torch.empty(((L + 1) ** 2, w.shape[0]), device=DEV, dtype=F64)
    for k, Y, _, _ in _sh_terms(w, L):
        B[k] = Y
    return coeffs.to(F64) @ B


def _fd_records(samples, base=0.0):
    """[..][N+2][N+2][4] records by central differences of a margin grid [..][N+4][N+4]."""
    c = samples[..., 1:-1, 1:-1]
    du = 0.5 * (samples[..., 1:-1, 2:] - samples[..., 1:-1, :-2])
    dv = 0.5 * (samples[..., 2:, 1:-1] - samples[..., :-2, 1:-1])
    duv = 0.25 * ((samples[..., 2:, 2:] - samples[..., :-2, 2:]) - (samples[..., 2:, :-2] - samples[..., :-2, :-2]))
    return torch.stack((c + base, du, dv, duv), dim=-1)


class _Chart:
    """Face, cell and chart coordinates of 64-bit directions (the index choices carry no derivative)."""

    def __init__(self, d, N):
        a = d.abs()
        k = torch.where(a[:, 1] > a[:, 0], 1, 0)
        k = torch.where(a[:, 2] > a.gather(1, k[:, None])[:, 0], 2, k)
        self.k = k
        at = lambda off: d.gather(1, ((k + off) % 3)[:, None])[:, 0]
        dk = at(0)
        self.sg = torch.where(dk < 0, -1.0, 1.0).to(F64)
        self.f = 2 * k + (dk < 0)
        m = dk * self.sg
        self.x, self.y = at(1) / m, at(2) / m
        self.i, self.s = self._cell(self.x, N)
        self.j, self.t = self._cell(self.y, N)

    @staticmethod
    def _cell(x, N):
        X = 0.5 * N * x + 0.5 * (N + 1)
        i = X.detach().floor().clamp(0, N)
        return i.to(torch.int64), X - i

    def surface(self, d, R, Ru, Rv):
        """(R, S^2 gradient, normal) from the value and its chart derivatives."""
        rho = torch.sqrt(1 + self.x ** 2 + self.y ** 2)
        fr = 0.5 * rho[:, None] * torch.stack((-self.sg * (self.x * Ru + self.y * Rv), Ru, Rv), dim=1)
        comp = (torch.arange(3, device=d.device)[None, :] - self.k[:, None]) % 3
        g = fr.gather(1, comp)
        w = d / d.norm(dim=1, keepdim=True)
        n = R[:, None] * w - g
        return R, g, n / n.norm(dim=1, keepdim=True)


def _herm(s):
    return ((1 + 2 * s) * (1 - s) ** 2, s * s * (3 - 2 * s), s * (1 - s) ** 2, s * s * (s - 1),
            6 * s * (s - 1), 6 * s * (1 - s), (1 - s) * (1 - 3 * s), s * (3 * s - 2))


def _query64(table, base, N, dirs, r0=0.0, value_only=False):
    """Hermite query in 64 bits on records table [n][4]; base: first record of each query's glyph."""
    d = dirs.to(F64) if dirs.dtype != F64 else dirs
    c = _Chart(d, N)
    P = N + 2
    rec = base + (c.f * P + c.j) * P + c.i
    a, b = _herm(c.s), _herm(c.t)
    r = rs = rt = 0.0
    for bb in range(2):
        for aa in range(2):
            v, vu, vv, vuv = table[rec + bb * P + aa].to(F64).unbind(1)
            p, q = a[aa] * v + a[2 + aa] * vu, a[aa] * vv + a[2 + aa] * vuv
            r = r + b[bb] * p + b[2 + bb] * q
            if not value_only:
                ps, qs = a[4 + aa] * v + a[6 + aa] * vu, a[4 + aa] * vv + a[6 + aa] * vuv
                rs = rs + b[bb] * ps + b[2 + bb] * qs
                rt = rt + b[4 + bb] * p + b[6 + bb] * q
    if value_only:
        return r
    return c.surface(d, r0 + r, N * rs, N * rt)


def _all_queries(table, glyph_base, N, dirs, r0=0.0, chunk=1 << 21):
    """(R, grad, normal) of all queries; glyph_base(lo, hi) gives the first records of a range's glyphs."""
    Q = dirs.shape[0]
    out = {"R": torch.empty(Q, dtype=F64, device=DEV), "grad": torch.empty((Q, 3), dtype=F64, device=DEV),
           "normal": torch.empty((Q, 3), dtype=F64, device=DEV)}
    for lo in range(0, Q, chunk):
        hi = min(Q, lo + chunk)
        for k, v in zip(("R", "grad", "normal"), _query64(table, glyph_base(lo, hi), N, dirs[lo:hi], r0)):
            out[k][lo:hi] = v
    return out


def _pcg(x, y, z):
    M = 0xFFFFFFFF
    mul = lambda a, b: (a * b) & M
    x, y, z = ((mul(v, 1664525) + 1013904223) & M for v in (x, y, z))
    x = (x + mul(y, z)) & M
    y = (y + mul(z, x)) & M
    z = (z + mul(x, y)) & M
    x, y, z = x ^ (x >> 16), y ^ (y >> 16), z ^ (z >> 16)
    return (x + mul(y, z)) & M


def _fbm64(w, keys, amplitude):
    """fBm of value noise at unit vectors w [n][3] in 64 bits (base frequency 2, lacunarity 2, gain 1/2)."""
    total = torch.zeros(w.shape[0], device=w.device, dtype=F64)
    for o in range(keys.shape[0]):
        p = w * (2.0 * 2.0 ** o)
        fl = p.floor()
        t = p - fl
        q = (t * t * t * (t * (t * 6 - 15) + 10)).unbind(1)
        i = fl.to(torch.int64)
        corner = lambda a, b, c: (_pcg((i[:, 0] + a + keys[o, 0]) & 0xFFFFFFFF, (i[:, 1] + b + keys[o, 1]) & 0xFFFFFFFF,
                                       (i[:, 2] + c + keys[o, 2]) & 0xFFFFFFFF) >> 8).to(F64) * (2.0 / 16777216.0) - 1.0
        e = []
        for c in range(2):
            rows = [torch.lerp(corner(0, b, c), corner(1, b, c), q[0]) for b in range(2)]
            e.append(torch.lerp(rows[0], rows[1], q[1]))
        total += 0.5 ** o * torch.lerp(e[0], e[1], q[2])
    return amplitude * total


def _terrain(N, g, dtype):
    """[6][N+2][N+2][4] records of a relief of plane waves of falling amplitude, 2 % of the radius high."""
    n = 24
    freq = torch.exp(torch.linspace(math.log(2.0), math.log(150.0), n, device=DEV, dtype=torch.float32))
    k = torch.nn.functional.normalize(torch.randn((n, 3), generator=g, device=DEV), dim=1) * freq[:, None]
    ph = torch.rand(n, generator=g, device=DEV) * 6.2831853
    _, w = _grid(N, 2)
    w = torch.nn.functional.normalize(w, dim=-1)
    h = torch.zeros(w.shape[:-1], device=DEV, dtype=F64)
    for i in range(n):
        h += (0.02 / (1.0 + float(freq[i]))) * torch.sin((w @ k[i].to(F64)) + ph[i].to(F64))
    return _fd_records(h).to(torch.float32)[None]


def _rotation(g):
    q, _ = torch.linalg.qr(torch.randn((3, 3), generator=g, device=DEV))
    return q


def _view_dirs(W, H, g, tile=8):
    """Hit points on the unit sphere of a view from distance 3 (45 degrees), pixels in 8 x 8 tiles."""
    th = math.tan(math.radians(22.5))
    ty, tx, ly, lx = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (H // tile, W // tile, tile, tile)),
                                    indexing="ij")
    xn = (2 * (tx * tile + lx + 0.5) / W - 1) * th * W / H
    yn = (1 - 2 * (ty * tile + ly + 0.5) / H) * th
    d = torch.stack((xn.reshape(-1), yn.reshape(-1), -torch.ones(xn.numel(), device=DEV)), dim=1)
    d = torch.nn.functional.normalize(d, dim=1)
    b = d[:, 2] * 3.0
    disc = b * b - 8.0
    hit = disc >= 0
    t = -b[hit] - disc[hit].sqrt()
    p = d[hit] * t[:, None]
    p[:, 2] += 3.0
    return (p @ _rotation(g).T).contiguous()


def _view_count(W, H):
    return int(0.85 * math.pi * (H / 2) ** 2 * (math.tan(math.asin(1 / 3)) / math.tan(math.radians(22.5))) ** 2)


# ------------------------------------------------------------------------------------------ prepare
def _prep_query(c, seed):
    g = _gen(seed, 1)
    co = _coeffs(c["G"], c["L"], g)
    Q = c["G"] * c["per"]
    s = dict(lut=_store(_sh_tables(co, c["N"], c["L"]), c["N"], c["dtype"], c["layout"]), dirs=_dirs(Q, g), seg=None,
             glyph=None)
    if c["select"] == "seg":
        s["seg"] = _ragged_seg(c["G"], c["per"], g)
    elif c["select"] == "ids":
        s["glyph"] = torch.randint(0, c["G"], (Q,), generator=g, device=DEV, dtype=torch.int32)
    return s


def _prep_view(c, seed):
    g = _gen(seed, 2)
    return dict(lut=_store(_terrain(c["N"], g, c["dtype"]), c["N"], c["dtype"], c["layout"], r0=[1.0]),
                dirs=_view_dirs(c["W"], c["H"], g))


def _prep_random(c, seed):
    g = _gen(seed, 3)
    lut = _store(_terrain(c["N"], g, c["dtype"]), c["N"], c["dtype"], c["layout"], r0=[1.0])
    Q = c["Q"]
    out = {k: torch.empty((Q,) + s, device=DEV) for k, s in (("R", ()), ("grad", (3,)), ("normal", (3,)))}
    return dict(lut=lut, dirs=_dirs(Q, g), ws=S.query_binned_workspace(lut, Q), out=out)


def _prep_bake(c, seed):
    keys = torch.randint(0, 1 << 32, (c["octaves"], 3), generator=_gen(seed, 4), device=DEV)
    k32 = torch.where(keys >= 1 << 31, keys - (1 << 32), keys).to(torch.int32)
    chain = [S.alloc_lut(1, c["N"], r0=[1.0])]
    for _ in range(c["levels"]):
        chain.append(S.mip_like(chain[-1]))
    src = S.Source(kind=S.SHM_SRC_FBM, octaves=c["octaves"], keys=k32.contiguous(), amplitude=0.02)
    return dict(keys=keys, src=src, chain=chain)


def _prep_field(c, seed):
    g = _gen(seed, 5)
    lut = S.alloc_lut(c["G"], c["N"])
    src = S.Source(kind=S.SHM_SRC_SH, L=c["L"], coeffs=_coeffs(c["G"], c["L"], g), basis=S.sh_basis(c["N"], c["L"]))
    Q = c["G"] * c["per"]
    out = {k: torch.empty((Q,) + s, device=DEV) for k, s in (("R", ()), ("grad", (3,)), ("normal", (3,)))}
    return dict(lut=lut, src=src, ws=S.build_workspace(lut, src), dirs=_dirs(Q, g), seg=_even_seg(c["G"], c["per"]),
                out=out)


def _upstream(Q, g):
    return [torch.randn(s, generator=g, device=DEV) for s in ((Q,), (Q, 3), (Q, 3))]


def _prep_train(c, seed):
    g = _gen(seed, 6)
    lut = S.alloc_lut(c["G"], c["N"])
    co = _coeffs(c["G"], c["L"], g)
    src = S.Source(kind=S.SHM_SRC_SH, L=c["L"], coeffs=co, basis=S.sh_basis(c["N"], c["L"]))
    Q = c["G"] * c["per"]
    return dict(lut=lut, L=c["L"], basis=src.basis, ws=S.build_workspace(lut, src), coeffs=co.requires_grad_(True),
                dirs=_dirs(Q, g).requires_grad_(True), seg=_ragged_seg(c["G"], c["per"], g), up=_upstream(Q, g))


def _prep_repro(c, seed):
    g = _gen(seed, 7)
    lut = _store(_sh_tables(_coeffs(c["G"], c["L"], g), c["N"], c["L"]), c["N"], "f32", "texel")
    Q = c["G"] * c["per"]
    return dict(lut=lut, dlut=S.like_lut(lut, zero=True), dirs=_dirs(Q, g), seg=_ragged_seg(c["G"], c["per"], g),
                up=_upstream(Q, g))


def _prep_fit(c, seed):
    """Mid-training: smooth tables, Adam's moments of earlier steps, targets near the current shape."""
    g = _gen(seed, 8)
    G, Q = c["G"], c["G"] * c["per"]
    co = _coeffs(G, 3, g)
    lut = _store(_sh_tables(co, c["N"], 3), c["N"], "f32", "texel")
    d = _dirs(Q, g)
    ax = 0.3 * torch.randn((G, 3), generator=g, device=DEV)
    at = (d * ax.repeat_interleave(c["per"], dim=0)).sum(1)
    Rt = co[:, 0].repeat_interleave(c["per"]) * 0.28209479 + at
    nt = torch.nn.functional.normalize(d * (1 + at[:, None]) - 0.5 * ax.repeat_interleave(c["per"], dim=0), dim=1)
    m = 0.5 * torch.randn(lut.data.shape, generator=g, device=DEV)
    v = 0.25 * (0.5 + torch.rand(lut.data.shape, generator=g, device=DEV))
    return dict(lut=lut, dl=S.like_lut(lut, zero=True), m=m, v=v, dirs=d, Rt=Rt, nt=nt, seg=_even_seg(G, c["per"]),
                loss=torch.zeros(1, device=DEV), step=100)


def _prep_targets(c, seed):
    g = _gen(seed, 9)
    return dict(L=c["L"], coeffs=_coeffs(c["G"], c["L"], g), dirs=_dirs(c["G"] * c["per"], g),
                seg=_even_seg(c["G"], c["per"]))


def _scene(c, seed):
    """Bump objects of mixed resolution on a cubic grid: CSR offsets, centres, amplitudes, widths, N."""
    h = torch.Generator()
    h.manual_seed(int(seed) * 7919 + 10)
    n = c["n"]
    counts = torch.randint(8, 65, (n,), generator=h)
    off = torch.zeros(n + 1, dtype=torch.int64)
    off[1:] = counts.cumsum(0)
    B = int(off[-1])
    mu = torch.nn.functional.normalize(torch.randn((B, 3), generator=h, dtype=F64), dim=1).to(torch.float32)
    amp = torch.rand(B, generator=h) * 0.4 - 0.2
    width = torch.rand(B, generator=h) * 0.35 + 0.05
    Ns = [(16, 32, 64, 128)[int(i) % 4] for i in torch.randperm(n, generator=h)]  # a quarter of the objects each
    return off, mu, amp, width, Ns


def _prep_impostors(c, seed):
    off, mu, amp, width, Ns = _scene(c, seed)
    n = c["n"]
    lut = S.alloc_lut(n, Ns, r0=[1.0] * n)
    src = S.Source(kind=S.SHM_SRC_BUMPS, bump_offset=off.to(DEV), mu=mu.to(DEV), amp=amp.to(DEV), width=width.to(DEV))
    e = math.ceil(round(n ** (1 / 3), 6))
    at = [((i % e) - (e - 1) / 2, (i // e % e) - (e - 1) / 2, (i // (e * e)) - (e - 1) / 2) for i in range(n)]
    objs = S.objects_tensor([[3.0 * x for x in p] for p in at], [1.0] * n, [1.0] * n, list(range(n)))
    dist = (math.sqrt(3) * 1.5 * (e - 1) + 2.0) / math.sin(math.radians(22.5))
    cam = S.make_camera((0.0, 0.0, dist), (0.0, 0.0, -1.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), 45.0, c["W"], c["H"])
    ws = torch.empty(S.raycast_workspace_bytes(n, c["W"], c["H"]), dtype=torch.uint8, device=DEV)
    H, W = c["H"], c["W"]
    out = dict(rgba=torch.empty((H, W, 4), device=DEV), depth=torch.empty((H, W), device=DEV),
               normal=torch.empty((H, W, 3), device=DEV), obj_id=torch.empty((H, W), dtype=torch.int32, device=DEV))
    return dict(lut=lut, src=src, objs=objs, n=n, cam=cam, prm=S.make_raycast_params(), ws=ws, out=out)


def _prep_recon(c, seed):
    g = _gen(seed, 11)
    lut = S.alloc_lut(c["G"], c["N"], DT[c["dtype"]], S.SHM_LAYOUT_VALUE)
    lut.data.copy_(_sh_values(_coeffs(c["G"], c["L"], g), c["N"], c["L"]).reshape(-1))
    Q = c["G"] * c["per"]
    out = {k: torch.empty((Q,) + s, device=DEV) for k, s in (("R", ()), ("grad", (3,)), ("normal", (3,)))}
    return dict(lut=lut, method=c["method"], dirs=_dirs(Q, g), seg=_even_seg(c["G"], c["per"]), out=out)


def prepare(case, seed):
    s = globals()["_prep_" + case["kind"]](case, seed)
    s["kind"] = case["kind"]
    return s


# ------------------------------------------------------------------------------------------ run
def _three(out):
    return {k: out[k] for k in ("R", "grad", "normal")}


def run(s):
    kind = s["kind"]
    if kind == "query":
        return S.query(s["lut"], s["dirs"], glyph=s["glyph"], seg=s["seg"])
    if kind == "view":
        return S.query(s["lut"], s["dirs"])
    if kind == "random":
        return _three(S.query_binned(s["lut"], s["dirs"], s["ws"], out=s["out"]))
    if kind == "bake":
        S.build_lut(s["chain"][0], s["src"])
        for fine, coarse in zip(s["chain"], s["chain"][1:]):
            S.build_mip(fine, coarse)
        return [t.data for t in s["chain"]]
    if kind == "field":
        S.build_lut(s["lut"], s["src"], ws=s["ws"])
        out = S.query(s["lut"], s["dirs"], seg=s["seg"], out=s["out"])
        return dict(_three(out), table=s["lut"].data)
    if kind == "train":
        table = S.sh_bake_fn(s["coeffs"], s["basis"], s["lut"], s["L"], ws=s["ws"])
        out = S.query_fn(table, s["dirs"], s["lut"], seg=s["seg"])
        dc, dd = torch.autograd.grad(out, (s["coeffs"], s["dirs"]), grad_outputs=s["up"])
        return dict(R=out[0].detach(), grad=out[1].detach(), normal=out[2].detach(), dcoeffs=dc, ddirs=dd)
    if kind == "repro":
        s["dlut"].data.zero_()
        dd = S.query_backward(s["lut"], s["dirs"], s["dlut"], gR=s["up"][0], ggrad=s["up"][1], gnormal=s["up"][2],
                              seg=s["seg"], deterministic=True)
        return dict(dtable=s["dlut"].data, ddirs=dd)
    if kind == "fit":
        S.fit_backward(s["lut"], s["dirs"], s["Rt"], s["nt"], s["dl"], 1.0, 1.0, loss=s["loss"], seg=s["seg"])
        S.adam_step(s["lut"].data, s["dl"].data, s["m"], s["v"], lr=1e-2, step=s["step"])
        s["step"] += 1
        return dict(table=s["lut"].data, m=s["m"], v=s["v"], loss=s["loss"])
    if kind == "targets":
        R, grad, normal = S.sh_eval(s["L"], s["coeffs"], s["dirs"], seg=s["seg"])
        return dict(R=R, grad=grad, normal=normal)
    if kind == "impostors":
        S.build_lut(s["lut"], s["src"])
        rmax = S.lut_bounds(s["lut"])
        s["objs"].view(torch.float32).view(-1, 6)[:, 4].copy_(rmax)
        o = S.raycast(s["lut"], s["objs"], s["n"], s["cam"], s["prm"], ws=s["ws"], out=s["out"])
        return dict(table=s["lut"].data, rmax=rmax, rgba=o["rgba"], depth=o["depth"], normal=o["normal"],
                    obj_id=o["obj_id"])
    out = S.query_recon(s["lut"], s["method"], s["dirs"], seg=s["seg"], out=s["out"])
    return _three(out)


# ------------------------------------------------------------------------------------------ work
def work(c):
    kind = c["kind"]
    if kind in ("query", "field", "train", "repro", "fit", "recon"):
        G, N, Q = c["G"], c["N"], c["G"] * c["per"]
        T = 6 * (N + 2) ** 2
    if kind == "query":
        rec = REC[c["dtype"]]
        table = min(G * (T if c["layout"] == "texel" else 24 * (N + 1) ** 2) * rec, 4 * rec * Q)
        sel = {"one": 0, "seg": 8 * (G + 1), "ids": 4 * Q}[c["select"]]
        return dict(bytes=table + sel + 40 * Q, flops=250 * Q)
    if kind == "view":
        Q, n = _view_count(c["W"], c["H"]), 6 * (c["N"] + 2) ** 2
        return dict(bytes=min(n * REC[c["dtype"]] // 4, 4 * REC[c["dtype"]] * Q) + 40 * Q, flops=250 * Q)
    if kind == "random":
        table = 6 * (c["N"] + 2) ** 2 * REC[c["dtype"]]
        return dict(bytes=min(table, 4 * REC[c["dtype"]] * c["Q"]) + 40 * c["Q"], flops=250 * c["Q"])
    if kind == "bake":
        n = [6 * ((c["N"] >> i) + 2) ** 2 for i in range(c["levels"] + 1)]
        return dict(bytes=16 * sum(n), flops=n[0] * c["octaves"] * 60 + 12 * sum(n[1:]))
    if kind == "field":
        K = (c["L"] + 1) ** 2
        return dict(bytes=4 * G * K + 16 * K * T + 16 * G * T + 40 * Q, flops=8 * G * K * T + 250 * Q)
    if kind == "train":
        K = (c["L"] + 1) ** 2
        return dict(bytes=8 * G * K + 16 * K * T + 16 * G * T + 80 * Q, flops=16 * G * K * T + 900 * Q)
    if kind == "repro":
        return dict(bytes=32 * G * T + 52 * Q, flops=650 * Q)
    if kind == "fit":
        return dict(bytes=96 * G * T + 28 * Q, flops=650 * Q + 60 * G * T)
    if kind == "targets":
        Q, K = c["G"] * c["per"], (c["L"] + 1) ** 2
        return dict(bytes=4 * c["G"] * K + 40 * Q, flops=12 * K * Q)
    if kind == "impostors":
        n = c["n"] * sum(6 * (N + 2) ** 2 for N in (16, 32, 64, 128)) // 4
        return dict(bytes=16 * n + 36 * c["W"] * c["H"], flops=n * 36 * 12 + 5 * 250 * c["W"] * c["H"])
    val = 4 if c["dtype"] == "f32" else 2
    return dict(bytes=G * 6 * (N + 4) ** 2 * val + 40 * Q, flops=300 * Q)


# ------------------------------------------------------------------------------------------ exact
def _texel_records(lut, N):
    """The stored records of a uniform table as [n][4] in texel order (cells hold copies of their corners)."""
    if lut.layout == S.SHM_LAYOUT_TEXEL:
        return lut.data.view(-1, 4)
    G, n = lut.n_glyphs, N + 1
    c = lut.data.view(G, 6, n, n, 4, 4)
    r = torch.empty((G, 6, N + 2, N + 2, 4), dtype=lut.data.dtype, device=DEV)
    for k in range(4):
        r[:, :, (k >> 1):(k >> 1) + n, (k & 1):(k & 1) + n] = c[..., k, :]
    return r.view(-1, 4)


def _grad_tables(table, G, N, dirs, seg, up_of, want_dirs):
    """64-bit reverse pass by autograd, a group of glyphs at a time: (dL/dtable, dL/ddirs, losses)."""
    T = 6 * (N + 2) ** 2
    dt = torch.zeros((G * T, 4), dtype=F64, device=DEV)
    dd = torch.zeros(dirs.shape, dtype=F64, device=DEV) if want_dirs else None
    cuts = seg.tolist()
    loss, g0 = 0.0, 0
    while g0 < G:
        g1 = g0 + 1
        while g1 < G and cuts[g1 + 1] - cuts[g0] <= 1 << 20 and (g1 + 1 - g0) * T <= 1 << 24:
            g1 += 1
        lo, hi = cuts[g0], cuts[g1]
        for a in range(lo, hi, 1 << 20):
            b = min(hi, a + (1 << 20))
            tab = table[g0 * T:g1 * T].to(F64).detach().requires_grad_(True)
            d = dirs[a:b].detach().to(F64).requires_grad_(True)
            out = _query64(tab, (_glyph_of(seg, a, b) - g0) * T, N, d)
            L = up_of(out, a, b)
            gt, gd = torch.autograd.grad(L, (tab, d))
            dt[g0 * T:g1 * T] += gt
            if want_dirs:
                dd[a:b] = gd
            loss += L.detach()
        g0 = g1
    return dt, dd, loss


def _dot_up(up):
    return lambda out, a, b: sum((o * u[a:b].to(F64)).sum() for o, u in zip(out, up))


def _ex_query(c, s):
    T = 6 * (c["N"] + 2) ** 2
    if c["select"] == "one":
        base = lambda lo, hi: 0
    elif c["select"] == "seg":
        base = lambda lo, hi: _glyph_of(s["seg"], lo, hi) * T
    else:
        base = lambda lo, hi: s["glyph"][lo:hi].to(torch.int64) * T
    return _all_queries(_texel_records(s["lut"], c["N"]), base, c["N"], s["dirs"])


def _ex_view(c, s):
    return _all_queries(_texel_records(s["lut"], c["N"]), lambda lo, hi: 0, c["N"], s["dirs"], r0=1.0)


_ex_random = _ex_view


def _ex_bake(c, s):
    N = c["N"]
    _, w = _grid(N, 2)
    w = w.view(6, -1, 3)
    h = torch.empty(w.shape[:2], dtype=F64, device=DEV)
    for f in range(6):
        for lo in range(0, h.shape[1], 1 << 21):
            v = w[f, lo:lo + (1 << 21)]
            h[f, lo:lo + (1 << 21)] = _fbm64(v / v.norm(dim=1, keepdim=True), s["keys"], 0.02)
    out = [_fd_records(h.view(6, N + 4, N + 4))]
    for _ in range(c["levels"]):
        fine, N = out[-1].reshape(-1, 4), N // 2
        ic = torch.arange(-1, N + 3, device=DEV)
        kids = torch.stack((2 * ic - 1, 2 * ic), dim=1).reshape(-1).to(F64)  # fine texels under each sample
        X = (2 * kids - 1 - 2 * N) / (2 * N)
        acc = torch.empty((6, len(X), len(X)), dtype=F64, device=DEV)
        for f in range(6):
            k, sg = f >> 1, (-1.0 if f & 1 else 1.0)
            for lo in range(0, len(X), 512):
                Y = X[lo:lo + 512]
                d = torch.empty((len(Y), len(X), 3), dtype=F64, device=DEV)
                d[..., k], d[..., (k + 1) % 3], d[..., (k + 2) % 3] = sg, X[None, :], Y[:, None]
                acc[f, lo:lo + 512] = _query64(fine, 0, 2 * N, d.view(-1, 3), value_only=True).view(len(Y), -1)
        acc = acc.view(6, N + 4, 2, N + 4, 2).mean(dim=(2, 4))
        out.append(_fd_records(acc))
    return [t.reshape(-1) for t in out]


def _ex_field(c, s):
    T = 6 * (c["N"] + 2) ** 2
    t = _sh_tables(s["src"].coeffs, c["N"], c["L"]).reshape(-1, 4)
    out = _all_queries(t, lambda lo, hi: _glyph_of(s["seg"], lo, hi) * T, c["N"], s["dirs"])
    return dict(out, table=t.reshape(-1))


def _ex_train(c, s):
    G, N, T = c["G"], c["N"], 6 * (c["N"] + 2) ** 2
    co, dirs = s["coeffs"].detach(), s["dirs"].detach()
    B = _sh_records(N, c["L"])
    t = (co.to(F64) @ B).view(-1, 4)
    out = _all_queries(t, lambda lo, hi: _glyph_of(s["seg"], lo, hi) * T, N, dirs)
    dt, dd, _ = _grad_tables(t, G, N, dirs, s["seg"], _dot_up(s["up"]), True)
    return dict(out, dcoeffs=dt.view(G, -1) @ B.T, ddirs=dd)


def _ex_repro(c, s):
    dt, dd, _ = _grad_tables(s["lut"].data.view(-1, 4), c["G"], c["N"], s["dirs"], s["seg"], _dot_up(s["up"]), True)
    return dict(dtable=dt.reshape(-1), ddirs=dd)


def _ex_fit(c, s):
    def loss_of(out, a, b):
        return ((out[0] - s["Rt"][a:b]) ** 2).sum() + ((out[2] - s["nt"][a:b]) ** 2).sum()

    dt, _, loss = _grad_tables(s["lut"].data.view(-1, 4), c["G"], c["N"], s["dirs"], s["seg"], loss_of, False)
    gr = dt.reshape(-1)
    m = 0.9 * s["m"].to(F64) + 0.1 * gr
    v = 0.999 * s["v"].to(F64) + 0.001 * gr * gr
    k = s["step"]
    p = s["lut"].data.to(F64) - 1e-2 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return dict(table=p, m=m, v=v, loss=loss.reshape(1))


def _ex_targets(c, s):
    Q = s["dirs"].shape[0]
    out = dict(R=torch.empty(Q, dtype=F64, device=DEV), grad=torch.empty((Q, 3), dtype=F64, device=DEV),
               normal=torch.empty((Q, 3), dtype=F64, device=DEV))
    for lo in range(0, Q, 1 << 19):
        hi = min(Q, lo + (1 << 19))
        d = s["dirs"][lo:hi].to(F64)
        w = d / d.norm(dim=1, keepdim=True)
        ck = s["coeffs"].to(F64).T.contiguous()
        gl = _glyph_of(s["seg"], lo, hi)
        R, g = 0.0, [0.0, 0.0, 0.0]
        for k, Y, dY, _ in _sh_terms(w, c["L"]):
            a = ck[k][gl]
            R = R + a * Y
            g = [u + a * v for u, v in zip(g, dY)]
        g = torch.stack(g, dim=1)
        g = g - w * (w * g).sum(1, keepdim=True)
        n = R[:, None] * w - g
        out["R"][lo:hi], out["grad"][lo:hi], out["normal"][lo:hi] = R, g, n / n.norm(dim=1, keepdim=True)
    return out


def _ex_impostors(c, s):
    """The tables and their bounds; the image follows from hit decisions and has no 64-bit counterpart."""
    src, parts, rmax = s["src"], [], []
    off = src.bump_offset.tolist()
    grids = {}
    for g, N in enumerate(s["lut"].N.tolist()):
        if N not in grids:
            grids[N] = torch.nn.functional.normalize(_grid(N, 2)[1].reshape(-1, 3), dim=1)
        h = torch.zeros(grids[N].shape[0], dtype=F64, device=DEV)
        b = slice(off[g], off[g + 1])
        mu, amp, wd = src.mu[b].to(F64), src.amp[b].to(F64), src.width[b].to(F64)
        d2 = (grids[N][:, None, :] - mu[None]).square().sum(-1)
        h = (amp * torch.exp(-d2 / (2 * wd * wd))).sum(1)
        t = _fd_records(h.view(6, N + 4, N + 4))
        a = t.abs()
        a[..., 0] = (1.0 + t[..., 0]).abs()
        cell = torch.stack([a[:, j:j + N + 1, i:i + N + 1] for j in range(2) for i in range(2)]).amax(0)
        rmax.append((cell[..., 0] + (cell[..., 1] + cell[..., 2]) / 4 + cell[..., 3] / 16).amax())
        parts.append(t.reshape(-1))
    return dict(table=torch.cat(parts), rmax=torch.stack(rmax), rgba=None, depth=None, normal=None, obj_id=None)


def _taps(method, s):
    """Weights of taps -1 .. 2 and their derivatives (Catmull-Rom), or the B-spline's weights."""
    if method == S.SHM_RECON_BICUBIC:
        w = [0.5 * (-s ** 3 + 2 * s ** 2 - s), 0.5 * (3 * s ** 3 - 5 * s ** 2 + 2), 0.5 * (-3 * s ** 3 + 4 * s ** 2 + s),
             0.5 * (s ** 3 - s ** 2)]
        dw = [0.5 * (-3 * s ** 2 + 4 * s - 1), 0.5 * (9 * s ** 2 - 10 * s), 0.5 * (-9 * s ** 2 + 8 * s + 1),
              0.5 * (3 * s ** 2 - 2 * s)]
        return w, dw
    r = 1 - s
    return [r ** 3 / 6, (3 * s ** 3 - 6 * s ** 2 + 4) / 6, (-3 * s ** 3 + 3 * s ** 2 + 3 * s + 1) / 6, s ** 3 / 6], None


def _ex_recon(c, s):
    N, n = c["N"], c["N"] + 4
    tab, method = s["lut"].data, c["method"]
    Q = s["dirs"].shape[0]
    out = dict(R=torch.empty(Q, dtype=F64, device=DEV), grad=torch.empty((Q, 3), dtype=F64, device=DEV),
               normal=torch.empty((Q, 3), dtype=F64, device=DEV))
    for lo in range(0, Q, 1 << 20):
        hi = min(Q, lo + (1 << 20))
        d = s["dirs"][lo:hi].to(F64)
        ch = _Chart(d, N)
        base = _glyph_of(s["seg"], lo, hi) * (6 * n * n) + ch.f * (n * n)
        V = lambda i, j: tab[base + (j + 1) * n + (i + 1)].to(F64)

        def bilinear(i, j):
            a = V(i, j) + ch.s * (V(i + 1, j) - V(i, j))
            b = V(i, j + 1) + ch.s * (V(i + 1, j + 1) - V(i, j + 1))
            return a + ch.t * (b - a)

        def sixteen(i, j, wu, wv):
            return sum(wv[b] * sum(wu[a] * V(i - 1 + a, j - 1 + b) for a in range(4)) for b in range(4))

        def spline(i, j):
            ic, jc = i.clamp(0, N), j.clamp(0, N)
            return sixteen(ic, jc, _taps(method, ch.s + (i - ic))[0], _taps(method, ch.t + (j - jc))[0])

        zero = torch.zeros_like(ch.s)
        if method == S.SHM_RECON_NEAREST:
            R, Ru, Rv = V((ch.i + (ch.s >= 0.5)).clamp(1, N), (ch.j + (ch.t >= 0.5)).clamp(1, N)), zero, zero
        elif method == S.SHM_RECON_BICUBIC:
            (wu, du), (wv, dv) = _taps(method, ch.s), _taps(method, ch.t)
            R, Ru, Rv = sixteen(ch.i, ch.j, wu, wv), N * sixteen(ch.i, ch.j, du, wv), N * sixteen(ch.i, ch.j, wu, dv)
        else:
            at = bilinear if method == S.SHM_RECON_BILINEAR else spline
            R = at(ch.i, ch.j)
            Ru = (at(ch.i + 1, ch.j) - at(ch.i - 1, ch.j)) * (0.5 * N)
            Rv = (at(ch.i, ch.j + 1) - at(ch.i, ch.j - 1)) * (0.5 * N)
        for k, v in zip(("R", "grad", "normal"), ch.surface(d, R, Ru, Rv)):
            out[k][lo:hi] = v
    return out


def exact(case, seed):
    return globals()["_ex_" + case["kind"]](case, prepare(case, seed))
