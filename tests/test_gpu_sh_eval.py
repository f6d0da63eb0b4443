"""GPU parity of shm_sh_eval against the FP64 oracle's direct spherical-harmonic evaluation: degrees
from 0 to 20, segments that are empty, shorter and longer than a warp's slab of 128 queries, queries
outside every segment, per-query glyph ids and one glyph; bars of the query parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
import shm_inputs as I
from gpu_common import best_us, check_query, shm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return shm()


def _check(S, L, c, dirs, owner, **sel):
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    R, grad, normal = S.sh_eval(L, torch.from_numpy(c).cuda(), torch.from_numpy(dirs).cuda(), dev_status=st, **sel)
    inside = (owner >= 0) & (np.abs(dirs).sum(1) > 0)
    ref = O.sh_eval(L, c.astype(np.float64), dirs[inside], glyph=owner[inside].astype(np.int32))
    keep = torch.from_numpy(inside).cuda()
    check_query({"R": R[keep], "grad": grad[keep], "normal": normal[keep]}, dict(zip(("R", "grad", "normal"), ref)))
    for t in (R, grad, normal):
        assert torch.isnan(t[~keep]).all()
    bits = (S.SHM_DEV_BOUNDS if (owner < 0).any() else 0) | (S.SHM_DEV_NONFINITE if (np.abs(dirs).sum(1) == 0).any() else 0)
    assert st.item() == bits


@pytest.mark.parametrize("L", [0, 1, 2, 7, 16, 20])
def test_sh_eval_segments(S, L):
    lens = [0, 1, 31, 32, 33, 64, 65, 127, 128, 129, 0, 0, 700, 5000, 3]
    G, lead, tail = len(lens), 70, 133
    seg = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64) + lead
    Q = int(seg[-1]) + tail
    owner = np.full(Q, -1)
    for g in range(G):
        owner[seg[g]:seg[g + 1]] = g
    dirs = I.directions(Q, 70 + L)
    dirs *= np.linspace(0.5, 3.0, Q, dtype=np.float32)[:, None]
    dirs[[seg[12] + 5, seg[13] + 200]] = 0.0
    _check(S, L, I.sh_coeffs(G, L, 71 + L).astype(np.float32), dirs, owner, seg=torch.from_numpy(seg).cuda())


@pytest.mark.parametrize("Q", [1, 33, 4097, 300001])
def test_sh_eval_one_glyph_and_ids(S, Q):
    dirs = I.directions(Q, 90)
    c = I.sh_coeffs(7, 9, 91).astype(np.float32)
    _check(S, 9, c, dirs, np.zeros(Q, dtype=np.int64))
    ids = I.random_glyph_ids(Q, 7, 92)
    ids[Q // 2] = 7 if Q > 40 else ids[Q // 2]
    _check(S, 9, c, dirs, np.where(ids < 7, ids, -1), glyph=torch.from_numpy(ids).cuda())


@pytest.mark.parametrize("L", [0, 3, 8, 20])
def test_sh_eval_short_segments(S, L):
    """Segments of 0 to 40 queries, runs of empty ones longer than a warp, a long one among them, short ones at
    both ends: below 16 queries the lanes of a warp are on glyphs of their own."""
    lens = [(g * 7) % 41 for g in range(90)] + [0] * 70 + [1] * 100 + [0, 2] * 40 + [0] * 33 + [900, 15, 16, 0, 0, 1]
    G, lead, tail = len(lens), 5, 45
    seg = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64) + lead
    Q = int(seg[-1]) + tail
    owner = np.full(Q, -1)
    for g in range(G):
        owner[seg[g]:seg[g + 1]] = g
    dirs = I.directions(Q, 170 + L)
    dirs[[seg[95] + 1, seg[170]]] = 0.0
    _check(S, L, I.sh_coeffs(G, L, 171 + L).astype(np.float32), dirs, owner, seg=torch.from_numpy(seg).cuda())


@pytest.mark.parametrize("lens", [[1] * 60000, [0] * 30000 + [2000] + [0] * 170000 + [2000]], ids=["one_each", "empties"])
def test_sh_eval_sparse_segments_cost_like_ids(S, lens):
    """A glyph's share of the work is bounded by its queries: batches of one query a glyph, or with almost
    every glyph empty, stay within four times the same queries with glyph ids."""
    L, n = 8, np.asarray(lens)
    seg = torch.from_numpy(np.concatenate([[0], np.cumsum(n)]).astype(np.int64)).cuda()
    ids = torch.from_numpy(np.repeat(np.arange(len(n), dtype=np.int32), n)).cuda()
    c = torch.randn((len(n), (L + 1) ** 2), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    d = torch.from_numpy(I.directions(int(n.sum()), 180)).cuda()
    a, b = S.sh_eval(L, c, d, glyph=ids), S.sh_eval(L, c, d, seg=seg)
    for x, y in zip(a, b):
        assert float((x - y).abs().max()) <= 2e-6 * float(x.abs().max()) * (L + 1) ** 2
    assert best_us(lambda: S.sh_eval(L, c, d, seg=seg)) <= 4 * best_us(lambda: S.sh_eval(L, c, d, glyph=ids))
