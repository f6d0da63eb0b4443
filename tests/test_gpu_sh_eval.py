"""GPU parity of shm_sh_eval against the FP64 oracle's direct spherical-harmonic evaluation: degrees
from 0 to 20, segments that are empty, shorter and longer than a warp's slab of 128 queries, queries
outside every segment, per-query glyph ids and one glyph; bars of the query parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
import shm_inputs as I
from gpu_common import check_query, shm

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
