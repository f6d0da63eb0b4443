"""The staged segment query with its work cut inside glyphs: bit-identical to the per-query path (the
same queries with glyph ids) for empty, short and very long segments, queries outside every segment,
one and two tables per CTA, every dtype, all outputs and the usual three."""
import numpy as np
import pytest
import torch

import shm_inputs as I
from gpu_common import shm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return shm()


def _table(S, G, N, dtype, seed):
    L = 4
    c = torch.from_numpy(I.sh_coeffs(G, L, seed).astype(np.float32)).cuda()
    lut = S.alloc_lut(G, N, dtype, r0=np.linspace(-0.2, 0.3, G).astype(np.float32))
    S.build_lut(lut, S.Source(kind=S.SHM_SRC_SH, L=L, coeffs=c, basis=S.sh_basis(N, L)))
    return lut


LENS = {"one": [70001], "long": [0, 3, 250000, 0, 1, 40000, 511, 0], "many": [900 + 37 * (g % 50) for g in range(700)],
        "ends_empty": [0] * 40 + [90000] + [0] * 20}


@pytest.mark.parametrize("lens", sorted(LENS))
@pytest.mark.parametrize("N,dtype", [(1, 0), (9, 0), (22, 0), (23, 0), (32, 0), (32, 1), (20, 2)])
def test_split_equals_per_query(S, N, dtype, lens):
    n = np.asarray(LENS[lens])
    G, lead, tail = len(n), 130, 75
    seg = np.concatenate([[0], np.cumsum(n)]).astype(np.int64) + lead
    Q = int(seg[-1]) + tail
    ids = np.full(Q, -1, dtype=np.int32)
    ids[lead:Q - tail] = np.repeat(np.arange(G), n)
    lut = _table(S, G, N, dtype, 5 + N)
    d = torch.from_numpy(I.directions(Q, 6 + N)).cuda()
    d[lead + 1] = 0.0
    every = ("R", "grad", "normal", "chart", "fij")
    st = torch.zeros(2, dtype=torch.int32, device="cuda")
    ref = S.query(lut, d, glyph=torch.from_numpy(ids).cuda(), want=every, dev_status=st[:1])
    sg = torch.from_numpy(seg).cuda()
    for want in (every, ("R", "grad", "normal")):
        st[1] = 0
        got = S.query(lut, d, seg=sg, want=want, dev_status=st[1:])
        for k in want:
            assert torch.equal(got[k].view(torch.int32), ref[k].view(torch.int32)), (k, want)
        assert st[0].item() == st[1].item() != 0


@pytest.mark.parametrize("method", [0, 1, 2, 3])
@pytest.mark.parametrize("N,dtype", [(1, 0), (2, 1), (9, 0), (9, 1), (32, 0), (33, 2), (44, 0), (45, 1), (64, 0)])
def test_split_value_tables_equal_per_query(S, method, N, dtype):
    """Value-only baselines: tables that are no multiple of 16 bytes (odd N), one and two per CTA, and
    (N = 64 f32, 111 KB) near the largest that is staged; the last glyph ends at the pool's end."""
    n = np.asarray([1300 + 211 * (g % 9) for g in range(23)] + [0, 120000])
    G, lead, tail = len(n), 33, 40
    seg = np.concatenate([[0], np.cumsum(n)]).astype(np.int64) + lead
    Q = int(seg[-1]) + tail
    ids = np.full(Q, -1, dtype=np.int32)
    ids[lead:Q - tail] = np.repeat(np.arange(G), n)
    lut = S.alloc_lut(G, N, dtype, S.SHM_LAYOUT_VALUE, r0=np.linspace(-0.2, 0.3, G).astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(N)
    lut.data.copy_(1.0 + 0.1 * torch.randn(lut.data.shape, generator=g, device="cuda"))
    d = torch.from_numpy(I.directions(Q, 60 + N)).cuda()
    d[lead + 1] = 0.0
    want = ("R", "grad", "normal", "chart", "fij")
    st = torch.zeros(2, dtype=torch.int32, device="cuda")
    ref = S.query_recon(lut, method, d, glyph=torch.from_numpy(ids).cuda(), want=want, dev_status=st[:1])
    got = S.query_recon(lut, method, d, seg=torch.from_numpy(seg).cuda(), want=want, dev_status=st[1:])
    for k in want:
        assert torch.equal(got[k].view(torch.int32), ref[k].view(torch.int32)), k
    assert st[0].item() == st[1].item() != 0


@pytest.mark.parametrize("lens", [[3000000, 0, 7, 1700000, 0, 511], [40000] * 9 + [1, 0, 0, 90001], [5000000] * 2])
@pytest.mark.parametrize("N,layout", [(47, 0), (9, 1)])
def test_long_unstaged_segments_equal_per_query(S, N, layout, lens):
    """Segments of many chunks on tables that are not staged (one to eight rounds a chunk, no search where a
    segment goes on): bit-identical to the same queries with glyph ids."""
    n = np.asarray(lens)
    G, lead, tail = len(n), 600, 75
    seg = np.concatenate([[0], np.cumsum(n)]).astype(np.int64) + lead
    Q = int(seg[-1]) + tail
    ids = np.full(Q, -1, dtype=np.int32)
    ids[lead:Q - tail] = np.repeat(np.arange(G), n)
    g = torch.Generator(device="cuda").manual_seed(N)
    lut = S.alloc_lut(G, N, 0, layout)
    lut.data.copy_(1.0 + 0.1 * torch.randn(lut.data.shape, generator=g, device="cuda"))
    d = torch.nn.functional.normalize(torch.randn(Q, 3, generator=g, device="cuda"), dim=1)
    want = ("R", "grad", "normal", "chart", "fij")
    st = torch.zeros(2, dtype=torch.int32, device="cuda")
    ref = S.query(lut, d, glyph=torch.from_numpy(ids).cuda(), want=want, dev_status=st[:1])
    got = S.query(lut, d, seg=torch.from_numpy(seg).cuda(), want=want, dev_status=st[1:])
    for k in want:
        assert torch.equal(got[k].view(torch.int32), ref[k].view(torch.int32)), k
    assert st[0].item() == st[1].item() == S.SHM_DEV_BOUNDS
