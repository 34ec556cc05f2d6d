"""Point -> index where the kernel can go wrong: block counts around its thread blocks, points at addresses that are not aligned, and bytes
that no point of a code holds."""
import numpy as np
import pytest
import torch

import llvq_inputs as gen
import paper_2603_11021_b200 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [(2, 13), (2, 20)])
@pytest.mark.parametrize("n,shift", [(1, 0), (255, 8), (256, 4), (257, 1), (1000, 0)])
def test_rank_inverts_the_oracle_at_any_address(oracle_mod, code, n, shift):
    ctx, o = P.Context(*code, device=0), oracle_mod.Code(*code)
    lo, hi = gen.random_indices(o.N, o.W, n, seed=n)
    pts = o.unrank_arrays(lo, hi)
    buf = torch.zeros(n * 24 + 16, dtype=torch.int8, device="cuda")
    buf[shift:shift + n * 24] = torch.from_numpy(pts).cuda().reshape(-1)
    idx = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert ctx._lib.llvq_rank_blocks(ctx._h, buf.data_ptr() + shift, n, idx.data_ptr(), stream) == 0
    assert np.array_equal(idx.cpu().numpy().view(np.uint64), lo)
    assert P.llvq_last_error(ctx) == (0, 0)


def test_rank_counts_every_point_outside_the_code(oracle_mod):
    ctx, o = P.Context(2, 13, device=0), oracle_mod.Code(2, 13)
    pts = o.unrank([o.N // 300 * j + j for j in range(300)])
    bad = pts.copy()
    for j in range(300):                                 # one coordinate each, from all values of a byte
        bad[j, j % 24] = np.int8((int(bad[j, j % 24]) + 1 + j % 255 + 128) % 256 - 128)
    got = P.llvq_rank_blocks(ctx, torch.from_numpy(bad).cuda()).cpu().numpy().view(np.uint64)
    inside = np.array([oracle_mod.is_member(r) >= 0 and (r.astype(int) ** 2).sum() % 16 == 0 and 2 <= (r.astype(int) ** 2).sum() // 16 <= 13 for r in bad])
    assert np.array_equal(got[~inside], np.zeros((~inside).sum(), dtype=np.uint64))
    assert P.llvq_last_error(ctx) == (int((~inside).sum()), 0)
    if inside.any():
        assert o.rank(bad[inside]) == [int(v) for v in got[inside]]
