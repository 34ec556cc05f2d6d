"""The encoder's search against the CPU oracle where it can go wrong: the change from a warp per vector to two lanes per vector, shares of a
thread block around a warp's and a block's vectors, more near-ties at a time than a block's list holds, the number of shells around which
radii are left out, outputs at odd addresses."""
import numpy as np
import pytest
import torch

import paper_2603_11021_b200 as P

pytestmark = pytest.mark.gpu

PAIRS_FROM = {"EUCLIDEAN": 384, "ANGULAR": 136}           # vectors per SM beyond which two lanes take a vector


def _inputs(n, seed, grid=7):
    """Gaussian vectors of many lengths; every `grid`-th on a half-integer grid (near-ties between cosets), every eleventh zero."""
    rng = np.random.default_rng(seed)
    v = rng.standard_normal((n, 24)) * np.exp(rng.uniform(-1, 2.2, (n, 1)))
    v[::grid] = np.round(v[::grid] * 2) / 2
    v[5::11] = 0
    return v.astype(np.float32)


def _check(oracle_mod, code, v, metric, shift=0):
    o, ctx = oracle_mod.Code(*code), P.Context(*code, device=0)
    want, index = o.encode(v.astype(np.float64), getattr(oracle_mod, metric), threads=16)
    n = len(v)
    d_v = torch.zeros(n * 24 + 4, dtype=torch.float32, device="cuda")
    d_v[shift:shift + n * 24] = torch.from_numpy(v).cuda().reshape(-1)
    out = torch.zeros(n * 24 + 4, dtype=torch.int8, device="cuda")
    idx = torch.zeros(n, dtype=torch.int64, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert ctx._lib.llvq_encode_blocks(ctx._h, d_v.data_ptr() + 4 * shift, n, getattr(P, "LLVQ_" + metric), out.data_ptr() + shift, idx.data_ptr(), stream) == 0
    assert np.array_equal(out[shift:shift + n * 24].cpu().numpy().reshape(n, 24), want)
    assert int(out[:shift].abs().sum()) == 0 and int(out[shift + n * 24:].abs().sum()) == 0
    assert np.array_equal(idx.cpu().numpy().view(np.uint64), np.array(index, dtype=np.uint64))


@pytest.mark.parametrize("metric", ["EUCLIDEAN", "ANGULAR"])
@pytest.mark.parametrize("vectors", ["one", "sms-1", "sms+1", "16sms+1", "last_warp_form", "first_pair_form", "pair_form_ragged"])
def test_shares_of_a_thread_block(oracle_mod, metric, vectors):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = PAIRS_FROM[metric] * sms
    n = {"one": 1, "sms-1": sms - 1, "sms+1": sms + 1, "16sms+1": 16 * sms + 1, "last_warp_form": edge, "first_pair_form": edge + 1,
         "pair_form_ragged": edge + 50 * sms + 77}[vectors]
    _check(oracle_mod, (2, 13) if metric == "EUCLIDEAN" else (2, 5), _inputs(n, 3, grid=2 if vectors == "pair_form_ragged" else 7), metric, shift=1 if n % 2 else 0)


@pytest.mark.parametrize("m_hi", [4, 5, 12, 24])
def test_angular_search_leaves_out_only_radii_that_cannot_win(oracle_mod, m_hi):
    _check(oracle_mod, (2, m_hi), _inputs(500, m_hi), "ANGULAR")
