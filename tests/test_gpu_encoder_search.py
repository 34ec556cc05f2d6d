"""The encoder's search against the CPU oracle where it can go wrong: the change from a warp per vector to two lanes per vector, shares of a
thread block around a warp's and a block's vectors, more near-ties at a time than a block's list holds, the number of shells around which
radii are left out, outputs at odd addresses; and with two lanes per vector what tests/test_gpu_encoder.py gives the other form: ties between
cosets, edges of the ball, extreme lengths, inputs that are not finite."""
import os
import re

import numpy as np
import pytest
import torch

import paper_2603_11021_b200 as P
from test_gpu_encoder import _edge_inputs

pytestmark = pytest.mark.gpu

# vectors per SM beyond which two lanes take a vector
_SOURCE = open(os.path.join(os.path.dirname(P.__file__), "csrc", "encode.cu")).read()
PAIRS_FROM = {m.upper(): int(re.search(r"kPairsFrom%s = (\d+)" % m.capitalize(), _SOURCE)[1]) for m in ("euclidean", "angular")}


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


def _pair_form(code, distinct, metric, seed=1):
    """Enough draws from the distinct vectors that two lanes take each: (points, indices, which one was drawn)."""
    ctx = P.Context(*code, device=0)
    n = PAIRS_FROM[metric] * torch.cuda.get_device_properties(0).multi_processor_count + 1001
    which = np.random.default_rng(seed).integers(0, len(distinct), n)
    pts, idx = P.llvq_encode_blocks(ctx, torch.from_numpy(distinct[which]).cuda(), getattr(P, "LLVQ_" + metric))
    return pts.cpu().numpy(), idx.cpu().numpy().view(np.uint64), which


@pytest.mark.parametrize("metric,code", [("EUCLIDEAN", (2, 13)), ("EUCLIDEAN", (2, 20)), ("ANGULAR", (2, 11)), ("ANGULAR", (2, 12)), ("ANGULAR", (2, 13)), ("ANGULAR", (2, 20))])
def test_hard_inputs_with_two_lanes_per_vector(oracle_mod, metric, code):
    o = oracle_mod.Code(*code)
    kinds = ["midpoints", "deep_holes", "half_integers", "near_the_sphere", "lattice_directions", "all_lengths"]
    distinct = np.concatenate([_inputs(400, 9)] + [_edge_inputs(o, kind, 157).astype(np.float32) for kind in kinds])
    want, index = o.encode(distinct.astype(np.float64), getattr(oracle_mod, metric), threads=16)
    index = np.array(index, dtype=np.uint64)
    # not finite: the point of index 0, whatever its neighbours in the warp are
    bad = _inputs(30, 10)
    bad[np.arange(30), np.arange(30) % 24] = np.array([np.nan, np.inf, -np.inf])[np.arange(30) % 3]
    zero = np.zeros((30, 24), dtype=np.int8)
    zero[:, :2] = 4
    distinct, want, index = np.concatenate([distinct, bad]), np.concatenate([want, zero]), np.concatenate([index, np.zeros(30, dtype=np.uint64)])
    pts, idx, which = _pair_form(code, distinct, metric)
    assert np.array_equal(pts, want[which]) and np.array_equal(idx, index[which])


@pytest.mark.parametrize("exponent", [-141, -126, -100, 60, 100, 124])
def test_angular_search_at_extreme_lengths_with_two_lanes_per_vector(oracle_mod, exponent):
    # a power of two changes neither the direction nor any rounding: eight significant bits stay exact also where the inputs are subnormal
    o = oracle_mod.Code(2, 12)
    v = torch.from_numpy(_inputs(500, 11)).bfloat16().float().clamp(-7, 7)
    v = ((v * 16).round() / 16).numpy()
    scaled = (v.astype(np.float64) * 2.0 ** exponent).astype(np.float32)
    assert np.array_equal(scaled.astype(np.float64), v.astype(np.float64) * 2.0 ** exponent)
    want, _ = o.encode(v.astype(np.float64), oracle_mod.ANGULAR, threads=16)
    pts, _, which = _pair_form((2, 12), scaled, "ANGULAR")
    assert np.array_equal(pts, want[which])


def test_more_vectors_wait_than_a_block_lists(oracle_mod):
    # of integers every other vector has several nearest cosets (some 140 of the 256 that a thread block has at a time, up to 32 each), midpoints have up to 48
    o = oracle_mod.Code(2, 13)
    distinct = np.concatenate([np.round(np.random.default_rng(12).standard_normal((600, 24)) * 2.5), _edge_inputs(o, "midpoints", 157)]).astype(np.float32)
    want, index = o.encode(distinct.astype(np.float64), oracle_mod.EUCLIDEAN, threads=16)
    pts, idx, which = _pair_form((2, 13), distinct, "EUCLIDEAN", seed=4)
    assert np.array_equal(pts, want[which]) and np.array_equal(idx, np.array(index, dtype=np.uint64)[which])
