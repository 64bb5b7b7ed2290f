"""Parity of tman_mpgemv (decode path) with the CPU oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import tman_oracle as orc
from paper_2511_11248_b200 import binding as B, helpers as H, synth
from parity import TOL, rel_err, run

pytestmark = pytest.mark.gpu


def run_gemv(c, dev=None, packed=None, pack="library"):
    y, ws, packed, dev = run(B.OP_GEMV, c, dev, packed, pack)
    return H.to_f64(y), ws, packed, dev


def check(c, pack="library"):
    got, *_ = run_gemv(c, pack=pack)
    ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
    e = rel_err(got, ref)
    assert e <= TOL, (c.name, e)
    return e


SMALL = [
    # (M, K, N, bits, group): ragged K-slices (K not a multiple of 1024), ragged column units,
    # single-slice K, every M, every bit width and group size
    (1, 128, 8, 4, 128), (1, 1024, 32, 2, 64), (1, 1152, 40, 2, 32), (1, 2048, 264, 4, 64),
    (1, 3584, 72, 3, 128), (2, 1024, 64, 2, 64), (2, 640, 24, 4, 32), (3, 2048, 136, 3, 64),
    (4, 1280, 520, 4, 128), (5, 1024, 48, 2, 128), (6, 512, 8, 3, 32), (7, 2304, 200, 4, 64),
    (8, 4096, 1032, 2, 64), (1, 18944, 16, 4, 128),
]


@pytest.mark.parametrize("M,K,N,bits,G", SMALL)
def test_small_cases(M, K, N, bits, G):
    check(synth.small_case(M, K, N, bits, G, seed=M * 1000 + bits * 10 + G))


@pytest.mark.parametrize("M,K,N,bits,G", SMALL[1::2] + [(1, 4096, 4096, 4, 64), (8, 4096, 14336, 2, 64)])
def test_on_a_buffer_the_oracle_packed(M, K, N, bits, G):
    # the kernels read a buffer that no GPU code produced: layout and lookup agree with the oracle's packing
    check(synth.small_case(M, K, N, bits, G, seed=M * 1000 + bits * 10 + G + 1), pack="oracle")


def test_pack_directly_followed_by_decode_on_one_stream():
    # the decode kernel reads weights before it waits for its predecessor; after a packing on the same
    # stream the library must order it behind the packing kernels.  No host synchronisation in between;
    # the result has to be bit-equal to a run on a buffer that was complete long before.
    c = synth.small_case(1, 4096, 4096, 2, 64, seed=77)
    dev = H.device_case(c)
    settled = H.pack_case(c, dev)
    torch.cuda.synchronize()
    want, *_ = run_gemv(c, dev, settled)
    ws = H.alloc_workspace(B.OP_GEMV, c.M, c.K, c.N, c.bits, c.group)
    fresh = H.alloc_packed(c.K, c.N, c.bits, c.group)
    for _ in range(5):
        fresh.zero_()
        y = H.alloc_y(c.M, c.N)
        B.tman_pack_weights(dev["codes"], dev["scales"], dev["zeros"], c.K, c.N, c.bits, c.group, fresh)
        B.tman_mpgemv(fresh, dev["x"], y, c.M, c.K, c.N, c.bits, c.group, ws)
        assert B.tman_read_status(ws) == 0
        assert np.array_equal(H.to_f64(y), want)


@pytest.mark.parametrize("M,rows_ws", [(8, 4), (8, 1), (3, 1), (5, 2)])
def test_smaller_workspace_means_more_passes_and_the_same_answer(M, rows_ws):
    # a workspace sized for fewer rows is accepted; the call then makes several passes over the weights
    K, N, bits, G = 2048, 264, 4, 64
    c = synth.small_case(M, K, N, bits, G, seed=60 + M)
    dev = H.device_case(c)
    packed = H.pack_case(c, dev)
    nbytes = B.tman_workspace_bytes(B.OP_GEMV, rows_ws, K, N, bits, G)
    plan = B.tman_debug_gemv_plan(M, K, N, bits, G, ws_limit=nbytes)
    assert len(plan["passes"]) >= 2
    ws = H.guarded_bytes(nbytes, "small workspace")
    B.tman_workspace_init(ws)
    y = H.alloc_y(M, N)
    B.tman_mpgemv(packed, dev["x"], y, M, K, N, bits, G, ws)
    assert B.tman_read_status(ws) == 0
    H.check_guards()
    ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
    assert rel_err(H.to_f64(y), ref) <= TOL


def test_a_wait_that_runs_out_ends_cleanly_with_status_timeout():
    # nothing ever writes the sums the kernel waits for: it must give up by itself and say so
    ws = H.alloc_workspace(B.OP_GEMV, 1, 4096, 4096, 2, 64)
    B.tman_debug_wait_timeout(ws, 2000)
    assert B.tman_read_status(ws) == 7          # TMAN_ERR_TIMEOUT
    # the context is intact and the workspace, prepared again, serves a real call
    B.tman_workspace_init(ws)
    c = synth.small_case(1, 1024, 32, 2, 64, seed=91)
    dev = H.device_case(c)
    y = H.alloc_y(1, 32)
    B.tman_mpgemv(H.pack_case(c, dev), dev["x"], y, 1, 1024, 32, 2, 64, ws)
    assert B.tman_read_status(ws) == 0
    assert rel_err(H.to_f64(y), orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)) <= TOL


@pytest.mark.parametrize("M,factor", [(2, 1.0), (4, 1.0), (8, 1.0), (2, 2.0 ** -12), (8, 2.0 ** 9)])
def test_rows_in_fp16_tables_stay_near_the_predicted_error(M, factor):
    # the CPU simulation of the fp16-row arithmetic (test_decode_precision_model.py) predicts <= 1.5e-3 whatever
    # the activations' magnitude; the kernel is held to 2e-3, well inside the 5e-3 bound
    c = synth.small_case(M, 4096, 520, 4, 128, seed=70 + M)
    c.x[:] = (c.x.astype(np.float32) * factor).astype(np.float16)
    got, *_ = run_gemv(c)
    ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
    assert rel_err(got, ref) <= 2e-3


@pytest.mark.parametrize("M,bits,G", [(1, 2, 64), (1, 3, 128), (1, 4, 32), (2, 4, 128), (3, 2, 32), (4, 4, 32)])
@pytest.mark.parametrize("K,N", [(128, 8), (1152, 40), (4096, 2304), (4096, 2312), (4096, 2368), (4096, 2376)])
def test_lookup_units_of_one_strip_and_the_line_above_them(M, bits, G, K, N):
    # 148 SMs: K = 4096 in slices of 512 or 1024 k leaves 576 or 592 strips of four columns to units of one strip.  One row: fp32
    # sums, the result rounded to fp16; more rows: fp16 tables, the bound of test_rows_in_fp16_tables_stay_near_the_predicted_error.
    c = synth.small_case(M, K, N, bits, G, seed=900 + M + K + N)
    dev = H.device_case(c)
    packed = H.pack_case(c, dev)
    ws = H.alloc_workspace(B.OP_GEMV, M, K, N, bits, G)
    ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
    for _ in range(2):                                       # the second call finds the workspace as the first left it
        y = H.alloc_y(M, N)
        B.tman_mpgemv(packed, dev["x"], y, M, K, N, bits, G, ws)
        assert B.tman_read_status(ws) == 0
        H.check_guards()
        assert rel_err(H.to_f64(y), ref) <= (5.1e-4 if M == 1 else 2e-3)


@pytest.mark.parametrize("M,bits,G", [(3, 3, 64), (3, 2, 128), (4, 2, 64), (4, 4, 128), (5, 2, 32), (5, 3, 64), (6, 2, 64), (7, 4, 32), (8, 2, 128), (8, 3, 128), (8, 4, 64)])
@pytest.mark.parametrize("K,Ns", [(128, (8,)), (640, (32, 40)), (2176, (264,)), (4096, (2056, 8, 40))])
def test_tensor_core_rows_at_the_edges_of_their_split(M, bits, G, K, Ns):
    check_grouped_twice(M, bits, G, K, Ns, 5.1e-4)


def check_grouped_twice(M, bits, G, K, Ns, bound):
    # one chunk of 128 k; a team with idle warps; a second K-slice of a single chunk; ragged groups of 32 columns and a
    # matrix narrower than one.  Codes and activations are exact operands and sums fp32, so what is left is the rounding of
    # the result to fp16, 2^-11 = 4.9e-4 of it, and fp32 sums of up to 4096 terms, below 1e-5.
    cases = [synth.small_case(M, K, N, bits, G, seed=800 + 10 * i + M, outliers=True) for i, N in enumerate(Ns)]
    for c in cases[1:]:
        c.x[:] = cases[0].x
    devs = [H.device_case(c) for c in cases]
    packed = [H.pack_case(c, d) for c, d in zip(cases, devs)]
    ws = H.alloc_workspace(B.OP_GEMV, M, K, sum(Ns), bits, G)
    for _ in range(2):                                       # the second call finds the workspace as the first left it
        ys = [H.alloc_y(M, N) for N in Ns]
        B.tman_mpgemv_grouped(packed, devs[0]["x"], ys, M, K, Ns, bits, G, ws)
        assert B.tman_read_status(ws) == 0
        H.check_guards()
        for c, y in zip(cases, ys):
            ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
            assert rel_err(H.to_f64(y), ref) <= bound


@pytest.mark.parametrize("M,bits,G,K,N", [(M, b, G, K, 4104) for K in (2176, 4096) for M, b, G in
                                          [(3, 3, 64), (3, 2, 64), (4, 2, 128), (4, 4, 128), (5, 2, 32), (6, 2, 64), (8, 2, 128), (8, 3, 128),
                                                       (8, 4, 32)]] + [(8, 3, 64, 16384, 4736)])
def test_tensor_core_rows_with_two_chunks_a_warp(M, bits, G, K, N):
    # an odd number of chunks (the last warp at work has one), one K-slice and four; the bound of the test above, whose chunks here
    # share a scale two by two (an activation below 2^-21 of a pair's largest is off by up to 2^-32 of that: below the fp32 sums' rounding)
    plan = B.tman_debug_gemv_plan(M, K, N, bits, G)
    assert plan["passes"][0]["words"] == 128, plan           # 16 warps x 2 chunks x 4 plane words
    test_tensor_core_rows_at_the_edges_of_their_split(M, bits, G, K, (N,))


@pytest.mark.parametrize("M,bits,G,K", [(4, 4, 128, 4096), (8, 3, 64, 4096), (8, 2, 32, 1152), (3, 2, 128, 640)])
def test_tensor_core_rows_with_a_large_spread_of_activations(M, bits, G, K):
    check_large_spread(M, bits, G, K, 40)


def check_large_spread(M, bits, G, K, N):
    # Activations from 2^-24 to 2^4 side by side (sums of larger ones would leave fp16's range): below 2^-21 of the largest neighbour
    # they lose bits as operands, at most 2^-32 of it each, far below the bound of the tests above
    c = synth.small_case(M, K, N, bits, G, seed=700 + M + K)
    rng = np.random.default_rng(M + K)
    x = rng.standard_normal((M, K)) * 2.0 ** rng.integers(-24, 0, size=(M, K))
    big = np.arange(0, K, 37)
    x[:, big] = 2.0 ** 4 * rng.choice([-1.0, 1.0], size=(M, big.size))
    c.x[:] = x.astype(np.float16)
    got, *_ = run_gemv(c)
    ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
    assert rel_err(got, ref) <= 5.1e-4


def on_digits(M, K, N, bits, G):
    """Whether the call is one pass on the integer tensor cores."""
    return [p["kernel"] for p in B.tman_debug_gemv_plan(M, K, N, bits, G)["passes"]] == ["digits"]


# (K, Ns, (M, bits, group) ...), all of them on the integer tensor cores
ONE_TILE = [(1, b, 64) for b in (2, 3, 4)] + [(M, b, 128) for M in (1, 2) for b in (2, 3, 4)]
TWO_TILES = [(1, 2, 32), (2, 2, 64), (2, 3, 64), (2, 4, 64)]
DIGIT_CASES = [
    # one chunk of 128 k, matrices narrower than a group of 32 columns; 15 chunks, a CTA's columns from several matrices
    (128, (64, 8, 8), ONE_TILE + TWO_TILES + [(1, 3, 32), (1, 4, 32)]), (1536, (8, 760, 16), ONE_TILE + TWO_TILES), (1920, (328, 1600), ONE_TILE + TWO_TILES),
    # model shapes and the longest K
    (2048, (2048, 512, 512), ONE_TILE + TWO_TILES), (4096, (4096,), [(1, 2, 64), (1, 4, 128), (2, 2, 128), (2, 3, 128)]),
    (4096, (2056, 1024, 1024), [(1, 2, 128), (1, 4, 64), (2, 4, 128)]), (4992, (2504,), [(2, 2, 128)]), (5120, (5120,), [(2, 4, 128)]),
    # two, four and eight teams of four, two and one warps
    (128, (4000, 776), ONE_TILE + TWO_TILES), (640, (9216,), [(1, 4, 32)]), (128, (9512,), [(1, 2, 64), (2, 3, 128), (2, 4, 64)]),
    (128, (19064,), [(2, 3, 128), (2, 4, 64)]),
    # two CTAs an SM, rings of one and of two units, teams of two warps and of one
    (640, (20000, 4104), [(1, 2, 64), (1, 3, 128), (1, 4, 64), (1, 4, 32), (2, 2, 128), (2, 4, 128)]), (128, (38216,), [(1, 2, 128), (2, 4, 64)]),
    (3200, (26120,), [(1, 2, 64), (1, 4, 64)]),
    # more turns than the warps' sums have room for: several reductions
    (1152, (4776,), [(2, 3, 128)]), (640, (11880,), [(2, 3, 128)]), (640, (24104,), [(2, 3, 128)]), (1920, (11288,), [(2, 4, 64)]),
    (1152, (24104,), [(1, 3, 64)]), (1920, (15536,), [(2, 2, 128)]), (1408, (20576,), [(2, 4, 128)]),
    # the other length of the rings, and all of an SM's shared memory
    (1408, (368,), [(2, 3, 64)]), (3712, (944,), [(2, 2, 128), (2, 4, 128)]), (2944, (3592,), [(2, 2, 64), (2, 4, 64)]), (2176, (4776,), [(2, 3, 128)]),
]


@pytest.mark.parametrize("K,Ns,M,bits,G", [(K, Ns, *c) for K, Ns, cs in DIGIT_CASES for c in cs])
def test_one_and_two_rows_on_the_integer_tensor_cores(K, Ns, M, bits, G):
    # Sums are exact up to a block; an activation is rounded by at most 2^-24 of its block's largest, so what is left is the rounding of
    # the result to fp16 and fp32 sums: the bound of test_tensor_core_rows_at_the_edges_of_their_split
    assert on_digits(M, K, sum(Ns), bits, G)
    check_grouped_twice(M, bits, G, K, Ns, 5.1e-4)


@pytest.mark.parametrize("K,Ns,M,bits,G", [(4096, (504,), 1, 4, 128), (2048, (1032,), 2, 2, 32), (4096, (16392,), 1, 4, 128), (5248, (2504,), 1, 2, 64),
                                           (3584, (1024, 2056), 1, 3, 64), (2304, (4096, 2056), 2, 3, 64)])
def test_one_and_two_rows_beyond_the_rule_by_lookup(K, Ns, M, bits, G):
    # (two rows: the bound of test_rows_in_fp16_tables_stay_near_the_predicted_error)
    assert [p["kernel"] for p in B.tman_debug_gemv_plan(M, K, sum(Ns), bits, G)["passes"]] == ["lookup"]
    check_grouped_twice(M, bits, G, K, Ns, 2e-3 if M > 1 else 5.1e-4)


@pytest.mark.parametrize("M,bits,G", [(1, 2, 64), (1, 4, 128), (2, 3, 128), (2, 2, 64), (1, 2, 32), (2, 4, 64)])
def test_digits_with_a_large_spread_of_activations(M, bits, G):
    # as above, 2^-24 to 2^4 side by side
    assert on_digits(M, 1536, 784, bits, G)
    check_large_spread(M, bits, G, 1536, 784)


@pytest.mark.parametrize("M,bits,G", [(1, 2, 64), (1, 3, 64), (1, 2, 32), (1, 4, 64), (2, 4, 64), (2, 2, 64)])
def test_digits_with_blocks_of_very_different_size(M, bits, G):
    # every other block has activations of about 1000 under the smallest scale, 2^-24, its neighbours activations of about 2^-10 under scales
    # near 1, which make up nearly all of the result.  Rounded to a part of the neighbours' largest (3000 x 2^-25 at 2 bits), they would be off
    # by percents; rounded to a part of their own block's, by nothing that shows.
    c = synth.small_case(M, 1536, 784, bits, G, seed=9 + M)
    assert on_digits(M, c.K, c.N, bits, G)
    rng = np.random.default_rng(bits * G)
    small = (np.arange(c.K) // G) % 2 == 1
    c.x[:] = (rng.standard_normal((M, c.K)) * np.where(small, 2.0 ** -10, 1000.0)).astype(np.float16)
    c.scales[:] = np.where(small[::G, None], rng.uniform(0.5, 1.0, c.scales.shape), 2.0 ** -24).astype(np.float16)
    got, *_ = run_gemv(c)
    assert rel_err(got, orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)) <= 5.1e-4


@pytest.mark.parametrize("bits,G", [(2, 128), (4, 64), (3, 64)])
def test_digits_with_an_infinity_and_a_nan(bits, G):
    # the definition column by column: s (q - z) inf is an infinity of the sign of q - z, NaN where q = z; a NaN reaches every column
    c = synth.small_case(2, 1536, 784, bits, G, seed=5)
    assert on_digits(2, c.K, c.N, bits, G)
    c.x[0, 700] = -np.inf
    c.x[1, 3] = np.nan
    dev = H.device_case(c)
    ws, y = H.alloc_workspace(B.OP_GEMV, 2, c.K, c.N, bits, G), H.alloc_y(2, c.N)
    B.tman_mpgemv(H.pack_case(c, dev), dev["x"], y, 2, c.K, c.N, bits, G, ws)
    got = H.to_f64(y)
    d = c.codes[700].astype(np.int64) - c.zeros[700 // G].astype(np.int64)
    assert np.all(np.isnan(got[1])) and np.all(np.isnan(got[0, d == 0]))
    assert np.all(np.isinf(got[0, d != 0])) and np.array_equal(got[0, d != 0] > 0, d[d != 0] < 0)


@pytest.mark.parametrize("M,bits,G", [(1, 2, 128), (2, 3, 128), (2, 4, 64), (1, 2, 32)])
@pytest.mark.parametrize("other", [701, 702, 736, 800, 1500])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_digits_with_two_infinities(M, bits, G, other, sign):
    # two infinities, of one block (the first two, and up to G = 128 the others) or of two: wherever the definition has infinities of both
    # signs, or an infinity that meets its zero-point, the sum is NaN; nothing finite comes out where it has an infinity
    c = synth.small_case(M, 1536, 784, bits, G, seed=6)
    assert on_digits(M, c.K, c.N, bits, G)
    c.x[M - 1, 700], c.x[M - 1, other] = np.inf, sign * np.inf
    dev = H.device_case(c)
    ws, y = H.alloc_workspace(B.OP_GEMV, M, c.K, c.N, bits, G), H.alloc_y(M, c.N)
    B.tman_mpgemv(H.pack_case(c, dev), dev["x"], y, M, c.K, c.N, bits, G, ws)
    got = H.to_f64(y)[M - 1]
    d0 = c.codes[700].astype(np.int64) - c.zeros[700 // G].astype(np.int64)
    d1 = (c.codes[other].astype(np.int64) - c.zeros[other // G].astype(np.int64)) * int(sign)
    nan = d0 * d1 <= 0
    assert nan.any() and not nan.all()
    assert np.all(np.isnan(got[nan])) and not np.any(np.isfinite(got))
    if other // G != 700 // G:
        assert np.array_equal(got[~nan], np.where(d0[~nan] > 0, np.inf, -np.inf))


def test_repeat_calls_share_workspace_and_agree():
    c = synth.small_case(2, 2048, 264, 4, 64, seed=21)
    dev = H.device_case(c)
    packed = H.pack_case(c, dev)
    ws = H.alloc_workspace(B.OP_GEMV, c.M, c.K, c.N, c.bits, c.group)
    ys = []
    for _ in range(3):
        y = H.alloc_y(c.M, c.N)
        B.tman_mpgemv(packed, dev["x"], y, c.M, c.K, c.N, c.bits, c.group, ws)
        ys.append(y)
    assert B.tman_read_status(ws) == 0
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[1], ys[2])   # fixed summation order


def test_exact_special_cases():
    # all-zero codes with z = 0 give exactly zero; codes == zero-point give (near) zero
    c = synth.small_case(1, 2048, 64, 4, 64, seed=22)
    c.codes[:] = 0
    c.zeros[:] = 0
    got, *_ = run_gemv(c)
    assert np.all(got == 0.0)
    # integers, unit scale, zero zero-point: exact (all sums are small integers)
    rng = np.random.default_rng(3)
    c = synth.small_case(2, 1024, 32, 3, 64, seed=23)
    c.x[:] = rng.integers(-4, 5, size=c.x.shape).astype(np.float16)
    c.scales[:] = 1.0
    c.zeros[:] = 0
    got, *_ = run_gemv(c)
    want = c.x.astype(np.int64) @ c.codes.astype(np.int64)
    assert np.array_equal(got, want.astype(np.float64))
    # one-hot activation reads out single weights
    c = synth.small_case(1, 1024, 32, 4, 64, seed=24)
    c.x[:] = 0
    c.x[0, 777] = 1.0
    got, *_ = run_gemv(c)
    want = c.scales.astype(np.float64)[777 // 64] * (c.codes[777].astype(np.float64) - c.zeros[777 // 64])
    assert np.allclose(got[0], want.astype(np.float16).astype(np.float64), rtol=1e-3, atol=1e-6)


def test_config1_full():
    check(synth.config1())


@pytest.mark.parametrize("spec", synth.config2_specs(), ids=lambda s: s[0])
def test_config2_full(spec):
    check(synth.case_from_spec(spec))


@pytest.mark.parametrize("spec", synth.config3_specs(), ids=lambda s: s[0])
def test_config3_full(spec):
    check(synth.case_from_spec(spec))


@pytest.mark.parametrize("M,K,Ns,bits,G", [
    (1, 2048, (264, 72), 4, 64), (1, 4096, (1032, 1032, 40), 2, 64), (3, 1024, (48, 8, 136, 24), 3, 128),
    (2, 1152, (40, 520), 2, 32), (1, 4096, (14336, 14336), 2, 64),
])
def test_grouped_matches_oracle_and_single_calls(M, K, Ns, bits, G):
    # several matrices that share the activations, one launch (shared table precomputation)
    cases = [synth.small_case(M, K, N, bits, G, seed=400 + i) for i, N in enumerate(Ns)]
    for c in cases[1:]:
        c.x[:] = cases[0].x
    devs = [H.device_case(c) for c in cases]
    packed = [H.pack_case(c, d) for c, d in zip(cases, devs)]
    ws = H.alloc_workspace(B.OP_GEMV, M, K, sum(Ns), bits, G)
    ys = [H.alloc_y(M, N) for N in Ns]
    B.tman_mpgemv_grouped(packed, devs[0]["x"], ys, M, K, Ns, bits, G, ws)
    assert B.tman_read_status(ws) == 0
    H.check_guards()
    for c, d, pk, y in zip(cases, devs, packed, ys):
        ref = orc.mpgemm(c.x, c.codes, c.scales, c.zeros, c.group)
        assert rel_err(H.to_f64(y), ref) <= TOL
        single, *_ = run_gemv(c, d, pk)
        assert rel_err(H.to_f64(y), single) <= 1e-3   # same kernels; the split-K summation order may differ
