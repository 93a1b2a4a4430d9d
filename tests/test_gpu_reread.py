"""The re-read score kernel where its rules change path: 64 / 65 text rows (pass 1
with M = 64 or 128, mixed in one batch), partial and single tiles, one and several
head groups, and logits that leave the reference of the first tile far behind
(upwards, so that pass 1 redoes a tile, and downwards)."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_scores_close, to_device
from paper_2506_07416_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sel():
    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_2506_07416_gb300 import select
    return select


def _w(name, n, t, hq, hkv, d=128, dtype="bf16", sigma=0.3, seed=41):
    return inputs.Workload(name, len(n), list(n), list(t), hq, hkv, d, 256, dtype, keep_ratio=0.3, sigma=sigma,
                           seed=seed)


CASES = [
    _w("rows_64_65_128", [300, 257, 128, 1, 640], [64, 65, 128, 1, 63], 8, 4),
    _w("rows_up_to_64", [129, 127, 900], [64, 17, 1], 8, 8),
    _w("d64_rows", [300, 513], [65, 33], 14, 2, d=64),
    _w("e4m3_rows", [700, 130, 128], [32, 128, 64], 8, 8, dtype="e4m3"),
    _w("long_one_head", [5000], [100], 1, 1),
    _w("pack7_126_rows", [300, 128, 77], [18, 5, 1], 14, 2),
    _w("pack7_63_rows", [300, 129], [9, 4], 7, 1, d=64),
    _w("pack4_128_rows", [513, 40, 1200], [32, 31, 7], 16, 4),
    _w("pack2_of_4", [257, 640], [64, 33], 8, 2),
    _w("pack4_e4m3", [400, 129], [16, 3], 8, 2, dtype="e4m3"),
]


def _scores(s, x, xd):
    g = s.score(xd["q"], xd["text_offsets"], xd["k"], xd["seq_offsets"], xd["q_scale"], xd["k_scale"],
                seq_offsets_h=x["seq_offsets"], text_offsets_h=x["text_offsets"])
    s.check_device()
    return g.cpu().numpy()


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_rows_tiles_and_groups(sel, w):
    x = inputs.make_numpy(w)
    xd = to_device(x, w)
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel="reread")
    assert s.score_plan(x["text_offsets"], x["seq_offsets"])[0] == 1
    o = oracle.score(x["q"], x["k"], x["seq_offsets"], x["text_offsets"], w.hq, w.hkv, w.head_dim, w.dtype,
                     x["q_scale"], x["k_scale"])
    g = _scores(s, x, xd)
    assert_scores_close(g, o, w.dtype)
    np.testing.assert_array_equal(g, _scores(s, x, xd))
    s.close()


RESIDENT = [
    (_w("rows_63", [300, 129], [9, 4], 7, 1), "resident"),          # hp 7: one row of the 64 is no head's
    (_w("rows_64", [513, 40, 1200], [16, 7, 1], 16, 4), "resident"),
    (_w("rows_64_uniform", [1500] * 9, [16] * 9, 8, 2), "resident_flat"),
    (_w("rows_8_d64", [700, 128], [1, 1], 16, 2, d=64), "resident_1buf"),
    (_w("rows_60_two_buffers", [900, 257, 1], [15, 8, 3], 16, 4), "resident_2buf"),
    (_w("rows_48_e4m3", [400, 1290], [16, 3], 12, 4, dtype="e4m3"), "resident"),
    (_w("not_packed", [400, 1290], [33, 3], 12, 4), "resident"),
]


@pytest.mark.parametrize("w,kernel", RESIDENT, ids=[w.name for w, _ in RESIDENT])
def test_packed_heads_in_the_resident_kernel(sel, w, kernel):
    x = inputs.make_numpy(w)
    xd = to_device(x, w)
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel=kernel)
    assert s.score_plan(x["text_offsets"], x["seq_offsets"])[0] >= 2
    o = oracle.score(x["q"], x["k"], x["seq_offsets"], x["text_offsets"], w.hq, w.hkv, w.head_dim, w.dtype,
                     x["q_scale"], x["k_scale"])
    g = _scores(s, x, xd)
    assert_scores_close(g, o, w.dtype)
    np.testing.assert_array_equal(g, _scores(s, x, xd))
    s.close()


@pytest.mark.parametrize("kernel", ["reread", "resident"])
@pytest.mark.parametrize("query", ["all", "last"])
@pytest.mark.parametrize("t", [[18, 7], [30, 11], [9, 3]])
def test_packed_heads_with_the_full_key_set(sel, t, query, kernel):
    w = _w("packed_full", [300, 150], t, 14, 2)
    x = inputs.make_numpy(w)
    xd = to_device(x, w)
    n_sys = [5, 0]
    c = inputs.context_keys_numpy(w, n_sys, seed=24)
    dev = lambda a: torch.from_numpy(a.view(np.int16).copy()).view(torch.bfloat16).cuda()
    sys_off = np.concatenate([[0], np.cumsum(n_sys)]).astype(np.int32)
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel=kernel,
                     query=query)
    out = s.score_full_keys(xd["q"], xd["text_offsets"], xd["k"], xd["seq_offsets"], dev(c["k_sys"]),
                            torch.from_numpy(sys_off).cuda(), dev(c["k_txt"]), seq_offsets_h=x["seq_offsets"],
                            text_offsets_h=x["text_offsets"], sys_offsets_h=sys_off)
    s.check_device()
    if query == "all":
        o = oracle.score_full(x["q"], x["k"], c["k_sys"], c["k_txt"], x["seq_offsets"], x["text_offsets"], sys_off,
                              w.hq, w.hkv, w.head_dim, w.dtype)
    else:  # the last text row sees every text key: a one-row request whose other text keys count as system keys
        to = x["text_offsets"]
        rows = np.array([to[1] - 1, to[2] - 1])
        ks = np.concatenate([c["k_sys"], c["k_txt"][:to[1] - 1], c["k_txt"][to[1]:to[2] - 1]])
        so2 = np.array([0, 5 + t[0] - 1, 5 + t[0] - 1 + t[1] - 1], np.int32)
        o = oracle.score_full(x["q"][rows], x["k"], ks, c["k_txt"][rows], x["seq_offsets"],
                              np.arange(3, dtype=np.int32), so2, w.hq, w.hkv, w.head_dim, w.dtype)
    assert_scores_close(out.cpu().numpy(), o, w.dtype)
    s.close()


@pytest.mark.parametrize("t", [20, 64, 100])
@pytest.mark.parametrize("later", [40.0, -40.0])
def test_logits_far_from_the_first_tiles_reference(sel, t, later):
    # every query is one unit direction times 10; the keys of the first 128 tokens lie near 0 along it, those
    # of token 200 on at `later` +- 1: logits 10 * later / sqrt(128) = +-35 and, times 4 in token 333, +-141 nats
    # (204 in log2), beyond the 12 that pass 1 lets a term exceed its reference by.
    # x = s * c - b is rounded at |x| <= 2 * 204: relative error of 2^x up to 408 * 2^-24 * ln 2 = 1.7e-5,
    # well inside the bf16 bound of 2e-3.
    w = _w("far", [700], [t], 4, 2)
    rng = np.random.Generator(np.random.PCG64(3))
    d = rng.standard_normal(128)
    d /= np.linalg.norm(d)
    q = 10.0 * d + 0.02 * rng.standard_normal((t, w.hq, 128))
    k = 0.1 * rng.standard_normal((700, w.hkv, 128))
    k[200:] += (later + rng.standard_normal((500, w.hkv, 1))) * d
    k[333] *= 4.0
    x = {"q": inputs.f32_to_bf16_bits(q.astype(np.float32)), "k": inputs.f32_to_bf16_bits(k.astype(np.float32)),
         "seq_offsets": w.seq_offsets(), "text_offsets": w.text_offsets(), "q_scale": 1.0, "k_scale": 1.0}
    xd = to_device(x, w)
    s = sel.Selector(1, 700, t, w.hq, w.hkv, 128, "bf16", score_kernel="reread")
    o = oracle.score(x["q"], x["k"], x["seq_offsets"], x["text_offsets"], w.hq, w.hkv, 128, "bf16")
    assert_scores_close(_scores(s, x, xd), o, "bf16")
    s.close()


@pytest.mark.parametrize("kernel", ["reread", "resident"])
def test_scales_whose_product_vanishes(sel, kernel):
    """Two e4m3 scales of 1e-25: every logit is 0 in 32 bits, so a request's tokens share its score, also where its
    last tile is partly empty."""
    w = _w("tiny_scales", [300, 128, 1], [20, 65, 3], 4, 2, dtype="e4m3")
    x = inputs.make_numpy(w)
    x["q_scale"] = x["k_scale"] = 1e-25
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel=kernel)
    g = _scores(s, x, to_device(x, w))
    for b in range(3):
        n0, n1 = x["seq_offsets"][b:b + 2]
        np.testing.assert_allclose(g[n0:n1], 1.0 / (n1 - n0), rtol=2e-6)  # fp32 sums of up to 300 ones and 260 rows
    s.close()


@pytest.mark.parametrize("count", [1, 7, 60])
def test_row_statistics_far_above_the_first_reference(sel, count):
    """One text row and head whose largest logits, `count` of them around 0, lie 60 to 90 log2 units above those of
    the first tiles. Each logit is one exact product, so a score's relative error is that of the row's statistic b and
    of one 2^x, in units of log2: half a step of an exponent up to 16 in pass 1 and of b (2^-21 each), of an exponent
    up to 8 in pass 2 (2^-22), one step of the logarithm of a sum below 2^22 (2^-19), and 2^-22 for either 2^x. Times
    ln 2: 2.4e-6 in all."""
    bound = (2 * 2.0 ** -21 + 2.0 ** -22 + 2.0 ** -19 + 2 * 2.0 ** -22) * np.log(2)
    rng = np.random.Generator(np.random.PCG64(count))
    n = 700
    c = 1.4426950408889634 / np.sqrt(128)
    q = np.zeros((1, 1, 128), np.float32)
    q[..., 0] = 8.0
    s = sel.Selector(1, n, 1, 1, 1, 128, "bf16", score_kernel="reread")
    so, to = np.array([0, n], np.int32), np.array([0, 1], np.int32)
    for gap in range(60, 92, 2):
        k = np.zeros((n, 1, 128), np.float32)
        k[:, 0, 0] = -gap / (8.0 * c) + 0.3 * rng.standard_normal(n)
        k[300:300 + count, 0, 0] = 0.3 * rng.standard_normal(count)
        x = {"q": inputs.f32_to_bf16_bits(q), "k": inputs.f32_to_bf16_bits(k), "seq_offsets": so, "text_offsets": to}
        o = oracle.score(x["q"], x["k"], so, to, 1, 1, 128, "bf16")
        g = _scores(s, x, to_device(x, None))
        top = slice(300, 300 + count)
        assert np.abs(g[top] / o[top] - 1).max() < bound, gap
    s.close()


@pytest.mark.parametrize("n,t,hq,hkv", [
    ([1537, 1700, 1410, 1664] * 8, [128, 33, 16, 65, 1], 16, 16),   # 128-row instance, all row counts in one batch
    ([1537, 1700, 1410, 1664] * 10, [16, 9, 31], 64, 16),            # packed heads, 124 rows
    ([1664, 3000, 129] * 10, [64, 17], 16, 16),                      # 64-row instance, 2-tile requests among them
], ids=["rows_128", "packed", "rows_64"])
def test_long_e4m3_requests(sel, n, t, hq, hkv):
    """From 12 tiles a request on, e4m3 runs on four epilogue warpgroups."""
    t = [t[i % len(t)] for i in range(len(n))]
    w = _w("long_e4m3", n, t, hq, hkv, dtype="e4m3")
    assert sum((x + 127) // 128 for x in n) >= 12 * len(n)
    x = inputs.make_numpy(w)
    xd = to_device(x, w)
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel="reread")
    assert tuple(s.score_plan(x["text_offsets"], x["seq_offsets"])[:2]) == (1, 1)
    o = oracle.score(x["q"], x["k"], x["seq_offsets"], x["text_offsets"], w.hq, w.hkv, w.head_dim, w.dtype,
                     x["q_scale"], x["k_scale"])
    g = _scores(s, x, xd)
    assert_scores_close(g, o, w.dtype)
    for _ in range(4):  # whichever CTA takes an item, and behind whichever items, its scores are the same
        np.testing.assert_array_equal(g, _scores(s, x, xd))
    s.close()


def test_no_alloc_limit_does_not_follow_the_plan(sel):
    """A batch whose chosen launch would need more partial rows than the static scratch holds, but whose fixed
    shape does not, is still taken."""
    for copies in (3, 4, 5, 6, 8, 10):
        w = _w("limit", [2600, 1800, 3000, 2400] * copies, [100, 65, 90, 128] * copies, 32, 8)
        so, to = w.seq_offsets(), w.text_offsets()
        s = sel.Selector(w.batch, w.total_vis, w.total_txt, 32, 8, 128, "bf16")
        plan = s.score_plan(to, so)
        if plan[3] * w.total_vis > 1 << 20:
            break
        s.close()
    else:
        pytest.fail("no batch among these splits its heads beyond the scratch")
    xd = inputs.make_torch(w, "cuda")
    ref = s.score(xd["q"], xd["text_offsets"], xd["k"], xd["seq_offsets"], seq_offsets_h=so, text_offsets_h=to)
    s.check_device()
    out = torch.full((w.total_vis,), float("nan"), device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    sel.score_noalloc(32, 8, 128, "bf16", w.batch, xd["q"], xd["text_offsets"], to, xd["k"], xd["seq_offsets"], so,
                      1.0, 1.0, out, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    # two kernels, sums in another order: 32-bit rounding over at most 128 * 32 terms a score
    assert float(((out - ref).abs() / ref).max()) < 1e-5
    s.close()


@pytest.mark.parametrize("n,t,hq,hkv,d", [
    ([130, 64, 0, 257, 1] * 40, [3, 64, 5, 20, 65], 4, 4, 128),  # five sizes, empty requests among them
    ([128] * 180, [16] * 5, 2, 1, 64),                            # one tile, one head block each
    ([900, 129] * 60, [100, 70, 30, 9, 128], 8, 2, 128),
], ids=["mixed_empty", "one_tile", "two_sizes"])
def test_more_items_than_ctas(sel, n, t, hq, hkv, d):
    """More (request, head group) items than CTAs run at once: the CTAs claim the
    rest among themselves, and the claims are back at zero for the next launch."""
    t = [t[i % len(t)] for i in range(len(n))]
    w = _w("claims", n, t, hq, hkv, d)
    x = inputs.make_numpy(w)
    xd = to_device(x, w)
    s = sel.Selector(w.batch, w.total_vis, w.total_txt, w.hq, w.hkv, w.head_dim, w.dtype, score_kernel="reread")
    plan = s.score_plan(x["text_offsets"], x["seq_offsets"])
    assert plan[0] == 1 and plan[1] == 1
    assert plan[3] * w.batch > torch.cuda.get_device_properties(0).multi_processor_count
    o = oracle.score(x["q"], x["k"], x["seq_offsets"], x["text_offsets"], w.hq, w.hkv, w.head_dim, w.dtype,
                     x["q_scale"], x["k_scale"])
    g = _scores(s, x, xd)
    assert_scores_close(g, o, w.dtype)
    for _ in range(2):  # whichever CTA takes an item, its scores are the same
        np.testing.assert_array_equal(g, _scores(s, x, xd))
    s.close()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        out = torch.full((w.total_vis,), float("nan"), device="cuda")
        sel.score_noalloc(w.hq, w.hkv, w.head_dim, w.dtype, w.batch, xd["q"], xd["text_offsets"], x["text_offsets"],
                          xd["k"], xd["seq_offsets"], x["seq_offsets"], x["q_scale"], x["k_scale"], out, err)
        assert_scores_close(out.cpu().numpy(), o, w.dtype)
        assert int(err.item()) == 0
