"""Kernels and dispatch rules at the sizes where they can go wrong, against the CPU oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_2609_35800_gb300 as hg
from paper_2609_35800_gb300 import workloads as wl
from paper_2609_35800_gb300.runner import CacheRunner

from parity import assert_close, attention_reference, bits16, check_arena_layer, n_salient, oracle_layer
from test_gpu_parity import _dequantize_bit_exact, _run_and_check

pytestmark = pytest.mark.gpu

SIGMA = float(np.float32(1.0 / np.sqrt(128.0)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_35800_gb300 import build
    build.build()


def _row_reference(runner, layer, row, k, v, q, news):
    """fp64 attention of one batch row: the oracle on that row's prefill plus the appended tokens."""
    w = runner.w
    o = oracle.quantize_layer(bits16(k[row:row + 1]), bits16(v[row:row + 1]), w.img_start, w.image, w.base, w.bits,
                              runner.mask[layer], int(w.keys_only), w.kivi_group_tokens, w.kivi_group_channels,
                              w.kivi_residual, meta16=w.meta_bits == 32, n_salient=n_salient(w))
    ak = [bits16(kn[layer, row:row + 1]) for kn, _ in news]
    av = [bits16(vn[layer, row:row + 1]) for _, vn in news]
    return attention_reference(runner, o, bits16(q[layer, row:row + 1]), ak, av, SIGMA)


@pytest.mark.parametrize("name,layers", [("internvl25_8b", 1), ("qwen25vl72b", 1), ("internvl25_8b", 3)])
def test_decode_in_several_waves(name, layers):
    """One layer of a large batch: heads too large to balance in one wave run as two to three waves of
    smaller chunks (more than 1,024 of them over three layers)."""
    w = dataclasses.replace(wl.WORKLOADS[name], layers=layers, decode_steps=2)
    runner = CacheRunner(w)
    kept = runner.quantize_all(keep=True)
    news = []
    for step in range(2):
        k_new, v_new = wl.step_new_kv(w, step, "cuda")
        q = wl.step_query(w, step, "cuda")
        out = runner.decode_step(step, q=q, k_new=k_new, v_new=v_new)
        news.append((k_new, v_new))
    for layer in {0, layers - 1}:
        for row in (0, w.batch - 1):
            ref = _row_reference(runner, layer, row, *kept[layer], q, news)
            assert_close(bits16(out[layer, row:row + 1]), ref, "%s layer %d row %d" % (name, layer, row))


@pytest.mark.parametrize("base,keys_only,prefix", [(wl.BASE_MINMAX, 0, 0), (wl.BASE_MINMAX, 1, 64),
                                                   (wl.BASE_AKVQ, 0, 64), (wl.BASE_KIVI, 1, 32)])
def test_decode_layers_with_different_appended_counts(base, keys_only, prefix):
    """Layers of one launch that hold 0, 1 and 70 appended tokens: the launch's chunk counts are the
    largest layer's, so the others have an empty last BF16 chunk (with no text at all, an empty only one)."""
    w = wl.custom("uneven", 3, 2, 8, 4, prefix, 320, 0, base, 2, keys_only, decode_steps=70, seed=5,
                  protected=[(0, 1), (1, 0), (2, 3)], residual=0)
    runner = CacheRunner(w)
    kept = runner.quantize_all(keep=True)
    counts = (0, 1, 70)
    news = [wl.step_new_kv(w, s, "cuda") for s in range(70)]
    for layer, n in enumerate(counts):
        for k_new, v_new in news[:n]:
            hg.hg_append_kv(runner.cache, layer, 1, k_new[layer], v_new[layer])
    q = wl.step_query(w, 0, "cuda")
    out = torch.full_like(q, float("nan"))
    hg.hg_decode_attention(runner.cache, 0, 3, q, out, SIGMA, runner.ws, runner.ws_bytes)
    for layer, n in enumerate(counts):
        for row in range(w.batch):
            ref = _row_reference(runner, layer, row, *kept[layer], q, news[:n])
            assert_close(bits16(out[layer, row:row + 1]), ref, "layer %d row %d" % (layer, row))


def test_more_layers_than_one_launch_holds():
    """70 layers in one call: launches of 64 and of 6 layers on one workspace, step after step."""
    w = wl.custom("deep", 70, 1, 8, 8, 8, 72, 8, wl.BASE_MINMAX, 2, 0, decode_steps=3, seed=19, protected=[(1, 0), (66, 3)])
    runner = CacheRunner(w)
    kept = runner.quantize_all(keep=True)
    news = []
    for step in range(3):
        k_new, v_new = wl.step_new_kv(w, step, "cuda")
        q = wl.step_query(w, step, "cuda")
        out = torch.full_like(q, float("nan"))
        runner.decode_step(step, q=q, k_new=k_new, v_new=v_new, out=out)
        news.append((k_new, v_new))
        for layer in (0, 1, 15, 16, 40, 63, 64, 66, 69):
            ref = _row_reference(runner, layer, 0, *kept[layer], q, news)
            assert_close(bits16(out[layer, :1]), ref, "step %d layer %d" % (step, layer))


@pytest.mark.parametrize("base,group", [(wl.BASE_MINMAX, 4), (wl.BASE_KIVI, 1)])
def test_layer_ranges_take_turns_on_one_workspace(base, group):
    """One layer, all layers, two layers, all layers on a workspace that was cleared once: the counters of the
    larger launches (2 KB) lie beyond those of a layer (384 bytes)."""
    w = wl.custom("turns", 6, 6, 16 * group, 16, 10, 96, 40, base, 2, 0, decode_steps=1, seed=21,
                  protected=[(0, 1), (4, 5)])
    runner = CacheRunner(w)
    kept = runner.quantize_all(keep=True)
    k_new, v_new = wl.step_new_kv(w, 0, "cuda")
    hg.hg_append_kv(runner.cache, 0, w.layers, k_new, v_new)
    q = wl.step_query(w, 0, "cuda")
    refs = {}
    for begin, count in ((0, 1), (0, 6), (3, 2), (0, 6), (5, 1), (1, 5), (0, 6)):
        out = torch.full_like(q[begin:begin + count], float("nan"))
        hg.hg_decode_attention(runner.cache, begin, count, q[begin:begin + count], out, SIGMA, runner.ws, runner.ws_bytes)
        for layer in range(begin, begin + count):
            for row in (0, 5):
                if (layer, row) not in refs:
                    refs[layer, row] = _row_reference(runner, layer, row, *kept[layer], q, [(k_new, v_new)])
                assert_close(bits16(out[layer - begin, row:row + 1]), refs[layer, row],
                             "layers %d+%d layer %d row %d" % (begin, count, layer, row))


def _decode_against_oracle(w, kept, steps, q_scale=1.0, v_max=1.0):
    """Append `steps` tokens in fused steps on a cache quantized from `kept`; the last step's outputs, every row.
    The tolerance is the suite's (2e-3 + 1e-2 |r| for values of order one) with its absolute part in units of
    the largest value: weights times value scales are FP16 products, so an output that cancels is off by up to
    2^-11 of the values that went into it, whatever its own size."""
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k for k, _ in kept], [v for _, v in kept])
    news = []
    for step in range(steps):
        k_new, v_new = wl.step_new_kv(w, step, "cuda")
        q = (wl.step_query(w, step, "cuda").float() * q_scale).bfloat16()
        out = runner.decode_step(step, q=q, k_new=k_new, v_new=v_new)
        news.append((k_new, v_new))
    for layer in range(w.layers):
        for row in range(w.batch):
            ref = _row_reference(runner, layer, row, *kept[layer], q, news)
            got = out[layer, row:row + 1].double().cpu().numpy()
            err = np.abs(got - ref)
            bad = ~(err <= 2e-3 * max(1.0, v_max) + 1e-2 * np.abs(ref))
            assert not bad.any(), (w.name, layer, row, int(bad.sum()), float(err.max()))


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("group", [1, 2])
def test_kivi_few_queries_per_head(group, bits, meta_bits):
    """One or two queries per KV head over KIVI-style codes: a single 32-token group (half a tile), an odd
    number of groups, and more than one tile per warp; quantized and keys-only heads."""
    for image, keys_only in ((33, 1), (100, 0), (1000, 1)):
        w = wl.custom("cols%d" % image, 1, 2, 4 * group, 4, 7, image, 37, wl.BASE_KIVI, bits, keys_only,
                      decode_steps=2, seed=3, protected=[(0, 2)], meta_bits=meta_bits)
        _decode_against_oracle(w, [wl.layer_kv(w, 0, "cuda")], 2)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("batch", [2, 24])
def test_kivi_grouped_queries_in_one_wave_and_more(batch, bits):
    """Four queries per KV head over KIVI-style codes in launches below and above four CTAs per SM (registers for
    three and for four CTAs)."""
    w = wl.custom("wave%d" % batch, 2, batch, 32, 8, 20, 150, 30, wl.BASE_KIVI, bits, 0, decode_steps=1, seed=16,
                  protected=[(0, 1)])
    _decode_against_oracle(w, [wl.layer_kv(w, layer, "cuda") for layer in range(2)], 1)


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("group", [3, 8, 12])
def test_kivi_groups_shared_by_two_warps(group, bits, meta_bits):
    """Three and more queries per KV head over KIVI-style codes: spans whose quarter ends in the middle of a
    32-token group (one to seven groups, and several chunks), so that its halves are two warps'."""
    for image in (32, 64, 96, 160, 224, 1120):
        w = wl.custom("halves%d" % image, 1, 2, 2 * group, 2, 7, image, 5, wl.BASE_KIVI, bits, 0, decode_steps=1, seed=23,
                      protected=[(0, 1)], residual=0, meta_bits=meta_bits)
        _decode_against_oracle(w, [wl.layer_kv(w, 0, "cuda")], 1)


@pytest.mark.parametrize("base,bits,group", [(wl.BASE_KIVI, 2, 1), (wl.BASE_KIVI, 3, 2), (wl.BASE_KIVI, 4, 1),
                                             (wl.BASE_MINMAX, 2, 4), (wl.BASE_MINMAX, 4, 12), (wl.BASE_AKVQ, 3, 7)])
def test_decode_scales_over_many_binades(base, bits, group):
    """Key and value scales that change by 2^16 between 32-token groups, grow along the sequence, vanish
    (constant groups) and meet zero and large queries: the power-of-two units of the FP16 operands."""
    w = wl.custom("binades", 1, 1, 2 * group, 2, 8, 640, 40, base, bits, 0, decode_steps=1, seed=9, protected=[])
    g = torch.Generator(device="cuda").manual_seed(4)
    e = torch.randint(-8, 9, (1, 2, w.seq_len // 32 + 1, 1), generator=g, device="cuda")
    e = e.sort(dim=2).values.repeat_interleave(32, 2)[:, :, :w.seq_len].float()
    k, v = wl.layer_kv(w, 0, "cuda")
    k = (k.float() * torch.exp2(-2 - e.abs())).bfloat16()
    v = (v.float() * torch.exp2(e)).bfloat16()
    k[:, :, 104:136] = 0.25  # a constant group: scale 0
    v[:, :, 200:232, 32:64] = -3.0
    for q_scale in (0.0, 1.0, 512.0):
        _decode_against_oracle(w, [(k, v)], 1, q_scale, float(v.abs().max()))


@pytest.mark.parametrize("base,bits,group", [(wl.BASE_KIVI, 2, 1), (wl.BASE_KIVI, 3, 2), (wl.BASE_KIVI, 4, 1),
                                             (wl.BASE_KIVI, 2, 4), (wl.BASE_MINMAX, 2, 4), (wl.BASE_MINMAX, 3, 12),
                                             (wl.BASE_AKVQ, 4, 7)])
@pytest.mark.parametrize("power", [-112, -80, 80, 112])
def test_keys_near_the_ends_of_the_range(power, base, bits, group):
    """Keys of 2^power, with a softmax scale that brings the scores back to order one: no intermediate of the
    scores may overflow, or lose bits as a subnormal, where the scores themselves do not."""
    w = wl.custom("range", 1, 1, 2 * group, 2, 8, 200, 40, base, bits, 0, decode_steps=1, seed=25, protected=[])
    k, v = wl.layer_kv(w, 0, "cuda")
    k = (k.float() * 2.0 ** power).bfloat16()
    sigma = SIGMA * 2.0 ** -power
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    q = wl.step_query(w, 0, "cuda")
    out = torch.empty_like(q)
    hg.hg_decode_attention(runner.cache, 0, 1, q, out, sigma, runner.ws, runner.ws_bytes)
    o = oracle_layer(runner, 0, bits16(k), bits16(v))
    ref = oracle.attention_layer(bits16(q[0]), o["k_att"], o["v_deq"].astype(np.float64), sigma)
    assert_close(bits16(out[0]), ref, "2^%d" % power)


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("base,bits,salient", [(wl.BASE_MINMAX, 3, 0), (wl.BASE_KIVI, 2, 0), (wl.BASE_KIVI, 3, 0),
                                               (wl.BASE_KIVI, 4, 0), (wl.BASE_AKVQ, 2, 0), (wl.BASE_AKVQ, 4, 30)])
@pytest.mark.parametrize("prefix,image,suffix", [(0, 1, 0), (3, 2, 1), (31, 33, 0), (1, 40, 64), (33, 257, 5)])
def test_dequantize_run_edges(prefix, image, suffix, base, bits, salient, meta_bits):
    """Eight-row runs that straddle the start, the image span's end and the last token, bit for bit."""
    w = wl.custom("runs", 2, 1, 4, 2, prefix, image, suffix, base, bits, int(image == 33), seed=2,
                  protected=[(0, 1)], residual=0, meta_bits=meta_bits, salient_permille=salient)
    _dequantize_bit_exact(w)


@pytest.mark.parametrize("bits,permille,image", [(2, 10, 63), (2, 500, 65), (2, 870, 129), (2, 880, 128), (3, 930, 200),
                                                 (4, 930, 200), (4, 970, 96), (2, 1000, 33)])
def test_salient_scores_beside_codes_or_rows(bits, permille, image):
    """The selection's scores wait in the head's value codes, or in its BF16 rows when the coded tokens are too
    few to hold them: both sides of the line, spans around the 64 tokens of a block; keys-only heads too."""
    w = wl.custom("scores", 2, 2, 8, 4, 5, image, 9, wl.BASE_AKVQ, bits, 1, decode_steps=1, seed=6,
                  protected=[(0, 1), (1, 2)], salient_permille=permille)
    _run_and_check(w)


@pytest.mark.parametrize("image", [511, 512, 513])
def test_salient_selection_in_one_or_two_launches(image):
    """Around the span length up to which the selection sums the key norms itself."""
    w = wl.custom("launches", 1, 2, 8, 4, 6, image, 9, wl.BASE_AKVQ, 4, 0, decode_steps=1, seed=8,
                  protected=[(0, 1)], salient_permille=20)
    _run_and_check(w)


@pytest.mark.parametrize("image", [11663, 11664, 11915, 11916])
def test_salient_spans_around_the_default_shared_memory(image):
    """Scores and bits of the span, with the selection's own arrays, around the 48 KB that a block may have
    without asking for more."""
    w = wl.custom("smem", 1, 1, 4, 2, 3, image, 9, wl.BASE_AKVQ, 4, 0, decode_steps=1, seed=9,
                  protected=[(0, 1)], salient_permille=20)
    _run_and_check(w)


@pytest.mark.parametrize("image", [97, 700])
@pytest.mark.parametrize("kind", ["one far above", "two sizes", "two values", "neighbours", "equal", "zero"])
def test_salient_selection_of_norms_in_few_digits(kind, image):
    """Keys whose squared norms differ in few bits, or in high and low ones at once (the selection starts at the
    highest bit in which two differ and ends at a digit that is taken whole).  Bit for bit."""
    w = wl.custom("digits", 1, 2, 4, 2, 5, image, 6, wl.BASE_AKVQ, 4, 0, seed=15, protected=[], residual=0,
                  salient_permille=100)
    g = torch.Generator(device="cuda").manual_seed(6)
    k = torch.randn(2, 2, w.seq_len, 128, generator=g, device="cuda")
    if kind == "one far above":
        k[:, :, 40] *= 1e8
    elif kind == "two sizes":
        k[:, :, ::3] *= 16.0
    elif kind == "two values":
        k = torch.where(torch.arange(w.seq_len, device="cuda")[:, None] % 7 == 0, 2.0, 1.0).expand_as(k)
    elif kind == "neighbours":  # 128 + small steps: only low bits differ
        k = torch.ones_like(k)
        k[..., 0] = 1.0 + torch.randint(0, 6, k.shape[:3], generator=g, device="cuda") * 2.0 ** -7
    else:
        k = torch.full_like(k, 0.0 if kind == "zero" else -1.5)
    k = k.bfloat16().contiguous()
    v = torch.randn(2, 2, w.seq_len, 128, generator=g, device="cuda").bfloat16()
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    torch.cuda.synchronize()
    check_arena_layer(runner, 0, bits16(k), bits16(v), oracle_layer(runner, 0, bits16(k), bits16(v)))


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("base", [wl.BASE_MINMAX, wl.BASE_KIVI, wl.BASE_AKVQ])
def test_two_bit_codes_by_comparison(base, meta_bits):
    """2-bit groups for the comparison rule and around what it leaves to the general one, bit for bit: one
    sign, boundaries at and next to zero and on BF16 values, signed zeros, constants, steps too small and too
    large, values many binades apart."""
    w = wl.custom("compare", 1, 1, 4, 2, 0, 32 * 14, 0, base, 2, 0, seed=12, protected=[], residual=0,
                  meta_bits=meta_bits)
    g = torch.Generator(device="cuda").manual_seed(3)
    r = torch.randn(14, 2, 2, 32, 128, generator=g, device="cuda")
    r[0] = r[0].abs() + 0.01
    r[1] = -r[1].abs() - 0.01
    r[2] = torch.where(r[2] > 0, 1.5, -1.5)                                   # middle boundary at zero
    r[3, ..., ::2], r[3, ..., 1::2] = -3.0, 3.0078125                         # ... and next to it
    r[4] = torch.randint(-6, 7, r[4].shape, generator=g, device="cuda") * 0.5  # quotients on half-integers
    r[5] = torch.where(r[5] > 0, 0.0, -0.0)
    r[6] = 0.375
    r[7] *= 1e-36
    r[8] *= 1e36
    r[9] *= torch.exp2(torch.randint(-30, 30, r[9].shape, generator=g, device="cuda").float())
    r[10] = torch.where(r[10].abs() < 1, r[10] * 1e-4, r[10])                 # many values around zero
    r[11] = r[11] * 0.01 + 100.0
    r[12] = r[12] * 0.01 - 100.0
    r[13, ..., :] = torch.linspace(-1.0, 2.0, 128, device="cuda")
    k = r[:, 0].permute(1, 0, 2, 3).reshape(1, 2, -1, 128).bfloat16().contiguous()
    v = r[:, 1].permute(1, 0, 2, 3).reshape(1, 2, -1, 128).bfloat16().contiguous()
    k, v = k.clone(), v.clone()
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    torch.cuda.synchronize()
    check_arena_layer(runner, 0, bits16(k), bits16(v), oracle_layer(runner, 0, bits16(k), bits16(v)))


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("base", [wl.BASE_MINMAX, wl.BASE_KIVI, wl.BASE_AKVQ])
def test_every_code_on_a_tie(base, bits, meta_bits):
    """Groups of half-integers from 0 to the top level (step 1): every element but the extremes is exactly on a
    tie, at every position of a chunk and of a key group, and each is coded again alone.  Bit for bit."""
    w = wl.custom("ties", 1, 2, 4, 2, 3, 96, 5, base, bits, 0, seed=14, protected=[], residual=0, meta_bits=meta_bits)
    g = torch.Generator(device="cuda").manual_seed(5)
    top = (1 << bits) - 1
    x = torch.randint(0, top, (2, 2, 2, w.seq_len, 128), generator=g, device="cuda") + 0.5
    tok, ch = torch.arange(w.seq_len, device="cuda")[:, None] - 3, torch.arange(128, device="cuda")
    x = torch.where((ch + tok) % 32 == 0, 0.0, x)        # one of each per 32 channels and per 32 tokens
    x = torch.where((ch + tok) % 32 == 17, float(top), x)
    x[..., 40:48] = torch.where(x[..., 40:48] % 1 == 0, x[..., 40:48], x[..., 40:48] + 0.125 * (tok % 2 == 0))
    x = x.clamp(max=float(top)).bfloat16()
    k, v = x[0].contiguous(), x[1].contiguous()
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    torch.cuda.synchronize()
    check_arena_layer(runner, 0, bits16(k), bits16(v), oracle_layer(runner, 0, bits16(k), bits16(v)))


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("base", [wl.BASE_MINMAX, wl.BASE_KIVI, wl.BASE_AKVQ])
def test_non_finite_elements_keep_to_themselves(base, bits, meta_bits):
    """A NaN or an infinity (at every position of a chunk, one per row and key group): the metadata and the
    codes of the group's other elements are the oracle's.  (The element's own code has no defined value; rotated
    keys have none to compare, since the rotation spreads it over the row.)"""
    w = wl.custom("nonfinite", 1, 1, 4, 2, 0, 128, 0, base, bits, 0, seed=18, protected=[], residual=0,
                  meta_bits=meta_bits)
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(2, 1, 2, 128, 128, generator=g, device="cuda")
    special = torch.zeros(128, 128, dtype=torch.bool, device="cuda")
    tok = torch.arange(128, device="cuda")
    # token t: channel (t * 9 + 1) % 128, never a group's first element (which starts the oracle's extremes)
    ch = (tok * 9 + 1) % 128
    keep = (ch % 32 != 0) & (tok % 32 != 0)
    special[tok[keep], ch[keep]] = True
    value = torch.where(tok % 2 == 0, float("nan"), float("inf"))
    x = torch.where(special, value[:, None], x).bfloat16()
    k, v = x[0].contiguous(), x[1].contiguous()
    if base == wl.BASE_AKVQ:
        k = torch.randn(k.shape, generator=g, device="cuda").bfloat16()
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    torch.cuda.synchronize()
    o = oracle_layer(runner, 0, bits16(k), bits16(v))
    arena = runner.arena.cpu().numpy()
    other = ~special.cpu().numpy()
    for h in range(2):
        r = hg.hg_cache_head_regions(runner.cache, 0, h)
        for off, moff, words, meta, name in ((r.kq, r.kqm, o["k_words"][0, h], o["k_meta"][0, h], "k"),
                                             (r.vq, r.vqm, o["v_words"][0, h], o["v_meta"][0, h], "v")):
            got = arena[off:off + words.nbytes].view(np.uint32)
            key_groups = name == "k" and base == wl.BASE_KIVI
            n = 32 if key_groups else 128  # codes of one packed run

            def codes(a):
                c = np.stack([oracle.unpack(row, n, bits) for row in a.reshape(-1, n * bits // 32)])
                return c.reshape(4, 128, 32).transpose(0, 2, 1).reshape(128, 128) if key_groups else c

            differ = codes(got) != codes(words)
            if name == "v" or base != wl.BASE_AKVQ:
                differ &= other
            assert not differ.any(), (name, h, np.argwhere(differ)[:4])
            m = arena[moff:moff + meta.size * (2 if meta_bits == 32 else 4)]
            want = meta.astype(np.float16) if meta_bits == 32 else meta
            assert np.array_equal(m.view(want.dtype), want), (name, h, "metadata")


@pytest.mark.parametrize("meta_bits", [64, 32])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_rotated_keys_with_one_channel_far_above_the_rest(bits, meta_bits):
    """Channel 0 up to a million times the others: every rotated value of a row is far from zero against the
    row's range, so the group minimum's subtraction shows whether the rotated values were rounded first.  Bit for
    bit."""
    w = wl.custom("onechannel", 1, 2, 4, 2, 3, 600, 5, wl.BASE_AKVQ, bits, 0, seed=17, protected=[], residual=0,
                  meta_bits=meta_bits)
    g = torch.Generator(device="cuda").manual_seed(8)
    k = torch.randn(2, 2, w.seq_len, 128, generator=g, device="cuda")
    v = torch.randn(2, 2, w.seq_len, 128, generator=g, device="cuda").bfloat16()
    k[..., 0] = torch.exp2(torch.rand(k.shape[:3], generator=g, device="cuda") * 14 + 6)
    k[:, 1, :, 0] *= -1
    k = k.bfloat16().contiguous()
    runner = CacheRunner(w)
    hg.hg_quantize_kv(runner.cache, 0, [k], [v])
    torch.cuda.synchronize()
    check_arena_layer(runner, 0, bits16(k), bits16(v), oracle_layer(runner, 0, bits16(k), bits16(v)))


@pytest.mark.parametrize("base,group", [(wl.BASE_MINMAX, 7), (wl.BASE_KIVI, 1), (wl.BASE_AKVQ, 12)])
def test_append_and_allocation_free_attention_back_to_back(base, group):
    """Tokens appended and attended layer by layer with nothing waiting in between (append, counter clear and
    decode overlap as programmatic dependent launches), against the oracle at the last token."""
    w = wl.custom("chain", 3, 2, 4 * group, 4, 20, 700, 40, base, 2, 0, decode_steps=8, seed=13,
                  protected=[(0, 1), (2, 3)])
    runner = CacheRunner(w)
    kept = runner.quantize_all(keep=True)
    news = [wl.step_new_kv(w, s, "cuda") for s in range(8)]
    qs = [wl.step_query(w, s, "cuda") for s in range(8)]
    outs = [torch.empty_like(q) for q in qs]
    torch.cuda.synchronize()
    for (k_new, v_new), q, out in zip(news, qs, outs):
        for layer in range(3):
            hg.hg_append_kv(runner.cache, layer, 1, k_new[layer], v_new[layer])
            hg.hg_decode_attention_noalloc(runner.cache, layer, 1, q[layer], out[layer], SIGMA)
    torch.cuda.synchronize()
    for step in (0, 7):
        for layer in range(3):
            ref = _row_reference(runner, layer, 1, *kept[layer], qs[step], news[:step + 1])
            assert_close(bits16(outs[step][layer, 1:2]), ref, "step %d layer %d" % (step, layer))


@pytest.mark.parametrize("base,salient", [(wl.BASE_MINMAX, 0), (wl.BASE_KIVI, 0), (wl.BASE_AKVQ, 20)])
def test_overlapping_launches_change_nothing(base, salient):
    """Prefills over the same arena, reconstructions, appends at a position used before and decode calls with
    nothing waiting in between (they overlap as programmatic dependent launches) give what the same calls give
    with a wait after each."""
    w = wl.custom("overlap", 2, 3, 8, 4, 10, 900, 30, base, 2, 1, decode_steps=2, seed=14, protected=[(0, 1), (1, 2)],
                  salient_permille=salient)
    prefills = [[wl.layer_kv(dataclasses.replace(w, seed=14 + i), l, "cuda") for l in range(2)] for i in range(3)]
    news = [wl.step_new_kv(dataclasses.replace(w, seed=20 + i), 0, "cuda") for i in range(3)]
    q = wl.step_query(w, 0, "cuda")

    def calls(wait):
        runner = CacheRunner(w)
        got = []
        for kv, (k_new, v_new) in zip(prefills, news):
            for l in range(2):
                hg.hg_quantize_kv(runner.cache, l, [kv[l][0]], [kv[l][1]])
                wait()
            for fused in (False, True):
                hg.hg_cache_reset_appended(runner.cache)
                out = torch.empty_like(q)
                if fused:
                    hg.hg_decode_step(runner.cache, 0, 2, q, v_new, k_new, out, SIGMA, runner.ws, runner.ws_bytes)
                else:
                    hg.hg_append_kv(runner.cache, 0, 2, k_new, v_new)
                    wait()
                    hg.hg_decode_attention_noalloc(runner.cache, 0, 2, q, out, SIGMA)
                wait()
                k_out = torch.empty(2, w.batch, w.kv_heads, w.seq_len + 1, 128, dtype=torch.bfloat16, device="cuda")
                v_out = torch.empty_like(k_out)
                hg.hg_dequantize_kv(runner.cache, 0, 2, k_out, v_out, False)
                wait()
                got += [out, k_out, v_out]
        torch.cuda.synchronize()
        return got

    for i, (a, b) in enumerate(zip(calls(lambda: None), calls(torch.cuda.synchronize))):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16)), i
