"""GPU parity of kvshot_draft_attn on an fp8 (e4m3) target cache (KVSHOT_TARGET_FP8).

The target K/V are e4m3 codes with power-of-two scales; the oracle decodes them
exactly (oracle/fp8.py) to the bf16 values the kernel must use and runs the
plain attention oracle on those, so the tolerances are the bf16 path's:
out max-abs <= 2e-2, rel-L2 <= 5e-3, lse max-abs <= 1e-3.  Unused cache rows
hold NaN codes and unused draft slots NaN.
"""
import numpy as np
import pytest
import torch

from oracle import fp8 as of8
from paper_2604_26412_gb300 import kvshot
from paper_2604_26412_gb300 import workloads as wl
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

CASES = [
    # lens, levels, tree, paged, page_size, hq, hkv, n_query
    ((128,), (1, 1, 1, 1), False, False, 16, 32, 8, 1),          # tiny chain, contiguous
    ((0,), (1, 1, 1), False, False, 16, 32, 8, 1),                # empty prefix
    ((1, 63, 64, 65), (1, 1), False, True, 16, 32, 8, 1),         # ragged around the tile size
    ((17, 130, 300), (4, 4), True, True, 8, 32, 8, 4),            # tree, 16 rows, P = 8
    ((4096, 1000), (8, 12, 12), True, True, 16, 32, 8, 12),       # 48 rows (tcgen05 when forced: spread rows)
    ((257, 513), (8, 12, 12), True, True, 64, 32, 8, 32),         # 128 rows, row blocks
    ((700,), (2, 3, 3), True, True, 128, 32, 8, 8),               # page larger than a tile
    ((333, 5), (3, 3), True, False, 16, 8, 8, 3),                 # G = 1
    ((65,), tuple([1] * 70), False, False, 16, 4, 4, 2),          # chain with N = 70 > one draft tile
    ((203, 64), tuple([1] * 40), False, False, 16, 32, 8, 32),    # 128 dense rows, contiguous l_cap % 8 != 0
    ((300, 200), (8, 12, 12, 12), True, True, 16, 32, 8, 40),     # 160 rows: two blocks
]


def _setup(case, seed):
    lens, levels, tree, paged, P, hq, hkv, nq = case
    spec = wl.Spec("fp8", len(lens), 1, list(lens), list(levels), tree, paged, page_size=P, hq=hq, hkv=hkv, seed=seed)
    inp = wl.make_inputs(spec, "cuda", seed=seed, tail_fill="nan")
    N = spec.n_nodes
    dk, dv = wl.random_draft_kv(spec, inp.n_max, N, "cuda", seed=seed + 1, tail=float("nan"))
    q = wl.random_queries(spec, nq, "cuda", seed=seed + 2)
    tk8, tv8 = wl.fp8_target(inp)
    hc = gh.HostCache(inp)
    hc.tk = of8.dequant_bf16_bits(tk8.cpu().numpy(), wl.FP8_K_EXP)
    hc.tv = of8.dequant_bf16_bits(tv8.cpu().numpy(), wl.FP8_V_EXP)
    return spec, inp, dk, dv, q, N, nq, tk8, tv8, hc


def _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, flags, num_ctas=0, k_exp=wl.FP8_K_EXP, v_exp=wl.FP8_V_EXP, scale=0.0):
    paged = inp.page_table is not None
    out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full(q.shape[:3], float("nan"), dtype=torch.float32, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    d = kvshot.make_desc(num_caches=spec.num_caches, num_seqs=spec.num_seqs, hq=spec.hq, hkv=spec.hkv, n_nodes=N,
                         n_query=Nq, n_max=inp.n_max, max_seq_len=spec.max_seq_len,
                         page_size=spec.page_size if paged else 0,
                         max_pages_per_seq=inp.page_table.shape[1] if paged else 0,
                         num_pages=inp.num_pages if paged else 0, l_cap=inp.l_cap, tree=spec.tree,
                         flags=flags | kvshot.KVSHOT_TARGET_FP8, num_ctas=num_ctas, err_flag=err, scale=scale,
                         k_scale_exp=k_exp, v_scale_exp=v_exp)
    ws = torch.empty(kvshot.workspace_size(d), dtype=torch.uint8, device="cuda")
    d.workspace, d.workspace_bytes = ws.data_ptr(), ws.numel()
    kvshot.draft_attn(d, q, tk8, tv8, inp.page_table, inp.seq_lens, dk, dv, inp.tree_parent[:, :N].contiguous(),
                      out, lse)
    torch.cuda.synchronize()
    assert int(err.item()) == 0, f"device error {int(err.item())}"
    return out, lse


@pytest.mark.parametrize("case", CASES, ids=[f"c{i}" for i in range(len(CASES))])
def test_fp8_target_matches_oracle(case):
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=3 + len(case[0]) + sum(case[1]))
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    rows = case[5] // case[6] * case[7]
    for flags in (0, kvshot.KVSHOT_FORCE_MMA) + ((kvshot.KVSHOT_FORCE_TC,) if rows <= 128 else ()):
        for num_ctas in (0, 1, 7):
            out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, flags, num_ctas)
            gh.compare(out, lse, ref_out, ref_lse, f"fp8 {case} flags={flags} ctas={num_ctas}")


@pytest.mark.parametrize("nq", [12, 32])
def test_fp8_tcgen05_matches_oracle_at_48_and_128_rows(nq):
    # The tcgen05 kernel decoding fp8 tiles: 48 stacked rows (spread) and 128 (dense), paged P = 16.
    case = ((3000, 517, 64), (8, 12, 12), True, True, 16, 32, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=nq)
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    for num_ctas in (0, 3, 152):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, kvshot.KVSHOT_FORCE_TC, num_ctas)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 tcgen05 nq={nq} ctas={num_ctas}")


# The m16n8k16 kernel's row paddings (8, 16, 32, 48, 64 and a second 64-row block) at prefix lengths around its
# 128-key tiles and 32-key chunks, and pages that tile 128 keys in every way (192: a tile spans two pages).
@pytest.mark.parametrize("nq,hq,hkv", [(1, 32, 8), (2, 32, 8), (3, 15, 5), (5, 32, 8), (8, 32, 8), (11, 32, 8),
                                       (15, 32, 8), (17, 32, 8)])
@pytest.mark.parametrize("paged,page", [(False, 16), (True, 8), (True, 192), (True, 256)])
def test_fp8_m16n8k16_rows_tiles_and_pages(nq, hq, hkv, paged, page):
    case = ((127, 128, 129, 31, 33, 0, 385), (17,), True, paged, page, hq, hkv, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=100 + nq + page)
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    for num_ctas in (0, 5):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, kvshot.KVSHOT_FORCE_MMA, num_ctas)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 mma nq={nq} {hq}/{hkv} page={page if paged else 0} ctas={num_ctas}")


# More than 128 rows: blocks of up to 128 rows on the tcgen05 kernel (2 x 80, 2 x 128, 2 x 68 rows
# with an idle node, 3 x 88, 2 x 96 rows of G = 32).
@pytest.mark.parametrize("nq,hq,hkv", [(40, 32, 8), (64, 32, 8), (33, 32, 8), (33, 64, 8), (6, 64, 2)])
def test_fp8_stacks_of_more_than_128_rows(nq, hq, hkv):
    case = ((700, 65, 0), (8, 12, 12, 12, 12, 8), True, True, 16, hq, hkv, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=200 + nq)
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    for num_ctas in (0, 5):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, 0, num_ctas)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 blocks nq={nq} {hq}/{hkv} ctas={num_ctas}")


@pytest.mark.parametrize("nq", [1, 4, 12, 20])
def test_fp8_one_cache_cut_into_pieces(nq):
    case = ((3001,), (8, 12), True, True, 16, 32, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=300 + nq)
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    for flags in (0, kvshot.KVSHOT_FORCE_MMA, kvshot.KVSHOT_FORCE_TC):
        for num_ctas in (0, 8, 24, 61, 152):
            out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, flags, num_ctas)
            gh.compare(out, lse, ref_out, ref_lse, f"fp8 one cache nq={nq} flags={flags} ctas={num_ctas}")


# Rows of very different magnitude, of zeros, with one large element, and full blocks of 1 to 64 rows, in one and in
# many pieces.
@pytest.mark.parametrize("nq,hq,hkv", [(1, 8, 8), (1, 32, 8), (5, 32, 8), (7, 16, 8), (16, 32, 8), (2, 64, 2)])
def test_fp8_split_q_rows(nq, hq, hkv):
    case = ((200, 63, 129, 0, 65), (8, 12), True, True, 16, hq, hkv, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=400 + nq)
    g = torch.Generator(device="cuda").manual_seed(nq)
    scale = 2.0 ** torch.randint(-9, 5, q.shape[:3], generator=g, device="cuda").float()
    q = (q.float() * scale[..., None]).to(torch.bfloat16)
    q[0, 0, 0] = 0
    q[1, :, 1, 7] = 3.0
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq)
    for num_ctas in (0, 1, 7):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, kvshot.KVSHOT_FORCE_TC, num_ctas)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 split q nq={nq} {hq}/{hkv} ctas={num_ctas}")


# One channel of q is 2^drop times the others and meets zero keys: the others alone make the scores (of a few units).
# lse: the codes are exact, and q where f16 holds it (2^-17 and more; below it errs by up to 2^-25), which leaves the fp32
# sums of 128 products of up to ~4 and of the exponentials: 128 * 4 * 2^-24 = 3e-5, and 1e-5 for exponent and logarithm.
@pytest.mark.parametrize("drop", [4, 8, 9, 10, 11, 13, 15])
@pytest.mark.parametrize("nq", [5, 12, 16])
def test_fp8_small_elements_of_q_beside_a_dominant_one(drop, nq):
    case = ((5, 63, 130, 1), (12, 8), True, True, 16, 32, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=700 + nq)
    q = (q.float() * 2.0 ** -drop * 64).to(torch.bfloat16)
    q[..., 5] = 64.0
    tk8[..., 5] = 0
    dk[..., 5] = 0
    hc.tk = of8.dequant_bf16_bits(tk8.cpu().numpy(), wl.FP8_K_EXP)
    scale = 2.0 ** (drop - 6)  # q as drawn gives scores of about 1
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq, scale=scale)
    inexact = int((q.float().abs() < 2.0 ** -17).sum(-1).max())  # elements of a row, times |k| < 5
    bound = 4e-5 + inexact * 2.0 ** -25 * 5 * scale
    for flags in (kvshot.KVSHOT_FORCE_TC, kvshot.KVSHOT_FORCE_MMA):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, flags, 5, scale=scale)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 dominant channel drop={drop} nq={nq} flags={flags}")
        assert np.abs(lse.cpu().numpy() - ref_lse).max() <= bound


# The whole range of value scales, on pieces that end in the prefix, in the draft and on either side of its first tile.
# Draft values of magnitude 1 (f16 holds them), and none, which leaves the prefix alone however small its scale; out is
# compared in units of its largest part.
@pytest.mark.parametrize("v_exp", [-64, -30, -16, -8, -7, -5, -4, 0, 4, 5, 8, 9, 15, 17, 30, 64])
@pytest.mark.parametrize("nq,flags", [(1, 0), (4, 0), (12, 0), (32, 0), (12, kvshot.KVSHOT_FORCE_MMA), (40, 0)])
def test_fp8_value_scales(v_exp, nq, flags):
    case = ((200, 63, 128, 0, 700), (20, 20), True, True, 16, 32, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=800 + nq)
    hc.tv = of8.dequant_bf16_bits(tv8.cpu().numpy(), v_exp)
    unit = 2.0 ** (v_exp - wl.FP8_V_EXP)
    for dvs, top in ((dv, max(1.0, unit)), (torch.where(dv.isnan(), dv, 0), unit)):
        ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dvs, N, Nq)
        for num_ctas in (0, 1, 7, 150):
            out, lse = _run(spec, inp, tk8, tv8, dk, dvs, q, N, Nq, flags, num_ctas, v_exp=v_exp)
            gh.compare(out.float() / top, lse, ref_out / top, ref_lse, f"fp8 v_exp={v_exp} nq={nq} ctas={num_ctas}")


# A chain of several draft tiles behind the prefix.
@pytest.mark.parametrize("v_exp", [-20, 20])
@pytest.mark.parametrize("nq,flags", [(2, 0), (16, 0), (12, kvshot.KVSHOT_FORCE_MMA), (16, kvshot.KVSHOT_FORCE_TC)])
def test_fp8_value_scale_with_several_draft_tiles(nq, flags, v_exp):
    case = ((200, 63, 0), tuple([1] * 200), False, True, 16, 16, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=850 + nq)
    hc.tv = of8.dequant_bf16_bits(tv8.cpu().numpy(), v_exp)
    draft = 2.0 ** (v_exp // 2)
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv * draft, N, Nq)
    top = max(draft, 2.0 ** (v_exp - wl.FP8_V_EXP))
    for num_ctas in (0, 1, 5, 30):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv * draft, q, N, Nq, flags, num_ctas, v_exp=v_exp)
        gh.compare(out.float() / top, lse, ref_out / top, ref_lse, f"fp8 chain v_exp={v_exp} nq={nq} ctas={num_ctas}")


# Rows of zeros and of tiny values where the score scale is smallest: masked keys of a part-filled tile stay masked.
@pytest.mark.parametrize("k_exp,scale", [(-22, 0.0), (-30, 0.0), (-64, 0.0), (-64, 2.0 ** -90), (-3, 2.0 ** -140)])
@pytest.mark.parametrize("nq,flags", [(1, 0), (5, 0), (5, kvshot.KVSHOT_FORCE_MMA), (20, 0)])
def test_fp8_zero_rows_at_small_key_scales(k_exp, scale, nq, flags):
    case = ((200, 63, 130), (12, 8), True, True, 16, 32, 8, nq)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=500 + nq)
    hc.tk = of8.dequant_bf16_bits(tk8.cpu().numpy(), k_exp)
    q[:, 0, 0] = 0
    q[:, 0, 1] = 2.0 ** -100
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq, scale=scale)
    for num_ctas in (0, 5):
        out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, flags, num_ctas, k_exp=k_exp, scale=scale)
        gh.compare(out, lse, ref_out, ref_lse, f"fp8 zero rows nq={nq} k_exp={k_exp} flags={flags} ctas={num_ctas}")


# The largest number of caches at every row padding of both kernels (G = 5: the m16n8k16 kernel at all of them).
@pytest.mark.parametrize("nq,hq,hkv", [(1, 5, 1), (2, 5, 1), (4, 5, 1), (6, 5, 1), (8, 5, 1), (12, 5, 1), (13, 5, 1),
                                       (6, 4, 1), (32, 4, 1), (33, 4, 1)])
def test_fp8_largest_number_of_caches(nq, hq, hkv):
    lens = [(37 * c) % 90 for c in range(1024)]
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup((lens, (nq + 2,), True, True, 16, hq, hkv, nq), seed=600 + nq)
    out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, 0)
    some = [0, 1, 500, 977, 978, 1022, 1023]
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq, caches=some)
    gh.compare(out[some], lse[some], ref_out, ref_lse, f"fp8 1024 caches nq={nq} {hq}/{hkv}")


# 256 rows over as many units as put 128-row blocks (912 + 152 of them) past the library's own scratch: 64-row blocks, which
# fit it, run there, with a workspace and with that scratch; 53 caches keep the 128-row blocks.
@pytest.mark.parametrize("caches", [53, 57])
def test_fp8_blocks_at_the_limit_of_the_static_scratch(caches):
    case = ([(29 * c) % 140 for c in range(caches)], (8, 12, 12, 12, 12, 8), True, True, 16, 32, 8, 64)
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(case, seed=caches)
    some = [0, 1, 30, caches - 1]
    ref_out, ref_lse = gh.oracle_attn(hc, q, dk, dv, N, Nq, caches=some)
    out, lse = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, 0)
    gh.compare(out[some], lse[some], ref_out, ref_lse, f"fp8 {caches} caches")
    d = kvshot.make_desc(num_caches=caches, num_seqs=caches, hq=32, hkv=8, n_nodes=N, n_query=Nq, n_max=inp.n_max,
                         max_seq_len=spec.max_seq_len, page_size=16, max_pages_per_seq=inp.page_table.shape[1],
                         num_pages=inp.num_pages, tree=True, flags=kvshot.KVSHOT_TARGET_FP8,
                         k_scale_exp=wl.FP8_K_EXP, v_scale_exp=wl.FP8_V_EXP)
    assert kvshot.workspace_size(d) <= 64 << 20
    assert kvshot.draft_attn_static_status(d, q, tk8, tv8, inp.page_table, inp.seq_lens, dk, dv, inp.tree_parent, out,
                                           lse) == kvshot.KVSHOT_OK
    torch.cuda.synchronize()
    gh.compare(out[some], lse[some], ref_out, ref_lse, f"fp8 {caches} caches, static scratch")


def test_fp8_is_deterministic_and_differs_from_bf16_only_by_quantisation():
    spec, inp, dk, dv, q, N, Nq, tk8, tv8, hc = _setup(((2000, 900), (4, 4), True, True, 16, 32, 8, 4), seed=21)
    a = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, 0)
    b = _run(spec, inp, tk8, tv8, dk, dv, q, N, Nq, 0)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    # the same call on the bf16 cache the codes were made from: close, but not equal (quantisation)
    hb = gh.HostCache(inp)
    ref_bf16, _ = gh.oracle_attn(hb, q, dk, dv, N, Nq)
    o = a[0].float().cpu().numpy().astype(np.float64)
    rel = np.linalg.norm(o - ref_bf16) / np.linalg.norm(ref_bf16)
    assert 1e-3 < rel < 0.1, rel
