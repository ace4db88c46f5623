"""Passes over many rows (prefill of more than 64 positions, validate calls of more than 64 rows): logits
against the oracle within the bf16 bar, at the edges of the row tiles, for both tile forms (one CTA, CTA
pair), whole and split K ranges, all attention forms and head sizes."""
import ctypes as C

import numpy as np
import pytest
import torch
from scipy.special import erfc

from oracle import stairs_oracle as so
from paper_2407_19947_b200 import workloads as wl
from tests import gpu_util as gu
from tests.test_gpu_parity import _stairs, small_a, small_b, sources

pytestmark = pytest.mark.gpu

SHAPES = {"gqa_hd16": small_b(8, 2, 16, d=128, f=192), "gqa_hd48": small_b(8, 4, 48, d=192, f=320), "gqa_hd64": small_b(8, 2, 64), "mha_hd80": small_b(4, 4, 80, d=320, f=640), "mqa_hd128": small_b(4, 1, 128, d=512, f=832),
          "hd96": small_b(4, 2, 96, d=384, f=448), "family_a": small_a()}


@pytest.mark.parametrize("cg,split", [(1, 1), (1, 4), (2, 0), (0, 0)], ids=["cta", "cta_split4", "pair", "planned"])
@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_long_prefill_matches_oracle(shape, cg, split):
    st = _stairs()
    tsrc, _ = sources(shape)
    tgt, _ = gu.oracle_pair(tsrc)
    eng = st.Stairs(tsrc, None, max_requests=1, max_seq_len=400, k_max=2, kv_page_tokens=16)
    eng.debug_tune(4, cg)
    eng.debug_tune(5, split)
    for n in (66, 129, 258, 333):        # 65 positions, one whole row tile, one whole pair of tiles + 1, ragged
        prompt = list(wl.zipf_tokens(n, shape.vocab, n))
        eng.prefill(0, prompt)
        tt, al, logits = eng.validate([0], [0], None, want_logits=True)
        eng.sync()
        ref = np.stack([so.forward_logits(tgt, prompt)])
        gu.check_rows_against_oracle(logits.cpu().numpy(), tt.cpu().numpy()[0], ref, gu.LOGIT_TOL_BF16)
    eng.close()


@pytest.mark.parametrize("k", [4, 17, 40])
@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_calls_of_more_than_64_rows_match_oracle(shape, k):
    # 75, 90 and 123 rows; 5 to 164 queries per kv head: every way the attention splits its warps, and
    # contexts short and long enough to be cut over several CTAs
    st = _stairs()
    tsrc, _ = sources(shape)
    tgt, _ = gu.oracle_pair(tsrc)
    n_req = {4: 15, 17: 5, 40: 3}[k]
    lens = [300 - 19 * i if i < 5 else 3 + 4 * i for i in range(n_req)]
    eng = st.Stairs(tsrc, None, max_requests=n_req, max_seq_len=400, k_max=k, kv_page_tokens=32)
    prompts = [list(wl.zipf_tokens(n, shape.vocab, 60 + i)) for i, n in enumerate(lens)]
    for i, p in enumerate(prompts):
        eng.prefill(i, p)
    drafts = np.random.default_rng(k).integers(0, shape.vocab, size=(n_req, k)).astype(np.int32)
    ks = [k] * n_req
    tt, al, logits = eng.validate(list(range(n_req)), ks, torch.from_numpy(drafts).cuda(), want_logits=True)
    eng.sync()
    logits, tt, al = logits.cpu().numpy(), tt.cpu().numpy(), al.cpu().numpy()
    for i in range(n_req):
        assert int(al[i]) == gu.first_mismatch(drafts[i], tt[i])
        if i in (0, n_req - 1):
            ref, _ = gu.oracle_stair_logits(tgt, prompts[i], drafts[i])
            gu.check_rows_against_oracle(logits[i * (k + 1):(i + 1) * (k + 1)], tt[i], ref, gu.LOGIT_TOL_BF16)
    eng.close()


def test_prefill_in_several_chunks_matches_one_chunk():
    st = _stairs()
    shape = small_b(8, 2, 64)
    tsrc, _ = sources(shape)
    prompt = list(wl.zipf_tokens(331, shape.vocab, 9))
    got = []
    for chunk in (0, 100):
        eng = st.Stairs(tsrc, None, max_requests=1, max_seq_len=400, k_max=2, kv_page_tokens=64, prefill_chunk=chunk)
        eng.prefill(0, prompt)
        _, _, lg = eng.validate([0], [0], None, want_logits=True)
        eng.sync()
        got.append(lg.cpu())
        eng.close()
    assert float((got[0] - got[1]).abs().max()) < 5e-3


@pytest.mark.parametrize("page", [32, 64, 128])
@pytest.mark.parametrize("name", ["gqa_hd64", "mqa_hd128", "family_a"])
def test_prefill_attention_over_many_chunks_matches_oracle(name, page):
    # several K/V chunks and query blocks, a second pass over cached positions, every page size's copies
    st = _stairs()
    shape = SHAPES[name].replace(max_pos=1024)
    tsrc, _ = sources(shape)
    tgt, _ = gu.oracle_pair(tsrc)
    eng = st.Stairs(tsrc, None, max_requests=1, max_seq_len=720, k_max=2, kv_page_tokens=page, prefill_chunk=400)
    prompt = list(wl.zipf_tokens(701, shape.vocab, page))
    eng.prefill(0, prompt)
    tt, _, logits = eng.validate([0], [0], None, want_logits=True)
    eng.sync()
    ref = np.stack([so.forward_logits(tgt, prompt)])
    gu.check_rows_against_oracle(logits.cpu().numpy(), tt.cpu().numpy()[0], ref, gu.LOGIT_TOL_BF16)
    eng.close()


def test_contexts_of_two_threads_with_different_head_sizes():
    # both head sizes run on one kernel, with different amounts of shared memory
    import threading
    st = _stairs()
    errors = []

    def work(hd, d):
        try:
            shape = small_b(4, 2, hd, layers=8, d=d, f=448)
            tsrc, _ = sources(shape)
            prompt = list(wl.zipf_tokens(131, shape.vocab, hd))
            eng = st.Stairs(tsrc, None, max_requests=1, max_seq_len=200, k_max=2, kv_page_tokens=16, stream=torch.cuda.Stream())
            want = None
            start.wait(60)
            for _ in range(400):
                eng.prefill(0, prompt)
                if want is None:
                    want = eng.validate([0], [0], None, want_logits=True)     # (kept whole: the streams differ from torch's)
            got = eng.validate([0], [0], None, want_logits=True)
            eng.sync()
            assert torch.equal(got[2], want[2])
            eng.close()
        except Exception as e:
            errors.append(e)

    start = threading.Barrier(2)
    threads = [threading.Thread(target=work, args=a) for a in ((96, 384), (112, 448))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


class _OneInputPerFeature(wl.WeightSource):
    """Attention adds nothing to the residual stream; every MLP feature sees one element of it, so its value is known to a few
    roundings."""

    def _draw_numpy(self, layer, name):
        a = super()._draw_numpy(layer, name)
        if name == "wo":
            a[:] = 0.0
        elif name == "w_gate_or_fc1":
            f = np.arange(a.shape[0])
            a[:] = 0.0
            a[f, f % a.shape[1]] = np.linspace(-3.5, 3.5, a.shape[0])
        return a


def test_gelu_of_many_row_calls_matches_64_bits():
    # the MLP activation itself, as stored (bf16 hi + lo: 2^-17), for arguments of both signs and all sizes that occur: the exact
    # GELU by erfc, which keeps its relative precision where 1 + erf cancels
    st = _stairs()
    shape = small_a(layers=1, f=1024)
    src = _OneInputPerFeature(shape, 11, "numpy", norm_jitter=0.1, std=0.03)
    eng = st.Stairs(src, None, max_requests=14, max_seq_len=32, k_max=4, kv_page_tokens=16)
    prompts = [list(wl.zipf_tokens(3 + i, shape.vocab, i)) for i in range(14)]
    for i, p in enumerate(prompts):
        eng.prefill(i, p)
    drafts = np.random.default_rng(2).integers(0, shape.vocab, size=(14, 4)).astype(np.int32)
    eng.validate(list(range(14)), [4] * 14, torch.from_numpy(drafts).cuda())          # 70 rows
    ptr, nbytes = C.c_void_p(), C.c_size_t()
    eng._ck(eng.lib.stairs_debug_buffer(eng.h, 4, C.byref(ptr), C.byref(nbytes)))
    rows = nbytes.value // (4 * shape.d_ff)
    got = eng.debug_buffer(4, torch.bfloat16, rows * shape.d_ff * 2).view(2, rows, shape.d_ff)[:, :70].double().sum(0).cpu().numpy()
    eng.close()
    w = lambda layer, name: so.widen(src.host_array(layer, name)).astype(np.float64)
    tok = np.concatenate([[p[-1], *d] for p, d in zip(prompts, drafts)])
    pos = np.concatenate([len(p) - 1 + np.arange(5) for p in prompts])
    x = w(-1, "tok_emb")[tok] + w(-1, "pos_emb")[pos]
    mean = x.mean(1, keepdims=True)
    xc = (x - mean) / np.sqrt(((x - mean) ** 2).mean(1, keepdims=True) + shape.norm_eps)
    h = xc * w(0, "norm2_w")
    v = h @ w(0, "w_gate_or_fc1").T + (w(0, "norm2_b") @ w(0, "w_gate_or_fc1").T)
    want = 0.5 * v * erfc(-v / np.sqrt(2))
    assert v.min() < -8 and v.max() > 8
    # the argument: the operand's hi + lo (2^-17), 1/std, mean and products (ten roundings of 2^-24), all relative to its terms; the
    # function: 8e-6 at most; the result: 2^-17.  d gelu / dv is at most (|v| + 1) |gelu / v| + 1 where v < 0, 1.13 elsewhere.
    term = np.abs(h) @ np.abs(w(0, "w_gate_or_fc1")).T + np.abs(v) + np.abs(mean / x.std(1, keepdims=True)) * np.abs(w(0, "w_gate_or_fc1") @ w(0, "norm2_w"))
    slope = np.abs(0.5 * erfc(-v / np.sqrt(2)) + v * np.exp(-v * v / 2) / np.sqrt(2 * np.pi))
    bound = np.abs(want) * (2.0 ** -17 + 8e-6) + 1.05 * slope * term * (2.0 ** -17 + 10 * 2.0 ** -24)
    seen = np.abs(want) > 1e-30                                      # (below, the lo part leaves bf16's range)
    assert np.all(np.abs(got - want)[seen] <= bound[seen])
    assert np.count_nonzero(seen & (v < -5)) > 100


def test_profile_times_every_gemm_of_a_many_row_call():
    st = _stairs()
    shape = small_b(8, 2, 64)
    tsrc, _ = sources(shape)
    eng = st.Stairs(tsrc, None, max_requests=2, max_seq_len=128, k_max=39, kv_page_tokens=16)
    for i in range(2):
        eng.prefill(i, list(wl.zipf_tokens(20 + i, shape.vocab, i)))
    drafts = torch.zeros((2, 39), dtype=torch.int32, device="cuda")
    eng.profile(True)
    eng.validate([0, 1], [39, 39], drafts)
    gemm_ms, launches, call_ms = eng.profile_read()
    eng.profile(False)
    assert launches == 4 * shape.n_layers + 1 and 0 < gemm_ms < call_ms     # QKV, O, gate + up, down; the LM head
    eng.close()


def test_prefill_pass_of_more_tiles_than_split_counters():
    # 72000 rows x 61440 gate and up columns in one pass: 67680 tiles (whole ones need no counter); against passes of 2048 rows
    st = _stairs()
    shape = small_b(1, 1, 64, layers=2, d=64, f=30720, v=512)
    tsrc, _ = sources(shape)
    prompt = list(wl.zipf_tokens(72001, shape.vocab, 3))
    got = []
    for chunk in (72000, 0):
        eng = st.Stairs(tsrc, None, max_requests=1, max_seq_len=72008, k_max=2, kv_page_tokens=128, prefill_chunk=chunk)
        eng.prefill(0, prompt)
        _, _, lg = eng.validate([0], [0], None, want_logits=True)
        eng.sync()
        got.append(lg.cpu())
        eng.close()
        del eng
    assert torch.isfinite(got[0]).all() and float((got[0] - got[1]).abs().max()) < 5e-3


# Distances between the two bf16 paths (2-norm over the logits' 2-norm).  Both take operands as bf16 hi + lo (2^-17) and K and V as
# fp16, so they differ by the order of fp32 sums and by what that flips in an operand's last bit: 1.5e-5 to 8.7e-5 measured.  The same
# passes emulated in numpy with the lo part of just one operand (norm 1, attention, norm 2, MLP or final norm) left out are off by at
# least 4.7e-4 where the rows themselves went through them, and by 1.6e-4 where only the cached positions did.
ROWS_BAR, PREFIX_BAR = 2.5e-4, 1.2e-4


def _distance(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_many_row_passes_agree_with_small_ones(shape):
    st = _stairs()
    tsrc, _ = sources(shape)
    eng = st.Stairs(tsrc, None, max_requests=26, max_seq_len=400, k_max=4, kv_page_tokens=16)
    # 65 positions prefilled in one many-row pass, against 64 by the persistent kernel and the last as a row of the call
    prompt = list(wl.zipf_tokens(66, shape.vocab, 5))
    eng.prefill(0, prompt)
    eng.prefill(1, prompt[:65])
    _, _, a = eng.validate([0], [0], None, want_logits=True)
    nxt = torch.tensor([[prompt[65], 0, 0, 0]], dtype=torch.int32, device="cuda")
    _, _, b = eng.validate([1], [1], nxt, want_logits=True)
    eng.sync()
    assert _distance(a[0], b[1]) < PREFIX_BAR
    # 65 rows (one tile) and 130 (two, or a pair) against calls of 5 rows
    for i in range(26):
        eng.prefill(i, list(wl.zipf_tokens(20 + 3 * i, shape.vocab, 60 + i))[:64])
    drafts = torch.from_numpy(np.random.default_rng(1).integers(0, shape.vocab, size=(26, 4)).astype(np.int32)).cuda()
    alone = torch.cat([eng.validate([i], [4], drafts[i:i + 1].contiguous(), want_logits=True)[2] for i in range(26)])
    for cg, n in ((0, 13), (1, 26), (2, 26)):
        eng.debug_tune(4, cg)
        _, _, many = eng.validate(list(range(n)), [4] * n, drafts[:n].contiguous(), want_logits=True)
        eng.sync()
        assert _distance(many, alone[: 5 * n]) < ROWS_BAR
    eng.close()


@pytest.mark.parametrize("pairs", [1, 3])
def test_expired_wait_of_a_call_of_one_row_tile_is_reported(pairs):
    # Of the kernels of a call of 70 rows only its GEMMs have bounded waits.  With a bound of about a microsecond they run out: every
    # launch must end by itself, the next sync report STAIRS_ETIMEOUT (5), and the same call with the default bound work afterwards.
    st = _stairs()
    shape = small_b()
    tsrc, _ = sources(shape)
    drafts = torch.from_numpy(np.random.default_rng(1).integers(0, shape.vocab, size=(14, 4)).astype(np.int32)).cuda()
    eng = st.Stairs(tsrc, None, max_requests=14, max_seq_len=64, k_max=4, kv_page_tokens=16)
    eng.debug_tune(6, pairs)
    for i in range(14):
        eng.prefill(i, list(wl.zipf_tokens(20 + i, shape.vocab, i)))
    alone = torch.cat([eng.validate([i], [4], drafts[i:i + 1].contiguous(), want_logits=True)[2] for i in range(14)])
    eng.sync()
    eng.debug_tune(8, 2000)
    with pytest.raises(st.StairsError) as e:
        eng.validate(list(range(14)), [4] * 14, drafts)
        eng.sync()
    assert e.value.code == 5
    eng.debug_tune(8, 0)
    _, _, many = eng.validate(list(range(14)), [4] * 14, drafts, want_logits=True)
    eng.sync()
    assert _distance(many, alone) < ROWS_BAR
    eng.close()


@pytest.mark.parametrize("pairs", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_calls_of_one_row_tile_at_every_cluster_size(shape, pairs):
    # the GEMMs of 65 to 128 rows: rows that end before, at and behind a 16-row box, shares of the rows that are no multiples of
    # anything, K cut over one to four pairs of CTAs, tiles of whole heads, an odd number of tiles
    st = _stairs()
    tsrc, _ = sources(shape)
    eng = st.Stairs(tsrc, None, max_requests=26, max_seq_len=128, k_max=4, kv_page_tokens=16)
    for i in range(26):
        eng.prefill(i, list(wl.zipf_tokens(20 + 3 * (i % 15), shape.vocab, 60 + i)))
    drafts = torch.from_numpy(np.random.default_rng(1).integers(0, shape.vocab, size=(26, 4)).astype(np.int32)).cuda()
    alone = [eng.validate([i], [4], drafts[i:i + 1].contiguous(), want_logits=True)[2] for i in range(26)]
    eng.debug_tune(6, pairs)
    for rows in (65, 81, 96, 97, 127, 128):
        ks = [4] * (rows // 5) + ([rows % 5 - 1] if rows % 5 else [])
        n = len(ks)
        _, _, many = eng.validate(list(range(n)), ks, drafts[:n].contiguous(), want_logits=True)
        eng.sync()
        assert _distance(many, torch.cat([alone[i][: k + 1] for i, k in enumerate(ks)])) < ROWS_BAR
    eng.close()
