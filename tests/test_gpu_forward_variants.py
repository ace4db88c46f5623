"""The compiled variants of the whole-pass kernel (head size, model family, attention path, at most 16 rows or more) against
the oracle at the edges: 16 and 17 rows, positions around a 64-position chunk, smallest and largest page slices, and bitwise
the same rows from a call on either side of the 16-row line."""
import numpy as np
import pytest
import torch

from paper_2407_19947_b200 import workloads as wl
from tests import gpu_util as gu
from tests.test_gpu_parity import _stairs, small_a, small_b, sources

pytestmark = pytest.mark.gpu

SHAPES = {"family_a": small_a(), "hd48": small_b(4, 2, 48, d=192, f=320), "hd64": small_b(8, 2, 64), "hd80": small_b(4, 4, 80, d=320, f=640),
          "hd96": small_b(4, 2, 96, d=384, f=448), "hd128": small_b(4, 1, 128, d=512, f=832)}


@pytest.mark.parametrize("page", [16, 128])
@pytest.mark.parametrize("attention", [0, 2], ids=["register", "tcgen05"])
@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_variant_matches_oracle_and_ignores_the_row_count(shape, attention, page):
    st = _stairs()
    tsrc, _ = sources(shape)
    tgt, _ = gu.oracle_pair(tsrc)
    lens = [63, 65, 300]
    eng = st.Stairs(tsrc, None, max_requests=len(lens), max_seq_len=400, k_max=16, kv_page_tokens=page)
    eng.debug_tune(3, attention)
    prompts = [list(wl.zipf_tokens(n, shape.vocab, n)) for n in lens]
    for i, p in enumerate(prompts):
        eng.prefill(i, p)
    drafts = np.random.default_rng(page).integers(0, shape.vocab, size=(3, 16)).astype(np.int32)
    dd = torch.from_numpy(drafts).cuda()
    _, _, two = eng.validate([0, 1], [7, 7], dd[:2].contiguous(), want_logits=True)       # 16 rows
    _, _, three = eng.validate([0, 1, 2], [7, 7, 7], dd, want_logits=True)                # 24
    tt, _, one = eng.validate([2], [16], dd[2:].contiguous(), want_logits=True)           # 17
    eng.sync()
    two, three, one, tt = two.cpu().numpy(), three.cpu().numpy(), one.cpu().numpy(), tt.cpu().numpy()
    assert np.array_equal(two, three[:16])
    for i in range(2):
        ref, _ = gu.oracle_stair_logits(tgt, prompts[i], drafts[i][:7])
        gu.check_rows_against_oracle(two[8 * i:8 * i + 8], ref.argmax(1), ref, gu.LOGIT_TOL_BF16)
    ref, _ = gu.oracle_stair_logits(tgt, prompts[2], drafts[2])
    gu.check_rows_against_oracle(one, tt[0][:17], ref, gu.LOGIT_TOL_BF16)
    eng.close()


def test_calls_of_a_row_box_wait_for_the_stream_once():
    # a model whose calls of few and of more rows take different programs (heads of 80): 16 rows first, then every smaller number while
    # the stream is busy
    st = _stairs()
    shape = wl.workload(3).target.replace(n_layers=1, vocab=2048)
    src = wl.WeightSource(shape, 1, "torch-cuda")
    eng = st.Stairs(src, None, max_requests=1, max_seq_len=64, k_max=15, kv_page_tokens=16)
    eng.prefill(0, list(wl.zipf_tokens(20, shape.vocab, 1)))
    draft = torch.zeros((1, 15), dtype=torch.int32, device="cuda")
    kept = [eng.validate([0], [15], draft)]
    eng.sync()
    torch.cuda._sleep(400_000_000)
    busy = torch.cuda.Event()
    busy.record()
    kept += [eng.validate([0], [k], draft) for k in range(15)]
    assert not busy.query()
    eng.close()


@pytest.mark.parametrize("wide_d", [False, True], ids=["", "33_tiles"])
@pytest.mark.parametrize("attention", [1, 2], ids=["register", "tcgen05"])
@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_both_ways_of_finishing_split_tiles_give_the_same_bits(shape, attention, wide_d):
    # rows that are fewer than a tile's CTAs, one to several a warp, in one and in several 16-row chunks; vocabularies of whole and of
    # cut tiles; row statistics over more than 32 column tiles
    st = _stairs()
    shape = shape.replace(vocab=2044, n_layers=2)
    if wide_d:
        if shape.d_model % 128:
            pytest.skip("one width is enough")
        shape = shape.replace(d_model=33 * 128)
    tsrc, _ = sources(shape)
    eng = st.Stairs(tsrc, None, max_requests=4, max_seq_len=200, k_max=15, kv_page_tokens=16)
    eng.debug_tune(3, attention)
    for i in range(4):
        eng.prefill(i, list(wl.zipf_tokens(100 + i, shape.vocab, i)))
    drafts = torch.from_numpy(np.random.default_rng(5).integers(0, shape.vocab, size=(4, 15)).astype(np.int32)).cuda()
    for ks in ([0], [4], [8], [15], [7, 9], [15, 15, 15, 15]):
        got = []
        for way in (1, 2):
            eng.debug_tune(7, way)
            tt, al, lg = eng.validate(list(range(len(ks))), ks, drafts[:len(ks)].contiguous(), want_logits=True)
            eng.sync()
            got.append((tt.clone(), al.clone(), lg.clone()))
        for a, b in zip(*got):
            assert torch.equal(a, b)
        for which in (7, 8):   # every word of the parked sums and states is empty again
            assert bool((eng.debug_buffer(which, torch.int32, 1 << 16) == -1).all())
    eng.close()
