"""Passes of small fp32 models in one launch of one cluster: logits within the fp32 bar and identical tokens
against the oracle, for both families, head sizes, row counts around the eight-row blocks, split contexts, and against
the per-operation kernels."""
import numpy as np
import pytest
import torch

from oracle import stairs_oracle as so
from paper_2407_19947_b200 import workloads as wl
from tests import gpu_util as gu
from tests.test_gpu_parity import _stairs, sources

pytestmark = pytest.mark.gpu

F32 = wl.WDTYPE_F32
SHAPES = {"family_a": wl.family_a(2, 256, 4, 1024, 1024, 512, F32), "odd_widths": wl.family_a(3, 200, 5, 328, 1003, 512, F32),
          "gqa_rope": wl.family_b(2, 256, 8, 2, 64, 520, 777, 512, F32), "hd128": wl.family_b(1, 384, 3, 1, 128, 800, 2050, 512, F32),
          "wide_ff": wl.family_b(1, 128, 4, 4, 24, 1600, 512, 512, F32)}


@pytest.mark.parametrize("shape", SHAPES.values(), ids=SHAPES.keys())
def test_small_fp32_passes_match_oracle(shape):
    st = _stairs()
    tsrc, dsrc = sources(shape, std=0.03)
    tgt, drf = gu.oracle_pair(tsrc, dsrc)
    lens = [9, 41, 150, 4]
    eng = st.Stairs(tsrc, dsrc, max_requests=4, max_seq_len=256, k_max=8, kv_page_tokens=16)
    plain = st.Stairs(tsrc, dsrc, max_requests=4, max_seq_len=256, k_max=8, kv_page_tokens=16, gemm_impl=1)
    prompts = [list(wl.zipf_tokens(n, shape.vocab, 70 + i)) for i, n in enumerate(lens)]
    for e in (eng, plain):
        for i, p in enumerate(prompts):
            e.prefill(i, p)
    drafts = np.random.default_rng(3).integers(0, shape.vocab, size=(4, 8)).astype(np.int32)
    for i in range(4):
        want = so.draft_tokens(drf, prompts[i], 5)
        launches = eng.launch_count()
        got = eng.draft(i, 5)
        eng.sync()
        assert got.cpu().numpy()[:5].tolist() == [int(x) for x in want]
        assert eng.launch_count() - launches == 1
        drafts[i, : 3] = want[:3]
    dd = torch.from_numpy(drafts).cuda()
    for reqs, ks in (([0, 1, 2, 3], [8, 0, 3, 5]), ([2], [8]), ([1, 3], [7, 6]), ([3], [0])):
        d = dd[reqs].contiguous()
        tt, al, lg = eng.validate(reqs, ks, d, want_logits=True)
        tt2, al2, lg2 = plain.validate(reqs, ks, d, want_logits=True)
        eng.sync(); plain.sync()
        assert float((lg - lg2).abs().max()) < 1e-4
        assert torch.equal(tt, tt2) and torch.equal(al, al2)
        row = 0
        for j, r in enumerate(reqs):
            ref, _ = gu.oracle_stair_logits(tgt, prompts[r], drafts[r, : ks[j]])
            gu.check_rows_against_oracle(lg[row: row + ks[j] + 1].cpu().numpy(), tt.cpu().numpy()[j], ref, gu.LOGIT_TOL_F32)
            # bit for bit the same alone as in a batch
            if len(reqs) == 4:
                _, _, alone = eng.validate([r], [ks[j]], d[j: j + 1].contiguous(), want_logits=True)
                eng.sync()
                assert torch.equal(alone, lg[row: row + ks[j] + 1])
            row += ks[j] + 1
    eng.close(); plain.close()


@pytest.mark.parametrize("k,n_req,launches", [(0, 16, 1), (1, 16, 1), (7, 16, 1), (8, 8, 1), (15, 8, 1), (16, 1, None), (8, 9, None)])
def test_requests_dealt_to_clusters_match_the_per_operation_kernels(k, n_req, launches):
    # one and two passes a cluster, every cluster in use, one row or one request too many
    st = _stairs()
    shape = SHAPES["odd_widths"]
    tsrc, _ = sources(shape, std=0.03)
    got = []
    for impl in (0, 1):
        eng = st.Stairs(tsrc, None, max_requests=16, max_seq_len=128, k_max=16, kv_page_tokens=16, gemm_impl=impl)
        for i in range(n_req):
            eng.prefill(i, list(wl.zipf_tokens(3 + 5 * i, shape.vocab, i)))
        drafts = torch.from_numpy(np.random.default_rng(k).integers(0, shape.vocab, size=(n_req, 16)).astype(np.int32)).cuda()
        before = eng.launch_count()
        tt, al, lg = eng.validate(list(range(n_req)), [k] * n_req, drafts, want_logits=True)
        eng.sync()
        if impl == 0:
            assert (eng.launch_count() - before == 1) == (launches == 1)
        got.append((tt.cpu(), al.cpu(), lg.cpu()))
        eng.close()
    assert torch.equal(got[0][0][:, : k + 1], got[1][0][:, : k + 1]) and torch.equal(got[0][1], got[1][1])
    assert float((got[0][2] - got[1][2]).abs().max()) < 1e-4


@pytest.mark.parametrize("k", [4, 11])
def test_rows_are_the_same_in_clusters_of_eight_and_sixteen_ctas(k):
    # eight requests: eight clusters, which run at once only in the smaller size; one request: one cluster of 16
    st = _stairs()
    shape = SHAPES["gqa_rope"]
    tsrc, _ = sources(shape, std=0.03)
    eng = st.Stairs(tsrc, None, max_requests=8, max_seq_len=320, k_max=k, kv_page_tokens=16)
    for i in range(8):
        eng.prefill(i, list(wl.zipf_tokens(3 + 41 * i, shape.vocab, i)))
    drafts = torch.from_numpy(np.random.default_rng(k).integers(0, shape.vocab, size=(8, k)).astype(np.int32)).cuda()
    before = eng.launch_count()
    tt, al, lg = eng.validate(list(range(8)), [k] * 8, drafts, want_logits=True)
    assert eng.launch_count() - before == 1
    for i in range(8):
        tt1, al1, lg1 = eng.validate([i], [k], drafts[i:i + 1].contiguous(), want_logits=True)
        assert torch.equal(lg1, lg[i * (k + 1):(i + 1) * (k + 1)]) and torch.equal(tt1[0], tt[i]) and torch.equal(al1[0], al[i])
    eng.sync()
    eng.close()


@pytest.mark.parametrize("vocab,launches", [(512, 1), (128256, None)])
def test_a_large_vocabulary_is_left_to_the_per_operation_kernels(vocab, launches):
    # one cluster reads the LM head at a fraction of the chip's rate; the results are the per-operation kernels' either way
    st = _stairs()
    shape = wl.family_a(1, 128, 2, 256, vocab, 128, F32)
    tsrc, dsrc = sources(shape, std=0.03)
    got = []
    for impl in (0, 1):
        eng = st.Stairs(tsrc, dsrc, max_requests=1, max_seq_len=64, k_max=8, kv_page_tokens=16, gemm_impl=impl)
        eng.prefill(0, list(wl.zipf_tokens(20, shape.vocab, 1)))
        before = eng.launch_count()
        draft = eng.draft(0, 4)
        mid = eng.launch_count()
        tt, al, lg = eng.validate([0], [8], draft, want_logits=True)
        if impl == 0:
            assert (mid - before == 1) == (launches == 1) and (eng.launch_count() - mid == 1) == (launches == 1)
        eng.sync()
        got.append((draft.cpu(), tt.cpu(), al.cpu(), lg.cpu()))
        eng.close()
    assert all(torch.equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))
    assert float((got[0][3] - got[1][3]).abs().max()) < 1e-4
