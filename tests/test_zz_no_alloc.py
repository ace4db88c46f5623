"""stairs_accept_static: the entry point for callers that cannot allocate device memory (code
running inside a pool that owns the device, or handed only finished buffers), so they have
neither a workspace nor a context.  Its scratch is a fixed array inside the library.  The
test feeds it the logits that stairs_validate dumped and expects exactly the tokens and accept
lengths stairs_validate itself returned (integers: the bar is equality), on two calls in a row
with different shapes, which also shows that stale keys from the first call are cleared."""
import numpy as np
import pytest
import torch

from paper_2407_19947_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_static_accept_matches_validate_on_two_calls_in_a_row():
    from paper_2407_19947_b200 import build, stairs
    build.build()
    shape = wl.family_b(2, 256, 8, 2, 64, 512, 4096, 256)
    src = wl.WeightSource(shape, 13, "numpy", norm_jitter=0.1, std=0.03)
    eng = stairs.Stairs(src, None, max_requests=2, max_seq_len=96, k_max=6, kv_page_tokens=16)
    eng.prefill(0, list(wl.zipf_tokens(30, shape.vocab, 1)))
    eng.prefill(1, list(wl.zipf_tokens(17, shape.vocab, 2)))
    rng = np.random.default_rng(0)
    for ks in ([6, 2], [0, 5]):
        # drafts that agree with the model for a while: take the model's own tokens, then corrupt one
        probe = torch.from_numpy(rng.integers(0, shape.vocab, size=(2, 6)).astype(np.int32)).cuda()
        tt0, _, _ = eng.validate([0, 1], ks, probe)
        eng.sync()
        drafts = probe.clone()
        drafts[0, 0] = tt0[0, 0]
        drafts[1, 0] = tt0[1, 0]
        tt, al, logits = eng.validate([0, 1], ks, drafts, want_logits=True)
        eng.sync()
        tt_s, al_s = stairs.accept_static(logits, ks, drafts, 6)
        torch.cuda.synchronize()
        for i, k in enumerate(ks):
            assert torch.equal(tt_s[i, : k + 1], tt[i, : k + 1])
        assert torch.equal(al_s, al)
        assert int(al[0]) >= (1 if ks[0] > 0 else 0)
    eng.close()


def test_static_accept_rejects_sizes_beyond_its_fixed_scratch():
    from paper_2407_19947_b200 import build, stairs
    build.build()
    logits = torch.zeros((4, 128), dtype=torch.float32, device="cuda")
    drafts = torch.zeros((70, 63), dtype=torch.int32, device="cuda")
    # the checks run on the host before anything is launched, so undersized buffers are safe here
    with pytest.raises(stairs.StairsError) as e:
        stairs.accept_static(logits, [0] * (stairs.STATIC_MAX_REQ + 1), drafts, 63)
    assert e.value.code == 2 and "n_req" in str(e.value)
    with pytest.raises(stairs.StairsError) as e:
        stairs.accept_static(logits, [63] * 64, drafts, 63)            # 4096 rows > 1024
    assert e.value.code == 2 and "rows" in str(e.value)
    with pytest.raises(stairs.StairsError) as e:
        stairs.accept_static(logits, [5], drafts, 4)                   # k above k_max
    assert e.value.code == 1


@pytest.mark.parametrize("vocab,ld", [(1, 1), (5, 8), (127, 128), (2049, 2051), (8192, 8192), (8193, 8196), (16384, 16384), (16385, 16388), (32000, 32000), (70001, 70004)])
@pytest.mark.parametrize("ks", [[0], [4], [63], [2, 0, 5], [1] * 64], ids=lambda k: f"{len(k)}x{max(k) + 1}")
def test_static_accept_equals_torch_argmax(vocab, ld, ks):
    # one cluster per request, and the many-block form for few long requests; odd row lengths, unaligned
    # rows, ties (lowest index wins), both sides of the lengths at which a slice is cut in two and in four
    from paper_2407_19947_b200 import build, stairs
    build.build()
    rows, k_max = sum(ks) + len(ks), max(ks)
    g = torch.Generator(device="cuda")
    g.manual_seed(vocab + rows)
    store = torch.randint(-4, 5 if vocab > 300 else 3, (rows, ld), generator=g, device="cuda").float()
    store[:, vocab:] = 100.0                                     # past the vocabulary: must not be looked at
    lg = store[:, :vocab].cpu().numpy()
    want = lg.argmax(axis=1)
    draft = torch.randint(0, vocab, (len(ks), max(k_max, 1)), generator=g, device="cuda", dtype=torch.int32)
    row = 0
    for i, k in enumerate(ks):
        for r in range(k // 2):
            draft[i, r] = int(want[row + r])
        row += k + 1
    tt, al = stairs.accept_static(store, ks, draft if k_max else None, k_max, vocab=vocab)
    torch.cuda.synchronize()
    tt, al, d, row = tt.cpu().numpy(), al.cpu().numpy(), draft.cpu().numpy(), 0
    for i, k in enumerate(ks):
        assert tt[i, : k + 1].tolist() == want[row: row + k + 1].tolist()
        assert (tt[i, k + 1:] == 0).all()
        miss = [r for r in range(k) if d[i, r] != tt[i, r]]
        assert int(al[i]) == (miss[0] if miss else k)
        row += k + 1


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n_req", [39, 40, 64])      # on both sides of the calls that are started behind the previous kernel
@pytest.mark.parametrize("ld", [16500, 16501], ids=["vectors", "scalars"])
def test_static_accept_waits_for_the_kernels_before_it(ld, n_req, captured):
    # the logits and drafts of every call are written by kernels right before it, and its results read right behind it; rows on
    # 16-byte boundaries (whole vectors are loaded) and others
    from paper_2407_19947_b200 import build, stairs
    build.build()
    vocab, k, calls = 16500, 3, 12
    g = torch.Generator(device="cuda")
    g.manual_seed(n_req)
    src = torch.randn((calls, n_req * (k + 1), ld), generator=g, device="cuda")
    want = src[:, :, :vocab].argmax(dim=2).view(calls, n_req, k + 1).to(torch.int32)
    logits, draft = torch.empty_like(src[0]), torch.zeros((n_req, k), dtype=torch.int32, device="cuda")
    got_t, got_a = torch.zeros_like(want), torch.zeros((calls, n_req), dtype=torch.int32, device="cuda")

    def one(i, stream=None):
        logits.copy_(src[i])
        draft.copy_(want[i, :, :k])
        draft[:, i % k] += 1                          # the first mismatch of every request
        tt, al = stairs.accept_static(logits, [k] * n_req, draft, k, stream=stream, vocab=vocab)
        got_t[i].copy_(tt)
        got_a[i].copy_(al)

    one(0)
    torch.cuda.synchronize()
    if captured:
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            for i in range(calls):
                one(i, side)
        for _ in range(3):
            got_t.zero_()
            got_a.zero_()
            graph.replay()
    else:
        for i in range(calls):
            one(i)
    torch.cuda.synchronize()
    assert torch.equal(got_t, want)
    assert torch.equal(got_a, (torch.arange(calls, device="cuda", dtype=torch.int32) % k).view(-1, 1).expand(calls, n_req))
