"""Row statistics that the residual GEMMs publish for the next normalisation (count, mean, centred sum of squares per part of a row),
against the same rows in 64 bits, where a channel far larger than the rest sits in the first column of a tile or further in: every way a
residual GEMM finishes its rows."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2407_19947_b200 import workloads as wl
from tests.test_gpu_parity import _stairs, small_a, small_b

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


class _OutlierChannels(wl.WeightSource):
    column = 0

    def _draw_numpy(self, layer, name):
        a = super()._draw_numpy(layer, name)
        if name == "tok_emb":
            a[:, self.column::128] = 100.0 * (1.0 + a[:, self.column::128])      # 3000 times the other channels
        return a


def _parts(eng, which, rows, stride, d):
    words = eng.debug_buffer(which, torch.float32, 4 * (rows * stride if stride else 2 * d // 32)).view(-1, 4).double().cpu().numpy()
    if not stride:       # as many parts as it takes to cover the first row
        stride = int(np.flatnonzero(np.cumsum(words[:, 2]) == d)[0]) + 1
        words = eng.debug_buffer(which, torch.float32, 4 * rows * stride).view(-1, 4).double().cpu().numpy()
    return words.reshape(rows, stride, 4)[:, :, :3]


# (requests of five rows, tuning knobs, roundings of a sum of squares on its way, as counted below)
FORMS = {"one_cta": (1, {7: 1}, 28), "shared": (1, {7: 2}, 28), "one_cta_40_rows": (8, {7: 1}, 28), "shared_40_rows": (8, {7: 2}, 28),
         "80_rows": (16, {}, 28), "80_rows_split": (16, {6: 3}, 28),
         "130_rows": (26, {4: 1, 5: 1}, 64), "130_rows_split": (26, {4: 1, 5: 4}, 64), "130_rows_pair": (26, {4: 2}, 64)}


@pytest.mark.parametrize("form", FORMS.values(), ids=FORMS.keys())
@pytest.mark.parametrize("column", [0, 77])
@pytest.mark.parametrize("shape", [small_b(8, 2, 64, d=512, layers=2), small_b(4, 4, 48, d=192, f=320, layers=2), small_a(layers=2)], ids=["gqa", "d192", "family_a"])
def test_row_statistics_with_outlier_channels(shape, column, form):
    n, knobs, roundings = form
    st = _stairs()
    src = _OutlierChannels(shape, 3, "numpy", norm_jitter=0.1, std=0.03)
    src.column = column
    eng = st.Stairs(src, None, max_requests=n, max_seq_len=64, k_max=4, kv_page_tokens=16)
    for what, value in knobs.items():
        eng.debug_tune(what, value)
    for i in range(n):
        eng.prefill(i, list(wl.zipf_tokens(10 + i, shape.vocab, i)))
    drafts = torch.from_numpy(np.random.default_rng(1).integers(0, shape.vocab, size=(n, 4)).astype(np.int32)).cuda()
    eng.validate(list(range(n)), [4] * n, drafts)
    rows, d = 5 * n, shape.d_model
    x = eng.debug_buffer(0, torch.float32, rows * d).view(rows, d).double().cpu().numpy()
    got = _parts(eng, 9, rows, (d + 127) // 128, d) if rows <= 64 else _parts(eng, 10, rows, 0, d)
    eng.close()
    count, mean, m2 = got[:, :, 2], got[:, :, 0], got[:, :, 1]
    assert (count.sum(1) == d).all()
    row_mean = (count * mean).sum(1) / d
    row_m2 = (m2 + count * (mean - row_mean[:, None]) ** 2).sum(1)
    want_mean = x.mean(1)
    want_m2 = ((x - want_mean[:, None]) ** 2).sum(1)
    # Means: four values (one of them large at most), then merged pair by pair or, in many-row passes, chunk by chunk; off by
    # EPS max|x| / 4 (2 + 2 (1 + 1/2 + ... + 1/8)) at most.  Squares around them: all terms are positive, so roundings are relative.  Pair by pair: 5 for
    # four values, 3 a level for five levels of additions and products, and a difference of means that is off by up to 4 in either, squared:
    # 28.  Chunk by chunk: up to 8 running merges of 4 more each: 64.  Between parts the error of a mean counts times its distance from the row's.
    off = 2 * EPS * np.abs(x).max(1)
    assert (np.abs(row_mean - want_mean) <= off).all()
    bound = roundings * EPS * want_m2 + 2 * off * (count * np.abs(mean - row_mean[:, None])).sum(1) + d * off ** 2
    assert (np.abs(row_m2 - want_m2) <= bound).all(), np.max(np.abs(row_m2 / want_m2 - 1)) / EPS
