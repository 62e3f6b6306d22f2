"""The forms a kernel takes by size, each at the sizes where it starts, ends or leaves a remainder, against the CPU checker."""
import numpy as np
import pytest
import torch

from paper_2601_01712_b200 import synth
from tests.helpers import TOL_BF16, bf16_noise_bounds, max_abs_err, oracle_model, oracle_scores, small_bf16_shape
from tests.test_gpu_parity import _setup, _tiny_batch

pytestmark = pytest.mark.gpu


# Rows of a ranking call (short-term + candidates) around the limits between the forms of the fused feed-forward kernel, 32-row tiles in
# clusters of 8 / 4 / 2, 64-row tiles in clusters of 2, 128-row tiles in clusters of 2, 256-row tiles in pairs, and its chunk
# counts: not a multiple of the cluster, fewer than the largest cluster, two per CTA.
@pytest.mark.parametrize("rows,ff", [(1, 1024), (33, 2048), (480, 1024), (481, 1024), (600, 1152), (97, 512), (1120, 1024), (1185, 256), (1200, 640),
                                     (2369, 1024), (2500, 256), (4737, 1024), (4800, 1408), (9473, 1024)])
def test_feed_forward_forms(rows, ff):
    shape = small_bf16_shape(vocab=3000, ff=ff)
    users = max(1, rows // 300)
    cand = [rows // users] * users
    cand[-1] += rows - sum(cand)
    short = [0 if c < 8 else c // 8 for c in cand]
    batch = _tiny_batch(shape, rows + ff, [70] * users, short, [c - s for c, s in zip(cand, short)])
    w, model, pool, db = _setup(shape, 61, batch)
    pool.preinfer(db)
    scores = pool.rank(db).cpu().numpy()
    assert model.device_status() == 0
    sample = sorted({0, users // 2, users - 1})
    om = oracle_model(shape, w)
    want = oracle_scores(om, batch, users=sample)
    max_bound, rms_bound, _ = bf16_noise_bounds(shape, w, batch, want)
    assert max_abs_err(scores, batch, want) <= max_bound
    err = np.concatenate([scores[batch.cand_off[i]:batch.cand_off[i + 1]] - v for i, v in want.items()])
    if len(err) >= 100:                                 # (a handful of errors is no sample of their size)
        assert np.sqrt(np.mean(err ** 2)) <= rms_bound
    pool.close(); model.close()


# The merge of split attention items: more partials than one batch of loads (17 per tile), and many tiles with few (the form for occupancy).
@pytest.mark.parametrize("prefix,cand,kind", [([4500], [40], 0), ([4500], [40], 1), ([1024] * 12, [60] * 12, 0)])
def test_attention_merge_forms(prefix, cand, kind):
    shape = small_bf16_shape(vocab=3000, attn_kind=kind)
    batch = _tiny_batch(shape, 7 + len(prefix), prefix, [3] * len(prefix), cand)
    w, model, pool, db = _setup(shape, 62, batch)
    pool.preinfer(db)
    scores = pool.rank(db).cpu().numpy()
    assert model.device_status() == 0
    want = oracle_scores(oracle_model(shape, w), batch, users=sorted({0, len(prefix) - 1}))
    max_bound, _, _ = bf16_noise_bounds(shape, w, batch, want)
    assert max_abs_err(scores, batch, want) <= max_bound
    pool.close(); model.close()
