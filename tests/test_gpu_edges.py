"""GPU parity at the sizes where a kernel's split or a dispatch changes: edges of tiles, strips,
runs and clusters, the smallest and largest of each range, against the fp64 oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import pace_oracle as O
from paper_2608_27206_gb300 import synth
from tests.helpers import assert_distances_close, assert_scores_close, bf16_tensor, f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pace():
    from paper_2608_27206_gb300 import build
    build.build()
    from paper_2608_27206_gb300 import pace as P
    P.pace_init(0)
    P.pace_device_status(clear=True)
    yield P
    assert P.pace_device_status(clear=True)[0] == 0


def _cu(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


# last query tile of 128 rows or fewer (half a tile) and above, alone (rows past the image are the
# tensor's zero fill) and followed by another image (rows overwritten), one tile and several
@pytest.mark.parametrize("lens", [(4,), (128,), (132,), (256,), (384,), (388, 4), (260, 128), (516, 1284, 1028)])
def test_vit_last_tile(pace, lens):
    cu = _cu(lens)
    q, k = (synth.random_small_qk(s + len(lens), int(cu[-1]), 3, 80) for s in (1, 2))
    got = pace.pace_vit_attn_importance(bf16_tensor(q), bf16_tensor(k), cu, merge=4).cpu().numpy()
    assert_scores_close(got, O.vit_attn_importance(f64(q), f64(k), cu, 80 ** -0.5, 4))


# few keys and several heads per KV head: pass 2 splits a group's heads over CTAs (7 heads; 1 and 2
# query tiles), down to one stream item per CTA
@pytest.mark.parametrize("tq,nv", [((1,), (1,)), ((128,), (300,)), ((129,), (128,)), ((257, 5), (40, 513))])
def test_llm_stream_splits(pace, tq, nv):
    cq, cv = _cu(tq), _cu(nv)
    q, k = synth.random_small_qk(3, int(cq[-1]), 14, 128), synth.random_small_qk(4, int(cv[-1]), 2, 128)
    got = pace.pace_llm_text_visual_importance(bf16_tensor(q), bf16_tensor(k), cq, cv).cpu().numpy()
    assert_scores_close(got, O.llm_text_visual_importance(f64(q), f64(k), cq, cv, 128 ** -0.5))


# causal streams whose lengths differ from CTA to CTA, split or not, in a batch
@pytest.mark.parametrize("before,nv,after", [((0,), (1,), (0,)), ((7,), (600,), (130,)), ((3, 20), (129, 700), (1, 300))])
@pytest.mark.parametrize("query_set", ["vision_text", "text", "last"])
def test_sequence_stream_splits(pace, before, nv, after, query_set):
    cu = _cu([a + b + c for a, b, c in zip(before, nv, after)])
    q, k = synth.random_small_qk(5, int(cu[-1]), 14, 128), synth.random_small_qk(6, int(cu[-1]), 2, 128)
    got = pace.pace_llm_sequence_importance(bf16_tensor(q), bf16_tensor(k), cu, before, nv, query_set).cpu().numpy()
    assert_scores_close(got, O.llm_sequence_importance(f64(q), f64(k), cu, before, nv, 128 ** -0.5, query_set))


# element widths 16, 4 and 1, blocks of 1024 elements with remainders, several tensors and slabs,
# rows out of range
@pytest.mark.parametrize("n_idx", [1, 63, 64, 65, 341])
def test_gather_multi_blocks(pace, n_idx):
    rng = np.random.default_rng(n_idx)
    idx = rng.integers(0, 50, n_idx).astype(np.int32)
    shapes = [((50, 8, 16), 0), ((3, 50), 1), ((2, 3, 50, 64), 2), ((50, 5), 0), ((2, 50, 3), 1)]
    src = [torch.from_numpy(rng.integers(0, 255, s, dtype=np.uint8)).cuda() for s, _ in shapes]
    src[1] = src[1].to(torch.int32)
    dst = [torch.zeros(s[:d] + (n_idx,) + s[d + 1:], dtype=t.dtype, device="cuda") for t, (s, d) in zip(src, shapes)]
    specs = [pace.gather_spec(a, b, d) for a, b, (_, d) in zip(src, dst, shapes)]
    pace.pace_gather_multi(specs, torch.from_numpy(idx).cuda())
    for a, b, (_, d) in zip(src, dst, shapes):
        assert torch.equal(b, a.index_select(d, torch.from_numpy(idx).cuda().long()))
    idx[0] = 50
    pace.pace_gather_multi(specs, torch.from_numpy(idx).cuda())
    assert pace.pace_device_status(clear=True) == (pace.PACE_ERR_INVALID_ARG, 13)
    for b, (_, d) in zip(dst, shapes):
        assert not b.select(d, 0).any()
