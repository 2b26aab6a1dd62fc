"""The append's cluster forms (a token tile's columns of c over 2, 3, 4 or 8
CTAs) against the oracle: every cluster size a width picks, clusters in two
rounds, ragged tiles, and an odd number of K blocks (a short last stage). And
its pairs of tiles: odd numbers of tiles, tiles of two batch elements in a pair,
fewer and more K blocks than ring stages, one to six rounds per pair."""

import pytest
import torch

from paper_2605_30351_gb300 import synth
from paper_2605_30351_gb300 import videomla as V

from test_gpu_parity import assert_close, f64, run_chunks, small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    V.load()
    V.mla_device_status(clear=True)
    yield
    assert V.mla_device_status(clear=True) == V.MLA_OK


@pytest.mark.parametrize("d_c,d_r,grid,batch,hidden", [
    (128, 64, (8, 8), 60, 1536),    # 60 tiles: pairs
    (192, 32, (5, 7), 20, 1472),    # 20 ragged tiles: threes; 23 K blocks
    (192, 64, (8, 8), 60, 1536),    # 60 tiles: pairs of 96 columns
    (256, 32, (10, 13), 10, 1536),  # 2 tiles per element, the second with 2 tokens: fours
    (256, 64, (8, 8), 60, 64),      # 60 tiles: pairs of 128 columns; one K block
    (512, 32, (1, 1), 1, 1536),     # one token: eights
    (512, 64, (8, 8), 30, 1472),    # fours
    (512, 32, (8, 8), 45, 1536),    # fours in two rounds
    (192, 32, (5, 7), 331, 192),    # persistent pairs: 331 tiles, three K blocks
    (192, 64, (10, 13), 155, 640),  # 310 tiles, two per element, both accumulators full
    (128, 32, (10, 13), 201, 64),   # one K block: every tile its own stage
    (64, 64, (1, 1), 807, 128),     # the odd CTA's weights are k^R alone; six rounds
    (64, 32, (5, 7), 305, 1536),    # one tile past two waves; the odd CTA has both
    (256, 32, (8, 8), 153, 1472),   # pairs of one tile each
    (512, 64, (8, 8), 101, 1536),   # and halves of c and k^R
    (512, 32, (10, 13), 40, 64),
])
def test_append_cluster_and_pair_forms(d_c, d_r, grid, batch, hidden):
    w = small(d_c=d_c, d_r=d_r, rope_pairs=(6, 5, 5) if d_r == 32 else (12, 10, 10),
              rope_axis_dims=(44, 42, 42) if d_r == 32 else (64, 64, 64), grid_h=grid[0],
              grid_w=grid[1], window_frames=3, batch=batch, hidden=hidden)
    weights = synth.draw_layer_weights(w, 41)
    weights["gamma_kv"] = synth.bf16(1.0 + 0.25 * torch.randn(
        d_c, generator=torch.Generator().manual_seed(42)).numpy())
    cache, oc = run_chunks(w, weights, [(0, 1), (1, 1)])
    valid = oc.valid_slots()
    assert_close(f64(cache.c)[:, valid], oc.c[:, valid], what="c")
    assert_close(f64(cache.kr)[:, valid], oc.kr[:, valid], what="k")
