"""The streaming attention kernels, reached through a Jacobi step with enough work for them, against the oracle: cached
lengths around the 32-key tiles (0, 1, 31, 32, 33 ..), rings that wrap, one, two and more query tiles per kv head, grouped
queries, both head sizes.  Bars and margin rule as in test_gpu_full_configs."""
import pytest

from paper_2311_08263_b200 import workload as wl
from test_gpu_full_configs import _random_kv_case

pytestmark = pytest.mark.gpu

EDGES = [1100, 0, 1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 191, 192, 193, 1023]

CASES = [
    # hq, hkv, hd, c, lens                  units (kv heads x sequences x query tiles) x 64-key tiles of the longest
    (16, 4, 64, 1, EDGES),                  # 64 x 18: grouped queries, one row per sequence
    (8, 8, 128, 1, EDGES),                  # 128 x 18: one query per tile
    (8, 8, 128, 20, [560, 0, 5, 12, 13, 300, 500, 559]),     # 128 x 10: two query tiles, the second ragged
    (8, 4, 64, 40, [900, 0, 23, 871]),      # 80 x 15: five query tiles in two groups of four, windows over tile edges
    (8, 4, 128, 64, [1000, 1, 64, 448]),    # 128 x 17: whole groups
]


@pytest.mark.parametrize("hq,hkv,hd,c,lens", CASES)
def test_step_over_streamed_cache(hq, hkv, hd, c, lens):
    cfg = wl.small_config(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_model=256, d_ffn=512, vocab=1000, seed=91 + hd + c)
    dec, _ = _random_kv_case(cfg, lens, c, range(len(lens)))
    # one kernel more per layer than with the fused attention (the vocabulary is no whole number of weight tiles, so that
    # the chained launch takes any number of rows)
    assert dec.fc_last_launch_count() == 3 * cfg.n_layers + 4


@pytest.mark.parametrize("heads,c", [(32, 32), (40, 24), (40, 50)])
def test_one_sequence_with_an_odd_number_of_key_splits(heads, c):
    """32 and 40 (kv head, query group) pairs: seven and six splits, as many clusters as run at the same time."""
    cfg = wl.small_config(n_layers=2, n_heads=heads, n_kv_heads=heads, head_dim=128, d_model=256, d_ffn=512, vocab=1000, seed=190 + c)
    dec, _ = _random_kv_case(cfg, [1471], c, [0])
    assert dec.fc_last_launch_count() == 3 * cfg.n_layers + 4
