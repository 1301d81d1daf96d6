"""The one-kernel forward of small fp32 models against the oracle: rows beyond one staging pass (32), more (row, head) pairs
than warps, all head sizes, grouped queries, batches, keys beyond one block per warp - and the same steps through the separate
kernels.  fp32 on both sides, sums in other orders: logits within 2e-4, streams and accept decisions equal."""
import numpy as np
import pytest

import oracle
from paper_2311_08263_b200 import engine, lib as _l, workload as wl

pytestmark = pytest.mark.gpu

CASES = [
    # hq, hkv, hd, d, d_ffn, vocab, c, lens
    (4, 4, 32, 128, 512, 512, 8, [32]),
    (4, 4, 32, 128, 512, 500, 1, [1, 2, 33, 200]),
    (8, 2, 64, 192, 360, 1000, 11, [40, 3, 70]),         # 33 rows: one more than a staging pass; 264 pairs on 512 warps
    (4, 1, 128, 256, 264, 77, 64, [300, 65]),            # 128 rows, window wider than the cache, 600 pairs
    (16, 16, 32, 128, 136, 300, 33, [129, 17]),          # 1056 pairs: several per warp group
]


@pytest.mark.parametrize("flags", [0, _l.FC_FLAG_NO_CHAIN])
@pytest.mark.parametrize("hq,hkv,hd,d,d_ffn,vocab,c,lens", CASES)
def test_small_forward(hq, hkv, hd, d, d_ffn, vocab, c, lens, flags):
    cfg = wl.small_config(dtype="f32", n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_model=d, d_ffn=d_ffn, vocab=vocab,
                          prompt_len=max(lens), bias_beta=4.0, seed=700 + c)
    B, steps = len(lens), 3
    w = wl.make_weights(cfg)
    ids, _ = wl.make_prompts(cfg, batch=B, lens=lens)
    max_seq = max(lens) + (steps + 1) * c
    dec = engine.Decoder(cfg, w, B, c, max_seq, flags=flags)
    dec.fc_prefill(ids.numpy(), lens, c)
    logits = dec.fc_debug_logits(True)
    orc = []
    for b, P in enumerate(lens):
        orc.append(oracle.Oracle(cfg, w, max_seq))
        orc[b].prefill(ids[b, :P].numpy(), c)
    for _ in range(steps):
        cnt, tok, win = dec.fc_jacobi_step()
        assert dec.fc_last_launch_count() == (1 if flags == 0 else 6 * cfg.n_layers + 3)
        lg = logits.cpu().numpy().reshape(B, c, vocab)
        for b in range(B):
            k, acc, wnew, ref = orc[b].jacobi_step(want_logits=True)
            assert np.abs(lg[b] - ref).max() < 2e-4
            assert cnt[b] == k and tok[b, :k].tolist() == acc.tolist() and win[b].tolist() == wnew.tolist()
    for o in orc:
        o.close()
    assert dec.fc_debug_check_guards() == 0
