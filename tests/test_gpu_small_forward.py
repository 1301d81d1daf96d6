"""The one-kernel forward of small fp32 models against the oracle: rows beyond one staging pass (32), more (row, head) pairs
than warps, all head sizes, grouped queries, batches, keys beyond one block per warp - and the same steps through the separate
kernels.  fp32 on both sides, sums in other orders: logits within 2e-4, streams and accept decisions equal."""
import numpy as np
import pytest
import torch

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


def _shifted(t):
    """The same values one element behind a 16-byte boundary, as in a packed buffer."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    assert flat.data_ptr() % 16 == 0
    flat[1:] = t.reshape(-1)
    return flat[1:].view(t.shape)


@pytest.mark.parametrize("dtype,names", [("f32", None), ("f32", ["w_down"]), ("bf16", ["tok_emb"])])
def test_weights_off_the_16_byte_boundaries(dtype, names):
    """Element-aligned weights are read element by element: by the separate kernels in place of the one of a small fp32 model, by
    the embedding kernel alone for bf16.  fp32 as in test_small_forward; bf16 against the aligned table (sums in another
    order, see test_bf16_step_run_to_run_spread_is_bounded)."""
    cfg = wl.small_config(dtype=dtype, n_layers=2, n_heads=4, n_kv_heads=2, head_dim=64, d_model=256, d_ffn=512, vocab=512, prompt_len=30)
    c = 7
    w = wl.make_weights(cfg)
    off = dict(w)
    for n in names or [k for k in w if k != "bias_perm"]:
        off[n] = [_shifted(t) for t in w[n]] if isinstance(w[n], list) else _shifted(w[n])
    ids, lens = wl.make_prompts(cfg, batch=1)
    got = []
    for weights in (w, off):
        dec = engine.Decoder(cfg, weights, 1, c, 64)
        dec.fc_prefill(ids.numpy(), lens.numpy(), c)
        logits = dec.fc_debug_logits(True)
        step = dec.fc_jacobi_step()
        got.append((logits.cpu().numpy(), step))
        if dtype == "f32":
            assert dec.fc_last_launch_count() == (1 if weights is w else 6 * cfg.n_layers + 3)
    o = oracle.Oracle(cfg, w, 64)
    o.prefill(ids[0].numpy(), c)
    k, acc, wnew, ref = o.jacobi_step(want_logits=True)
    lg, (cnt, tok, win) = got[1]
    if dtype == "f32":
        assert np.abs(lg - ref).max() < 2e-4
        assert cnt[0] == k and tok[0, :k].tolist() == acc.tolist() and win[0].tolist() == wnew.tolist()
    else:
        assert np.abs(lg - got[0][0]).max() < 3e-4
    o.close()


def test_small_model_over_a_long_cache_takes_the_separate_kernels():
    """16 heads over 1631 keys: with 64 rows (and the later blocks of the prompts) beyond the line of small_forward_pays, with 2
    rows of the same context below it."""
    hq, c, lens = 16, 32, [1600, 700]
    cfg = wl.small_config(dtype="f32", n_layers=2, n_heads=hq, n_kv_heads=4, head_dim=32, d_model=128, d_ffn=256, vocab=300,
                          prompt_len=max(lens), bias_beta=4.0, seed=733)
    w = wl.make_weights(cfg)
    ids, _ = wl.make_prompts(cfg, batch=2, lens=lens)
    dec = engine.Decoder(cfg, w, 2, c, max(lens) + 3 * c)
    dec.fc_prefill(ids.numpy(), lens, c)
    logits = dec.fc_debug_logits(True)
    orc = []
    for b, P in enumerate(lens):
        orc.append(oracle.Oracle(cfg, w, max(lens) + 3 * c))
        orc[b].prefill(ids[b, :P].numpy(), c)
    for width, launches in ((c, 6 * cfg.n_layers + 3), (1, 1), (c, 6 * cfg.n_layers + 3)):
        dec.fc_set_window(width)
        cnt, tok, win = dec.fc_jacobi_step()
        assert dec.fc_last_launch_count() == launches
        lg = logits[:2 * width].cpu().numpy().reshape(2, width, cfg.vocab)
        for b in range(2):
            orc[b].set_window(width)
            k, acc, wnew, ref = orc[b].jacobi_step(want_logits=True)
            assert np.abs(lg[b] - ref).max() < 2e-4
            assert cnt[b] == k and tok[b, :k].tolist() == acc.tolist() and win[b].tolist() == wnew.tolist()
    for o in orc:
        o.close()
    assert dec.fc_debug_check_guards() == 0
