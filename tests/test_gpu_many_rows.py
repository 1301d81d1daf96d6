"""Forwards of many rows (one dense GEMM per projection), against the oracle: prompts packed into blocks that cut through
sequences, steps whose rows end inside a row tile, grouped queries, both head sizes.  Bars and margin rule as in
test_gpu_full_configs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2311_08263_b200 import engine, lib as _l, workload as wl
from test_gpu_full_configs import _check_step, _random_kv_case

pytestmark = pytest.mark.gpu


def _cfg(hq, hkv, hd, d_ffn=768, **kw):
    return wl.small_config(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_model=512, d_ffn=d_ffn, vocab=1024, **kw)


STEPS = [
    # hq, hkv, hd, d_ffn, c, lens: rows = c x sequences
    (8, 4, 64, 768, 43, [0, 33, 70]),                      # 129 rows: one more than the chained launch takes
    (4, 4, 128, 512, 20, [100, 0, 1, 31, 32, 33, 64, 95]),  # 160
    (8, 8, 64, 1280, 61, [40, 0, 7, 64, 129]),              # 305: a ragged third row tile
    (4, 2, 128, 256, 64, [5, 200, 64, 0, 17, 90, 128, 33]),  # 512: one tile of weights in the feed-forward block
]


@pytest.mark.parametrize("hq,hkv,hd,d_ffn,c,lens", STEPS)
def test_many_row_step(hq, hkv, hd, d_ffn, c, lens):
    cfg = _cfg(hq, hkv, hd, d_ffn, seed=300 + c)
    dec, _ = _random_kv_case(cfg, lens, c, range(len(lens)))
    assert dec.fc_last_launch_count() == 8 * cfg.n_layers + 4


PROMPTS = [
    (8, 4, 64, [130]),                                      # 129 rows of one sequence
    (8, 2, 128, [1, 2, 130, 300, 65, 64, 33, 1]),           # empty and one-row segments between longer ones
    (4, 4, 64, [700, 517, 300, 41]),                        # 1554 rows: two blocks, the cut inside the second prompt
]


@pytest.mark.parametrize("hq,hkv,hd,lens", PROMPTS)
def test_packed_prompts(hq, hkv, hd, lens):
    cfg = _cfg(hq, hkv, hd, seed=500 + len(lens), prompt_len=max(lens))
    c, B = 4, len(lens)
    w = wl.make_weights(cfg)
    ids, _ = wl.make_prompts(cfg, batch=B, lens=lens)
    dec = engine.Decoder(cfg, w, B, c, max(lens) + 2 * c)
    dec.fc_prefill(ids.numpy(), lens, c)
    kv = dec.kv_view().float().cpu().numpy()
    logits = dec.fc_debug_logits(True)
    cnt, tok, win = dec.fc_jacobi_step()
    lg = logits.cpu().numpy().reshape(B, c, cfg.vocab)
    for b, P in enumerate(lens):
        o = oracle.Oracle(cfg, w, max(lens) + 2 * c)
        o.prefill(ids[b, :P].numpy(), c)
        window = np.array([ids[b, P - 1]] + [ids[b, (j - 1) % P] for j in range(1, c)], np.int32)
        k_ref, acc_ref, win_ref, lg_ref = o.jacobi_step(want_logits=True)
        _check_step(lg[b], lg_ref, window, cnt[b], tok[b], win[b], k_ref, acc_ref, win_ref)
        if P > 1:
            # layer 0 has no attention in front of it: fp32 sums in another order, so a stored value is at most one bf16
            # step (2^-8 of its size, 2^-7 above a power of two) away, and nearly all are the same
            for half, ref in enumerate(o.get_kv(0, P - 1)):
                got = kv[0, half, b, :, :P - 1].transpose(1, 0, 2).reshape(P - 1, -1)
                assert np.all(np.abs(got - ref) <= 2.0 ** -7 * np.abs(ref) + 1e-6)
                assert np.mean(got != ref) < 0.01
        o.close()
    assert dec.fc_debug_check_guards() == 0


def test_step_that_stores_many_values_adds_up_as_the_chained_launch():
    """The same step of 512 rows (1.34e8 stored values) through the dense GEMMs and through the chained launch: layer 0's new K/V rows
    come from the same embedding rows, so they differ only where an fp32 sum lies so near a bf16 rounding boundary that the
    order of its few additions decides: some 2^-24 roundings against steps of 2^-8, 3 to 6 in 100000.  Sums over other runs
    of k-blocks add the tensor core's own rounding: 7.0e-4 with six k-blocks per accumulator.  The logits behind 32 layers (the
    down projection's 44 k-blocks end inside a chunk) differ by the few values that fall apart on the way: 1.5e-4 measured
    on such shapes, a tile or a piece gone wrong is of order one."""
    B, c = 16, 32
    cfg = wl.small_config(n_layers=32, n_heads=32, n_kv_heads=32, head_dim=128, d_model=2048, d_ffn=2816, vocab=1024, seed=811)
    w = wl.make_weights(cfg, device="cuda")
    window = wl.make_random_window(cfg, B, c).numpy()
    lens = [40 + 3 * b for b in range(B)]
    rows, logits = [], []
    for flags in (0, _l.FC_FLAG_NO_CTA_PAIRS):
        dec = engine.Decoder(cfg, w, B, c, max(lens) + c, flags=flags)
        logits.append(dec.fc_debug_logits(True))
        kv = dec.kv_view()
        kv.normal_(generator=torch.Generator(device="cuda").manual_seed(5))
        dec.fc_debug_set_state(lens, window[:, 0], c)
        dec.fc_jacobi_step(window)
        assert (dec.fc_last_launch_count() == 8 * cfg.n_layers + 4) == (flags == 0)
        rows.append(torch.stack([kv[0, :, b, :, lens[b]:lens[b] + c] for b in range(B)]).float())
        assert dec.fc_debug_check_guards() == 0
    assert float((rows[0] != rows[1]).float().mean()) < 2e-4
    assert float((logits[0] - logits[1]).norm() / logits[1].norm()) < 1e-3


@pytest.mark.parametrize("batch,c,short,last", [(17, 64, 69, 65), (33, 32, 36, 33)])
def test_packed_prompts_when_the_step_capacity_is_no_whole_tile(batch, c, short, last):
    """17 x 64 = 1088 and 33 x 32 = 1056 rows of a step, prompts of 1152 ids in one block: its last rows are beyond what a step
    uses.  The sequences that hold them, and the first, against the oracle."""
    cfg = _cfg(8, 8, 64, seed=900 + c, prompt_len=short)
    lens = [short] * (batch - 1) + [last]
    assert sum(lens) - batch == 1152
    w = wl.make_weights(cfg)
    ids, _ = wl.make_prompts(cfg, batch=batch, lens=lens)
    max_seq = short + 2 * c
    dec = engine.Decoder(cfg, w, batch, c, max_seq)
    dec.fc_prefill(ids.numpy(), lens, c)
    kv = dec.kv_view().float().cpu().numpy()
    logits = dec.fc_debug_logits(True)
    cnt, tok, win = dec.fc_jacobi_step()
    lg = logits.cpu().numpy().reshape(batch, c, cfg.vocab)
    for b in (0, batch - 3, batch - 2, batch - 1):
        P = lens[b]
        o = oracle.Oracle(cfg, w, max_seq)
        o.prefill(ids[b, :P].numpy(), c)
        window = np.array([ids[b, P - 1]] + [ids[b, (j - 1) % P] for j in range(1, c)], np.int32)
        k_ref, acc_ref, win_ref, lg_ref = o.jacobi_step(want_logits=True)
        _check_step(lg[b], lg_ref, window, cnt[b], tok[b], win[b], k_ref, acc_ref, win_ref)
        for layer in range(cfg.n_layers):
            for half, ref in enumerate(o.get_kv(layer, P - 1)):
                got = kv[layer, half, b, :, :P - 1].transpose(1, 0, 2).reshape(P - 1, -1)
                # bf16 steps (2^-8) here and there; layer 1 has one attention over such values in front of it
                assert np.linalg.norm(got - ref) < 2.0 ** -8 * np.linalg.norm(ref)
        o.close()
    assert dec.fc_debug_check_guards() == 0


COMPACTED = [
    # route, hq, hkv, hd, vocab, c, lens; sequences 0, 5 and 9 have the same prompt and end at the first iteration
    ("dense", 8, 4, 64, 1024, 16, [60, 33, 70, 1, 64, 60, 20, 95, 31, 60, 47, 80]),              # 192 rows, then 144
    ("dense", 4, 4, 128, 1024, 40, [30, 33, 70, 2, 64, 30, 20, 95, 31, 30, 47, 80]),             # 480, then 360
    ("stream", 8, 8, 64, 1000, 2, [40, 33, 960, 1, 64, 40, 20, 95, 31, 40, 47, 500]),            # 72 units x 16 tiles of 64 keys
    ("short", 4, 4, 128, 1008, 5, [40, 33, 300, 1, 64, 40, 20, 95, 31, 40, 47, 80]),             # 60 rows, then 45
    ("one-writer-stream", 16, 16, 64, 1008, 5, [40, 29, 2140, 1, 64, 40, 20, 95, 31, 40, 47, 80]),     # 144 units x 34 tiles
]


@pytest.mark.parametrize("route,hq,hkv,hd,vocab,c,lens", COMPACTED)
def test_finished_sequences_leave_the_rows_of_the_many_row_routes(route, hq, hkv, hd, vocab, c, lens):
    cfg = wl.small_config(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_model=512, d_ffn=768, vocab=vocab, prompt_len=max(lens),
                          seed=1200 + c)
    B, gone = len(lens), [0, 5, 9]
    w = wl.make_weights(cfg)
    ids = wl.make_prompts(cfg, batch=B, lens=lens)[0].numpy()
    ids[5], ids[9] = ids[0], ids[0]
    max_seq = max(lens) + 3 * c
    orc = []
    for b, P in enumerate(lens):
        orc.append(oracle.Oracle(cfg, w, max_seq))
        orc[b].prefill(ids[b, :P], c)
    eos = int(orc[0].generate(1)[0][0])
    orc[0].prefill(ids[0, :lens[0]], c)
    dec = engine.Decoder(cfg, w, B, c, max_seq)
    dec.fc_prefill(ids, lens, c)
    out, out_lens, _ = dec.fc_generate(2 * c, eos_id=eos, max_iters=1)
    logits = dec.fc_debug_logits(True)
    first = [o.generate(2 * c, eos_id=eos, max_iters=1)[0].tolist() for o in orc]
    assert [b for b in range(B) if eos in first[b]] == gone
    for b in range(B):
        assert out[b, :out_lens[b]].tolist() == first[b]
    cnt, tok, win = dec.fc_jacobi_step()
    assert dec.fc_last_launch_count() == {"dense": 8, "short": 2}.get(route, 3) * cfg.n_layers + 4 + 1      # and the gather of the windows
    assert dec.fc_last_route() == {"dense": _l.FC_ROUTE_DENSE | _l.FC_ATTN_STREAM, "stream": _l.FC_ROUTE_CHAIN | _l.FC_ATTN_STREAM,
                                   "short": _l.FC_ROUTE_ONE_WRITER | _l.FC_ATTN_SHORT,
                                   "one-writer-stream": _l.FC_ROUTE_ONE_WRITER | _l.FC_ATTN_STREAM}[route]
    lg = logits[:(B - len(gone)) * c].cpu().numpy().reshape(B - len(gone), c, vocab)
    live = [b for b in range(B) if b not in gone]
    for i, b in enumerate(live):
        k, acc, wnew, ref = orc[b].jacobi_step(want_logits=True)
        _check_step(lg[i], ref, np.zeros(c, np.int32), cnt[b], tok[b], win[b], k, acc, wnew)
    assert all(cnt[b] == 0 for b in gone)
    kl, _ = dec.fc_get_state()
    for b in live:
        assert kl[b] == orc[b].kv_len
    assert dec.fc_debug_check_guards() == 0
    for o in orc:
        o.close()


def test_more_prompts_than_segments_of_a_block():
    """70 prompts of 2 to 6 ids: 210 rows, but a block takes 64 segments at most."""
    cfg = _cfg(8, 8, 64, seed=1300, prompt_len=6)
    lens, c = [2 + (3 * b) % 5 for b in range(70)], 3
    w = wl.make_weights(cfg)
    ids = wl.make_prompts(cfg, batch=70, lens=lens)[0].numpy()
    dec = engine.Decoder(cfg, w, 70, c, 16)
    dec.fc_prefill(ids, lens, c)
    logits = dec.fc_debug_logits(True)
    cnt, tok, win = dec.fc_jacobi_step()
    lg = logits.cpu().numpy().reshape(70, c, cfg.vocab)
    for b in (0, 1, 62, 63, 64, 65, 69):
        o = oracle.Oracle(cfg, w, 16)
        o.prefill(ids[b, :lens[b]], c)
        k, acc, wnew, ref = o.jacobi_step(want_logits=True)
        _check_step(lg[b], ref, np.zeros(c, np.int32), cnt[b], tok[b], win[b], k, acc, wnew)
        o.close()
    assert dec.fc_debug_check_guards() == 0


def test_dense_and_chained_steps_after_a_reported_timeout():
    """Dense step that reports a timeout, prompts again, then a one-writer step (64 rows), a chained one (96) and a dense one (132) over
    the same buffers."""
    cfg = _cfg(8, 4, 64, seed=1400, prompt_len=60)
    B, c, lens = 4, 33, [60, 41, 3, 50]
    w = wl.make_weights(cfg)
    ids = wl.make_prompts(cfg, batch=B, lens=lens)[0].numpy()
    dec = engine.Decoder(cfg, w, B, c, 60 + 4 * c)
    dec.fc_prefill(ids, lens, c)
    dec.fc_debug_inject_timeout()
    with pytest.raises(engine.FcError) as e:
        dec.fc_jacobi_step()
    assert e.value.code == _l.FC_ERR_DEVICE_TIMEOUT
    dec.fc_prefill(ids, lens, c)
    logits = dec.fc_debug_logits(True)
    orc = []
    for b, P in enumerate(lens):
        orc.append(oracle.Oracle(cfg, w, 60 + 4 * c))
        orc[b].prefill(ids[b, :P], c)
    for width, per_layer, route in ((16, 2, _l.FC_ROUTE_ONE_WRITER), (24, 2, _l.FC_ROUTE_CHAIN), (c, 8, _l.FC_ROUTE_DENSE)):
        dec.fc_set_window(width)
        cnt, tok, win = dec.fc_jacobi_step()
        assert dec.fc_last_launch_count() == per_layer * cfg.n_layers + 4
        assert dec.fc_last_route() & _l.FC_ROUTE_MASK == route
        lg = logits[:B * width].cpu().numpy().reshape(B, width, cfg.vocab)
        for b in range(B):
            orc[b].set_window(width)
            k, acc, wnew, ref = orc[b].jacobi_step(want_logits=True)
            assert _check_step(lg[b], ref, np.zeros(width, np.int32), cnt[b], tok[b], win[b], k, acc, wnew)
    assert dec.fc_debug_check_guards() == 0
    for o in orc:
        o.close()
