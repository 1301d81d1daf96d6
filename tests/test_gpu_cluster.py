"""The projections with one writer per output (up to 64 rows), reached through Jacobi steps, against the oracle: widths 16, 32 and
64 at their edges, fewer weight units than clusters, column ranges of several tiles, a k range shorter than the cluster's shares,
cached lengths around the key tiles, grouped queries, both head sizes.  Bars and margin rule as in test_gpu_full_configs.  Nothing
in this route is added up in the order of arrival: a step repeated gives the same bits (the other tensor-core routes' steps
differ in their last bits)."""
import numpy as np
import pytest

from paper_2311_08263_b200 import lib as _l, workload as wl
from test_gpu_full_configs import _random_kv_case

pytestmark = pytest.mark.gpu

CASES = [
    # hq, hkv, hd, d, f, vocab, c, lens
    (2, 1, 64, 128, 128, 528, 1, [0]),                             # one pair of k-blocks for four shares; one row, no cached key
    (2, 2, 64, 256, 4480, 9600, 16, [33]),                         # two column ranges of gate and up, three of the LM head
    (8, 2, 128, 640, 1408, 1040, 1, [700, 31, 0, 1, 32, 95]),      # six rows of a width of 16, grouped queries
    (4, 4, 128, 512, 9088, 1024, 17, [640]),                       # 17 rows: a width of 32; three ranges, cut in front of the last
    (10, 5, 64, 640, 896, 4240, 8, [64, 63, 65, 300]),             # 32 rows
    (2, 2, 128, 256, 4480, 4240, 33, [96]),                        # 33 rows: a width of 64, windows over three 16-key blocks
    (6, 3, 64, 384, 4480, 9600, 16, [5, 160, 0, 31]),              # 64 rows, passes of two tiles
    (2, 1, 64, 128, 256, 528, 64, [40]),                           # a window of 64 rows of one sequence
    (32, 32, 128, 256, 512, 1040, 16, [1471]),                     # 32 units, four key splits, rings that wrap
    (32, 32, 128, 256, 512, 1040, 8, [700, 33]),                   # 64 units, four key splits of half the ring
    (40, 40, 128, 256, 512, 1040, 16, [1300, 64]),                 # 80 units, three key splits of half the ring
    (24, 24, 128, 256, 512, 1040, 12, [1300, 64, 5, 900]),         # 96 units, no split
    (32, 4, 64, 256, 512, 1040, 16, [2500]),                       # head_dim 64, eight key splits
    (16, 16, 128, 256, 512, 1040, 1, [2300] + [31 + 61 * i for i in range(15)]),       # 256 units x 36 tiles: the streaming pair
    (32, 4, 64, 256, 512, 1040, 16, [2200, 5, 64, 300]),           # head_dim 64: 128 units x 35 tiles, short
    (32, 4, 64, 256, 512, 1040, 16, [2290, 5, 64, 300]),           # 128 x 37: the streaming pair
    (40, 40, 128, 256, 512, 1040, 16, [2300, 5, 64, 300]),         # more units than SMs: 160 x 37, short
    (40, 40, 128, 256, 512, 1040, 16, [2420, 5, 64, 300]),         # 160 x 39: the streaming pair
    (20, 20, 128, 256, 512, 1040, 16, [900]),                      # 20 units: six key splits
    (8, 4, 64, 256, 512, 1040, 64, [1300]),                        # 64 rows of one sequence, 32 units, ring halves
    (12, 12, 128, 256, 512, 1040, 13, [1300, 64, 5, 900]),         # 48 units: five key splits of half the ring
    (32, 32, 128, 256, 512, 1040, 4, [1100, 0, 1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 191, 192, 193, 1023]),     # 64 rows, 512 x 18: the same
]


@pytest.mark.parametrize("hq,hkv,hd,d,f,vocab,c,lens", CASES)
def test_step_against_the_oracle_and_again(hq, hkv, hd, d, f, vocab, c, lens):
    cfg = wl.small_config(n_layers=2, n_heads=hq, n_kv_heads=hkv, head_dim=hd, d_model=d, d_ffn=f, vocab=vocab, seed=2000 + c + hd)
    dec, _ = _random_kv_case(cfg, lens, c, range(len(lens)))
    assert dec.fc_last_route() & _l.FC_ROUTE_MASK == _l.FC_ROUTE_ONE_WRITER
    units, tiles = len(lens) * hkv * ((hq // hkv * c + 15) // 16), (max(lens) + c + 63) // 64
    stream = units * tiles >= (4600 if hd == 64 else 6000 if units > 148 else 8600)
    assert dec.fc_last_route() & _l.FC_ATTN_MASK == (_l.FC_ATTN_STREAM if stream else _l.FC_ATTN_SHORT)
    assert dec.fc_last_launch_count() == (3 if stream else 2) * cfg.n_layers + 4
    logits = dec.fc_debug_logits(True)
    pending = wl.make_random_window(cfg, len(lens), 1, salt=3).numpy()[:, 0]
    window = wl.make_random_window(cfg, len(lens), c, salt=4).numpy()
    window[:, 0] = pending
    seen = []
    for _ in range(3):
        dec.fc_debug_set_state(lens, pending, c, pad_id=0)
        logits.zero_()
        dec.fc_jacobi_step(window)
        seen.append(logits[:len(lens) * c].cpu().numpy().copy())
    assert np.array_equal(seen[0], seen[1]) and np.array_equal(seen[0], seen[2])
    assert dec.fc_debug_check_guards() == 0


@pytest.mark.parametrize("b,c,length", [(16, 1, 500), (1, 16, 800), (2, 16, 300), (1, 24, 300), (1, 33, 500), (4, 16, 300), (16, 1, 2048)])
def test_wide_steps_repeat_bit_for_bit(b, c, length):
    """Two layers of the 7B shape, fifty times the same step: exchange buffers that are written again before they are read, or
    read before they are written, show as rows that differ."""
    import dataclasses
    import torch
    from paper_2311_08263_b200 import engine
    cfg = dataclasses.replace(wl.CONFIGS["7b"], n_layers=2)
    w = wl.make_weights(cfg, device="cuda")
    dec = engine.Decoder(cfg, w, b, c, length + c + 8)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    dec.kv_view().normal_(generator=gen)
    window = wl.make_random_window(cfg, b, c, salt=4).numpy()
    lens = [length - 31 * i % length for i in range(b)]
    logits = dec.fc_debug_logits(True)
    first = None
    for _ in range(50):
        dec.fc_debug_set_state(lens, window[:, 0], c, pad_id=0)
        dec.fc_jacobi_step(window)
        got = logits[:b * c].clone()
        first = got if first is None else first
        assert torch.equal(got, first)


def test_rows_where_the_route_changes():
    """Two layers as wide as 13B: 9 and 32 rows take these projections, 8 and 33 the chained launch.  A row's logits depend on the rows in front of it
    only, so the shorter window's rows are the longer one's first."""
    import dataclasses
    import torch
    from paper_2311_08263_b200 import engine
    cfg = dataclasses.replace(wl.CONFIGS["13b"], n_layers=2, vocab=2048)
    w = wl.make_weights(cfg, device="cuda")
    window = wl.make_random_window(cfg, 1, 33, salt=4).numpy()
    got = {}
    for c in (8, 9, 32, 33):
        dec = engine.Decoder(cfg, w, 1, c, 300)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(5)
        dec.kv_view().normal_(generator=gen)
        dec.fc_debug_set_state([200], window[:, 0], c, pad_id=0)
        logits = dec.fc_debug_logits(True)
        dec.fc_jacobi_step(window[:, :c].copy())
        got[c] = logits[:c].float().cpu().clone()
        assert dec.fc_last_route() & _l.FC_ROUTE_MASK == (_l.FC_ROUTE_ONE_WRITER if 9 <= c <= 32 else _l.FC_ROUTE_CHAIN)
        assert dec.fc_debug_check_guards() == 0
    for c in (8, 9, 32):
        assert float((got[c] - got[33][:c]).abs().max()) < 3e-2 * float(got[33].pow(2).mean().sqrt())


def test_second_model_in_the_buffers_of_the_first():
    """fc_init on the K/V slab and workspace that another context's projections ran from, with weights elsewhere: the step is
    that of the second model bit for bit, as in buffers of its own."""
    import ctypes as C
    import dataclasses
    import torch
    from paper_2311_08263_b200 import engine
    cfg = wl.small_config(n_layers=3, n_heads=8, n_kv_heads=8, head_dim=64, d_model=512, d_ffn=1536, vocab=1024, seed=61)
    first, second = (wl.make_weights(c, device="cuda") for c in (cfg, dataclasses.replace(cfg, seed=62)))
    B, c, lens = 2, 16, [70, 33]
    window = wl.make_random_window(cfg, B, c, salt=4).numpy()

    def step(dec):
        dec.kv_view().normal_(generator=torch.Generator(device="cuda").manual_seed(5))
        dec.fc_debug_set_state(lens, window[:, 0], c)
        logits = dec.fc_debug_logits(True)
        dec.fc_jacobi_step(window)
        return logits.cpu().numpy().copy()

    want = step(engine.Decoder(cfg, second, B, c, 100))
    dec = engine.Decoder(cfg, first, B, c, 100)
    other = step(dec)
    donor = engine.Decoder(cfg, second, B, c, 100)
    dec.close()
    h = C.c_void_p()
    assert dec.lib.fc_init(C.byref(h), C.byref(dec.shape), C.byref(donor.weights), dec.kv.data_ptr(), dec._kv_bytes,
                           dec.ws.data_ptr(), dec._ws_bytes, dec.stream.cuda_stream) == _l.FC_OK
    dec.h = h
    got = step(dec)
    assert np.array_equal(got, want) and not np.array_equal(got, other)
    assert dec.fc_debug_check_guards() == 0


@pytest.mark.parametrize("c", [16, 24, 50])
def test_wait_that_runs_out_is_reported_and_the_next_prompt_is_as_before(c):
    """A grid barrier that one arrival is missing from (widths 16, 32, 64): the waits of every CTA run out, the exchange and the copies
    on their way are waited for, the step reports it.  The buffers and the context are as good as new."""
    from paper_2311_08263_b200 import engine
    cfg = wl.small_config(n_layers=2, n_heads=8, n_kv_heads=8, head_dim=64, d_model=512, d_ffn=4608, vocab=1024, prompt_len=60, seed=71)
    ids = wl.make_prompts(cfg)[0][0].numpy()
    dec = engine.Decoder(cfg, wl.make_weights(cfg, device="cuda"), 1, c, 60 + 4 * c)
    logits = dec.fc_debug_logits(True)
    dec.fc_prefill(ids, [60], c)
    want = dec.fc_jacobi_step()
    first = logits.clone()
    dec.fc_debug_withhold_arrival()
    with pytest.raises(engine.FcError) as e:
        dec.fc_jacobi_step()
    assert e.value.code == _l.FC_ERR_DEVICE_TIMEOUT
    assert dec.fc_debug_check_guards() == 0
    dec.fc_prefill(ids, [60], c)
    got = dec.fc_jacobi_step()
    assert all(np.array_equal(a, b) for a, b in zip(got, want)) and bool((logits == first).all())
    assert dec.fc_debug_check_guards() == 0
