"""The C ABI on a machine without a GPU: the library builds, loads, exports every function that
include/fastcot.h declares, and its host-only entry points (sizes, status strings, argument checks) behave."""
import ctypes as C
import os
import re

import pytest

from paper_2311_08263_b200 import build, lib

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "fastcot.h")


def _declared_functions():
    text = open(HEADER).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)          # comments mention names too
    names = set(re.findall(r"\b(fc_[a-z0-9_]+)\s*\(", text))
    assert len(names) >= 20
    return sorted(names)


@pytest.fixture(scope="module")
def cdll():
    path = build.build()
    return C.CDLL(path)


def test_library_exports_every_declared_function(cdll):
    missing = [n for n in _declared_functions() if not hasattr(cdll, n)]
    assert not missing, missing


def test_binding_names_match_the_header():
    l = lib.load()
    for n in _declared_functions():
        assert hasattr(l, n), n


def test_status_strings(cdll):
    cdll.fc_strerror.restype = C.c_char_p
    seen = set()
    for code in (lib.FC_OK, lib.FC_ERR_ARG, lib.FC_ERR_SHAPE, lib.FC_ERR_CAPACITY, lib.FC_ERR_TOKEN_RANGE, lib.FC_ERR_STATE,
                 lib.FC_ERR_BAD_WINDOW, lib.FC_ERR_DEVICE_TIMEOUT, lib.FC_ERR_CUDA):
        s = cdll.fc_strerror(code)
        assert s and s not in seen
        seen.add(s)
    assert cdll.fc_strerror(-12345) == b"unknown status"


def _shape(**kw):
    s = lib.fc_model_shape()
    vals = dict(n_layers=2, d_model=128, n_heads=4, n_kv_heads=4, head_dim=32, d_ffn=512, vocab=512, dtype=lib.FC_F32,
                rms_eps=1e-5, rope_theta=1e4, max_batch=1, max_c=8, max_seq=64, bias_beta=0.0, flags=0)
    vals.update(kw)
    for k, v in vals.items():
        setattr(s, k, v)
    return s


def test_sizes_are_host_arithmetic(cdll):
    cdll.fc_kv_bytes.restype = C.c_size_t
    cdll.fc_workspace_bytes.restype = C.c_size_t
    s = _shape()
    # [layer][K|V][batch][kv_head][max_seq][head_dim] fp32
    assert cdll.fc_kv_bytes(C.byref(s)) == 2 * 2 * 1 * 4 * 64 * 32 * 4
    assert cdll.fc_kv_bytes(C.byref(_shape(dtype=lib.FC_BF16))) == 2 * 2 * 1 * 4 * 64 * 32 * 2
    ws = cdll.fc_workspace_bytes(C.byref(s))
    assert ws > 0 and ws % 256 == 0
    assert cdll.fc_workspace_bytes(C.byref(_shape(max_batch=4))) > ws
    # shapes the library refuses report size 0
    for bad in (dict(head_dim=48), dict(n_heads=3, n_kv_heads=2), dict(max_c=65), dict(d_model=100), dict(dtype=7),
                dict(max_seq=8)):
        assert cdll.fc_kv_bytes(C.byref(_shape(**bad))) == 0
        assert cdll.fc_workspace_bytes(C.byref(_shape(**bad))) == 0


def test_init_rejects_bad_arguments_before_touching_the_device(cdll):
    ctx = C.c_void_p()
    s = _shape()
    w = lib.fc_weights()
    assert cdll.fc_init(C.byref(ctx), None, C.byref(w), None, 0, None, 0, None) == lib.FC_ERR_ARG
    assert cdll.fc_init(C.byref(ctx), C.byref(s), C.byref(w), None, 0, None, 0, None) == lib.FC_ERR_ARG
    assert ctx.value is None
    cdll.fc_destroy(None)                                          # destroying nothing is allowed
    cdll.fc_last_launch_count.restype = C.c_int64
    assert cdll.fc_last_launch_count(None) == 0


@pytest.mark.parametrize("rows", [(17, 64), (33, 32), (40, 30), (21, 50)])
def test_workspace_of_the_dense_route_holds_whole_row_tiles(cdll, rows):
    """Blocks of prompts are whole 128-row tiles up to the capacity, so a capacity that is no multiple of 128 needs the
    activation buffers of the next one: what one more row costs is then no row of the residual and the QKV buffer."""
    cdll.fc_workspace_bytes.restype = C.c_size_t
    batch, c = rows
    full = (batch * c + 127) // 128 * 128
    bulk = dict(dtype=lib.FC_BF16, d_model=512, n_heads=8, n_kv_heads=8, head_dim=64, d_ffn=512, vocab=1024, max_c=1, max_seq=80)
    got = [cdll.fc_workspace_bytes(C.byref(_shape(**bulk, max_batch=n))) for n in (batch * c, full)]
    # per sequence and row of the step: window, accepted tokens, argmax, state words, the prompt and the output ids
    per_seq = 4 * 12 + 2 * 4 * 80 + 4 * bulk["n_kv_heads"] + 16 * 64 * 4 * bulk["n_kv_heads"]      # and a query tile per kv head
    slack = 256 * 16
    assert got[0] <= got[1] <= got[0] + (full - batch * c) * per_seq + slack
    row = 4 * (512 + 3 * 512)
    assert (full - batch * c) * row > slack


def test_workspace_holds_no_tensor_maps(cdll):
    """A kernel that takes a tensor map from memory that was copied to needs a proxy fence in front; maps go by value in the
    launch's parameters.  What a layer adds to the workspace are its synchronisation words, a few hundred bytes."""
    cdll.fc_workspace_bytes.restype = C.c_size_t
    shape = dict(dtype=lib.FC_BF16, d_model=512, n_heads=8, n_kv_heads=8, head_dim=64, d_ffn=1536, vocab=1024, max_c=16, max_seq=80)
    few, many = (cdll.fc_workspace_bytes(C.byref(_shape(**shape, n_layers=n))) for n in (8, 40))
    assert many - few < 32 * 512 + 1024


def test_workspace_without_the_operands_of_a_route_that_the_vocabulary_is_too_large_for(cdll):
    """Two million ids are beyond what the one-writer projections' tile arithmetic is exact for: as with a vocabulary that is no multiple
    of 16, no operands for them."""
    cdll.fc_workspace_bytes.restype = C.c_size_t
    shape = dict(dtype=lib.FC_BF16, d_model=512, n_heads=8, n_kv_heads=8, head_dim=64, d_ffn=1536, max_c=16, max_seq=80)
    large, ragged, small = (cdll.fc_workspace_bytes(C.byref(_shape(**shape, vocab=n))) for n in (2000000, 2000001, 32016))
    assert large == ragged < small
