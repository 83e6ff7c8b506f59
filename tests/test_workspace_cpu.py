"""What heads and training calls ask for in device memory (no GPU needed): a head that is told to draft few positions reserves nothing
for long drafts, and scratch for cut GEMM tiles is reserved by what the shapes can use."""
import ctypes

import pytest

from paper_2511_11346_b200 import binding as B

MB = 1e6


def config(**kw):
    base = dict(family=B.MTPC_CP, n=8, r=16, v=320, d=4096, io_dtype=B.MTPC_BF16, max_positions=8192, max_windows_per_pos=1, flags=0,
                v_valid=0)
    base.update(kw)
    return B.MtpcConfig(*[base[f] for f, _ in B.MtpcConfig._fields_])


def size(call, *args):
    out = ctypes.c_size_t(0)
    code = getattr(B.lib(), call)(*args, ctypes.byref(out))
    return code, out.value


def head(cfg):
    return size("mtpc_workspace_bytes", ctypes.byref(cfg))


@pytest.mark.parametrize("kw,sums", [
    (dict(), 1), (dict(family=B.MTPC_HMM, n=16, r=32), 1), (dict(family=B.MTPC_BTREE, n=16, r=32, v=256, d=3072, max_positions=4096), 449),
    (dict(family=B.MTPC_HMM, r=32, flags=B.MTPC_FLAG_HMM_CONTEXTUAL), 225), (dict(max_windows_per_pos=64), 1),
])
def test_a_head_of_short_drafts_reserves_no_long_ones(kw, sums):
    full, short = config(**kw), config(**{**kw, "flags": kw.get("flags", 0) | B.MTPC_FLAG_SHORT_DRAFTS})
    (code, all_bytes), (code2, few_bytes) = head(full), head(short)
    assert code == 0 and code2 == 0
    c = short
    rows = max(c.max_positions, 128 * c.max_windows_per_pos)
    # evidence and messages per window, log omega, hidden states and targets of a host call, prefixes and loss terms; 128 positions' logits
    want = (8.0 * rows * c.n * c.r + 4.0 * c.max_positions * sums * c.r + 2.0 * c.max_positions * c.d + 24.0 * rows * c.n +
            4.0 * 128 * c.n * c.r * (c.v + 1))
    assert few_bytes <= 1.02 * want + MB
    assert all_bytes > few_bytes + 0.4 * min(4.0 * c.max_positions * c.n * c.r * c.v, 2.0 ** 32)


def test_heads_of_few_positions_need_no_flag():
    for wpp in (1, 16):
        plain, short = config(max_positions=128, max_windows_per_pos=wpp), config(max_positions=128, max_windows_per_pos=wpp, flags=4)
        assert head(plain) == head(short)


@pytest.mark.parametrize("kw", [dict(flags=8), dict(flags=2), dict(flags=5), dict(flags=6)])
def test_other_flags_are_refused(kw):
    assert head(config(**kw))[0] == -3


def test_scratch_of_cut_tiles_goes_by_the_shape():
    code, small = size("mtpc_lowrank_workspace_bytes", ctypes.byref(config(max_positions=8, max_windows_per_pos=4)), 16)
    assert code == 0 and small <= 20 * MB                  # 80 parts of 128 KB is what eight positions can use
    few = config(n=4, r=8, v=64, d=256, max_positions=64)
    code, train = size("mtpc_backward_workspace_bytes", ctypes.byref(few), 40)
    assert code == 0 and train <= 3 * MB
    code, train = size("mtpc_backward_workspace_bytes", ctypes.byref(config()), 2048)
    assert code == 0 and train <= 2048 * 40960 * 6 * 1.01 + 60 * MB


def test_the_size_of_a_head_for_very_many_positions_is_found_at_once():
    import time
    start = time.perf_counter()
    for positions in (1 << 30, (1 << 31) - 1):
        code, _ = size("mtpc_lowrank_workspace_bytes", ctypes.byref(config(n=1, r=1, v=16, d=4096, max_positions=positions)), 16)
        assert code == 0
    assert time.perf_counter() - start < 0.2
    # the tiles of a last round repeat every 148 row tiles, so beyond that only the buffers per position grow
    step = 148 * 128
    a, b, c = (size("mtpc_lowrank_workspace_bytes", ctypes.byref(config(max_positions=k * step, flags=B.MTPC_FLAG_SHORT_DRAFTS)), 16)[1] for k in (1, 2, 3))
    assert c - b == b - a
