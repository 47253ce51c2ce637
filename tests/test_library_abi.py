"""The C-ABI library builds, loads without a GPU and exports every symbol include/efq.h declares."""
import ctypes
import os
import re
import subprocess
import threading
import time

import pytest
import torch

from paper_2609_09721_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "efq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(efq_\w+|exp_then_quantize_\w+)\s*\(", text)))


def test_header_symbols_are_exported():
    lib = ctypes.CDLL(build.build())
    names = _declared_symbols()
    assert "efq_probgen" in names and "efq_attention_fwd" in names and "exp_then_quantize_attention_fwd" in names
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTS) == names


def test_no_read_only_loads_of_what_the_kernel_before_writes():
    """Blocks of an overlapped launch may be there while the kernel before still writes, so its data are not read through the read-only
    path.  The tables of a packed batch are: a copy from the host writes them, and a copy overlaps no kernel."""
    tables = ("groups[mid].first_item", "first_cta + ", "places + ")
    for name in os.listdir(build.CSRC):
        for line in open(os.path.join(build.CSRC, name)):
            if "__ldg(" in line:
                assert name == "quantize_qkv.cu" and any(t in line for t in tables), (name, line)


def test_status_strings_and_version():
    assert binding.version().startswith("efq-b200")
    assert binding.status_string(0) == "ok"
    assert "timed out" in binding.status_string(7)
    assert len({binding.status_string(i) for i in range(8)}) == 8


def test_host_side_validation_needs_no_gpu():
    L = binding.lib()
    # negative sizes and null pointers are rejected before any CUDA call
    assert L.efq_probgen(None, 0, None, -1, 4, 1.0, None, None, None, None) == 1
    assert L.efq_probgen(None, 0, None, 0, 0, 1.0, None, None, None, None) == 0      # empty problem is a no-op
    assert L.efq_probgen(None, 64, None, 4, 64, 1.0, None, None, None, None) == 1
    p = binding.EfqParams(-3.06, -1.0, 0, 0)
    assert L.efq_probgen(16, 64, 16, 4, 64, 1.0, ctypes.byref(p), 16, 16, None) == 1   # h <= 0
    p = binding.EfqParams(-3.06, 2.3, 0, 0)
    assert L.efq_probgen(16, 32, 16, 4, 64, 1.0, ctypes.byref(p), 16, 16, None) == 1   # ld < cols
    assert L.efq_probgen(20, 64, 16, 4, 64, 1.0, ctypes.byref(p), 16, 16, None) == 3   # misaligned scores
    assert L.efq_probgen(16, 66, 16, 4, 64, 1.0, ctypes.byref(p), 16, 16, None) == 3   # ld % 4 != 0
    assert L.exp_then_quantize_probgen(16, 64, 16, 4, 64, 1.0, 5, 16, 16, None) == 1   # bad scale_mode
    assert L.exp_then_quantize_probgen(16, 64, 16, 4, 64, 1.0, -1, 16, 16, None) == 1


def _varlen_bytes(cu_q, cu_k, Hq, Hkv, d=128):
    n = len(cu_q) - 1
    cq = (ctypes.c_int64 * len(cu_q))(*cu_q)
    ck = (ctypes.c_int64 * len(cu_k))(*cu_k)
    return int(binding.lib().efq_attention_varlen_workspace_bytes(cq, ck, n, Hq, Hkv, d))


def test_workspace_planning_is_host_logic():
    """Sizes of the workspaces follow from the shapes alone (no GPU): the MXFP4 copies take about 0.53 B per
    element, a packed batch needs room for all of its sequences side by side, a decode step packs the query heads
    of a KV group into one tile, and bad prefix sums are refused."""
    one = binding.efq_attention_workspace_bytes(1, 8, 2, 1000, 3000, 128)
    # Q codes + scales of 8 heads x 1024 padded rows, K and V of 2 heads x 3072 padded keys: (64 + 4) B per row
    assert one >= 8 * 1024 * 68 + 2 * 2 * 3072 * 68 and one < 1.2 * (8 * 1024 * 68 + 2 * 2 * 3072 * 68) + 8192
    assert binding.efq_attention_workspace_bytes(1, 8, 3, 128, 128, 128) == 0          # Hq % Hkv != 0
    assert binding.efq_attention_workspace_bytes(1, 8, 2, 128, 128, 64) == 0           # d != 128
    two = _varlen_bytes([0, 1000, 2000], [0, 3000, 6000], 8, 2)
    assert two >= 2 * (one - 8192) and two < 2.2 * one                                # both sequences resident
    with_empty = _varlen_bytes([0, 1000, 1000, 2000], [0, 3000, 3500, 6500], 8, 2)    # a sequence without queries adds nothing
    assert abs(with_empty - two) < 4096
    decode = _varlen_bytes(list(range(65)), [512 * i for i in range(65)], 8, 2)        # 64 sequences, one query token each
    unpacked_q = 64 * 8 * 128 * 68                                                     # one padded tile per query head
    packed_q = 64 * 2 * 128 * 68                                                       # one per KV head
    kv = 64 * 2 * 2 * 512 * 68
    assert decode < kv + packed_q + (unpacked_q - packed_q) // 2 and decode > kv + packed_q
    assert _varlen_bytes([1, 5], [0, 5], 8, 2) == 0                                    # prefix sums must start at 0
    assert _varlen_bytes([0, 5, 3], [0, 5, 9], 8, 2) == 0                              # and never decrease
    assert _varlen_bytes([0, 5], [0, 5], 8, 3) == 0
    assert _varlen_bytes([0], [0], 8, 2) > 0                                           # an empty batch is valid


def _round_up(x, a):
    return (x + a - 1) // a * a


def _mxfp4_bytes(B, Hq, Hkv, Sq, Sk):
    """Status words and the MXFP4 copies of Q, K and V, each part on a 1 KiB boundary: what the general path lays out."""
    q, k = B * Hq * _round_up(Sq, 128), B * Hkv * _round_up(Sk, 128)
    return 1024 + sum(_round_up(rows * 64, 1024) + _round_up(rows * 4, 1024) for rows in (q, k, k))


def test_few_row_shapes_need_no_more_workspace_than_the_general_path():
    """The path for few query rows lays the workspace out differently but never needs more of it, so what fits a workspace (the
    4 MiB of efq_attention_fwd_static among them) does not depend on the path, and a workspace that is large enough for some
    query length is so for every shorter one."""
    size = binding.efq_attention_workspace_bytes
    for G in (1, 2, 3, 8, 24):
        for Sq in range(1, 26 // G + 1):
            for Hkv in (1, 2, 8, 31, 65):
                for Sk in list(range(64, 6000, 128)) + [129, 8192, 16383, 60001]:
                    assert size(1, G * Hkv, Hkv, Sq, Sk, 128) == _mxfp4_bytes(1, G * Hkv, Hkv, Sq, Sk), (G, Sq, Hkv, Sk)
    assert size(3, 8, 8, 24, 777, 128) == _mxfp4_bytes(3, 8, 8, 24, 777)
    # at the edge of the built-in scratch
    for Hq, Hkv, Sq, Sk in ((32, 8, 6, 3400), (24, 24, 24, 1100), (65, 65, 24, 300)):
        assert size(1, Hq, Hkv, Sq, Sk, 128) <= binding.STATIC_SCRATCH_BYTES


@pytest.mark.parametrize("lens", [[(24, 8100)] + [(1, 1900)] * 63, [(16, 1500)] + [(1, 128)] * 200, [(1 + n % 24, 1 + 137 * n) for n in range(150)]])
def test_few_row_sequences_of_a_packed_batch_take_no_more_than_their_copies(lens):
    """The size of a packed batch is that of its sequences (MXFP4 copies, which the path for few rows stays below), also where a
    sequence of 24 rows among sequences of one row makes room for 24 rows in each."""
    Hkv = 4
    cu_q = [sum(a for a, _ in lens[:i]) for i in range(len(lens) + 1)]
    cu_k = [sum(b for _, b in lens[:i]) for i in range(len(lens) + 1)]
    copies = sum(Hkv * (128 + 2 * _round_up(lk, 128)) * 68 for _, lk in lens)
    assert _varlen_bytes(cu_q, cu_k, Hkv, Hkv) <= copies + 1024 * len(lens) + 16384        # a table entry each on the general path


def test_workspace_of_a_packed_batch_grows_with_it():
    """A workspace that is large enough for a batch is so for every smaller one, across the number of items (2368) up to which their
    order may take more places than they are: a query tile more never needs less."""
    sizes = [_varlen_bytes([0, 128 * n, 128 * n + 300], [0, 300, 600], 1, 1) for n in range(2340, 2400)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))


def test_calls_do_not_hold_the_interpreter_lock(tmp_path):
    """While a call of the extension waits (here in functions that sleep in the place of the library's), other Python threads
    run: the counting thread gets on during each of the six calls."""
    (tmp_path / "slow.c").write_text("#include <unistd.h>\nlong slow(void) { usleep(200000); return 0; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", str(tmp_path / "slow.c"), "-o", str(tmp_path / "slow.so")], check=True)
    slow = ctypes.cast(ctypes.CDLL(str(tmp_path / "slow.so")).slow, ctypes.c_void_p).value
    fast = binding._fastcall()
    count, stop = [0], threading.Event()

    def run():
        while not stop.is_set():
            count[0] += 1
            time.sleep(0.002)

    thread = threading.Thread(target=run)
    fast.set_functions(*[slow] * 6)
    try:
        thread.start()
        for name, call in {"attention": lambda: fast.attention(*[0] * 11, 0.0, *[0] * 5),
                           "etq_attention": lambda: fast.etq_attention(*[0] * 11, 0.0, *[0] * 5),
                           "probgen": lambda: fast.probgen(*[0] * 5, 1.0, *[0] * 4),
                           "etq_probgen": lambda: fast.etq_probgen(*[0] * 5, 1.0, *[0] * 4),
                           "varlen_bytes": lambda: fast.varlen([0], [0], *[0] * 5, None, *[0] * 4, 0.0, *[0] * 5),
                           "varlen": lambda: fast.varlen([0], [0], *[0] * 10, 0.0, *[0] * 5)}.items():
            before = count[0]
            assert call() == 0
            assert count[0] - before >= 5, f"{name}: the other thread stood still"
    finally:
        stop.set()
        thread.join()
        binding._fast = None
        binding._fastcall()             # the library's own functions again


@pytest.mark.parametrize("cu_q,cu_k", [([0, 4], [0, 9]), ([0, 5], [0, 8]), ([0, 2, 5], [0, 9]), ([0, 5], [0, 4, 9])])
@pytest.mark.parametrize("workspace", [None, torch.empty(64, dtype=torch.uint8)])
def test_prefix_sums_that_do_not_fit_the_tensors_are_an_assertion(cu_q, cu_k, workspace):
    """Found by the binding before the library is called, with a workspace of the caller's or without."""
    q, k = torch.empty(5, 2, 128, dtype=torch.bfloat16), torch.empty(9, 2, 128, dtype=torch.bfloat16)
    with pytest.raises(AssertionError, match="prefix sums"):
        binding.efq_attention_fwd_varlen(q, k, k, cu_q, cu_k, workspace=workspace, stream=0)
