"""Host-side checks that need no GPU: the library loads and exports every symbol the header declares."""
import ctypes
import os
import re

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    src = open(os.path.join(ROOT, "include", "bpc.h")).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(bpc_[a-z_0-9]+)\s*\(", src)))


def test_library_exports_every_declared_symbol():
    from paper_2608_04405_b200 import binding as B
    names = _declared()
    assert len(names) >= 20
    lib = ctypes.CDLL(B.LIB_PATH)
    for n in names:
        assert hasattr(lib, n), "missing export %s" % n
    assert set(B.EXPORTS) == set(names)
    assert b"sm_100a" in B.lib.bpc_version()


def test_size_queries_and_config_validation_without_gpu():
    import torch
    from paper_2608_04405_b200 import binding as B
    cfg = B.make_config(4, 32, 8, 131072 + 256, 128, torch.bfloat16)
    assert B.lib.bpc_codes_bytes(ctypes.byref(cfg)) == 4 * 8 * (131072 + 256) * 16
    cfg64 = B.make_config(1, 1, 1, 4096, 64, torch.float32)
    assert B.lib.bpc_codes_bytes(ctypes.byref(cfg64)) == 4096 * 8        # one 64-bit word per key
    cfg32 = B.make_config(1, 4, 1, 4096, 32, torch.float32)
    assert B.lib.bpc_codes_bytes(ctypes.byref(cfg32)) == 4096 * 4        # half a word per key
    bad = B.make_config(1, 4, 1, 1024, 96, torch.bfloat16)
    assert B.lib.bpc_codes_bytes(ctypes.byref(bad)) == 0
    off = B.lib.bpc_fit_codes_offset(ctypes.byref(cfg64))
    assert 0 <= off < B.lib.bpc_fit_workspace_bytes(ctypes.byref(cfg64))   # (the fitted codes open the workspace)
    assert off % 256 == 0


def test_device_error_word_maps_to_a_status_and_library_reads_no_environment():
    """A non-zero device error word is reported as BPC_ERR_DEVICE (6); diagnostic switches are explicit calls, so no
    source file of the library reads the environment."""
    from paper_2608_04405_b200 import binding as B
    assert B.lib.bpc_status_of_device_error(0) == B.BPC_OK
    for word in (1, 2, 4, 7):
        assert B.lib.bpc_status_of_device_error(word) == 6 and B.STATUS_NAMES[6] == "BPC_ERR_DEVICE"
    csrc = os.path.join(ROOT, "paper_2608_04405_b200", "csrc")
    for f in os.listdir(csrc):
        assert "getenv" not in open(os.path.join(csrc, f)).read(), "%s reads the environment" % f


def test_product_path_does_not_import_the_checker():
    pkg = os.path.join(ROOT, "paper_2608_04405_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                txt = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in txt, "%s mentions the checker" % f
    for f in os.listdir(os.path.join(ROOT, "oracle")):
        if f.endswith(".py"):
            txt = open(os.path.join(ROOT, "oracle", f)).read()
            assert "paper_2608_04405_b200" not in txt and "ctypes" not in txt


def _binding():
    from paper_2608_04405_b200 import binding as B
    return B


def _b200_like_limits():
    """Resident clusters per size as a 148-SM part answers them: one block per SM, a cluster stays inside one GPC, GPCs of
    unequal size (this split reproduces the counts seen on a B200: 74 clusters of 2, 7 of 12 to 16, fewer than 16 of 8)."""
    gpcs = [10, 18, 20, 20, 20, 20, 20, 20]
    return [0] + [sum(g // c for g in gpcs) for c in range(1, 17)]


@pytest.mark.parametrize("batch,n_kv,n_max,want", [
    (1, 8, 131072 + 256, 10),      # 8 units: the largest size with all clusters resident (12+ hold only 7)
    (4, 8, 131072 + 256, 4),       # 32 units: 5 blocks each would need two waves
    (2, 8, 131072 + 256, 6),       # 16 units: 6 x 16 = 96 blocks in one wave, 8 x 16 would not be resident
    (5, 8, 131072 + 256, 3),       # 40 units
    (16, 8, 65536 + 64, 1),        # 128 units: one block each
    (1, 8, 1048576 + 64, 16),      # needs >= 13 blocks per unit; two waves either way, the smaller blocks win
    (1, 8, 4096, 4),               # a block keeps at least 1024 keys
])
def test_cluster_size_plan_on_given_device_limits(batch, n_kv, n_max, want):
    """The automatic cluster choice is host arithmetic over the device's occupancy answers: checked here on a table
    shaped like a 148-SM part, without a GPU."""
    B = _binding()
    cfg = B.make_config(batch, 4 * n_kv, n_kv, n_max, 128, torch.bfloat16)
    got = B.plan_cluster_size(cfg, _b200_like_limits(), 87000)
    assert got == want, (got, want)


def test_cluster_size_plan_edge_cases():
    B = _binding()
    cfg = B.make_config(1, 8, 8, 131072, 128, torch.bfloat16)
    ma = _b200_like_limits()
    assert B.plan_cluster_size(cfg, [0] * 17, 87000) == 0                 # nothing schedulable
    assert B.plan_cluster_size(cfg, ma, 1024) == 0                         # n_max fits no cluster: streaming applies
    only_pow2 = [v if c in (1, 2, 4, 8, 16) else 0 for c, v in enumerate(ma)]
    assert B.plan_cluster_size(cfg, only_pow2, 87000) == 8                 # sizes the device refuses are never chosen
    small = B.make_config(1, 8, 8, 1500, 128, torch.bfloat16)
    assert B.plan_cluster_size(small, ma, 87000) == 1                      # short contexts stay in one block
    got = B.plan_cluster_size(cfg, ma, 20000)                              # 131072 keys need >= 7 blocks of 20000
    assert got >= 7 and ma[got] >= 8


# resident clusters by size on a B200: blocks that take a whole SM, and half of one
WHOLE = [0, 148, 74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7]
HALF = [0, 296, 148, 93, 71, 56, 45, 37, 33, 30, 26, 21, 21, 17, 14, 14, 14]


@pytest.mark.parametrize("batch,heads,group,bits,score,lens,ppm,count,appends,plain,want", [
    (16, 8, 4, 128, 0, [65536] + [4096] * 15, 20000, 0, 1, 1, 2),            # one long sequence
    (16, 8, 4, 128, 0, [65536 - 3000 * i for i in range(16)], 20000, 0, 1, 1, 2),
    (16, 8, 4, 128, 0, [60000] * 16, 20000, 0, 1, 1, 0),                     # equal lengths: nothing to pair
    (16, 8, 4, 128, 0, [0] * 16, 20000, 0, 1, 1, 0),
    (16, 8, 4, 128, 0, [16384 - 700 * i for i in range(16)], 20000, 0, 1, 1, 0),   # too short to pay for the variant
    # the budget counts: with every unit gathering as many rows only the scan can be saved
    (16, 8, 4, 128, 0, [34000] + [8192] * 15, 50000, 0, 1, 1, 2), (16, 8, 4, 128, 0, [34000] + [8192] * 15, 10000, 0, 1, 1, 0),
    (16, 8, 4, 128, 0, [52000 - 2500 * i for i in range(16)], 20000, 0, 1, 1, 2), (16, 8, 4, 128, 0, [52000 - 2500 * i for i in range(16)], 0, 1040, 1, 1, 0),
    # 256 bits: appending costs both units of an SM their sign sweeps; decoding alone does not
    (16, 8, 4, 256, 0, [60000 - 1500 * i for i in range(16)], 20000, 0, 1, 1, 0), (16, 8, 4, 256, 0, [60000 - 1500 * i for i in range(16)], 20000, 0, 0, 1, 2),
    # score histograms beyond four bins per thread: weighted scores, 256 bits x 7 heads
    (16, 8, 4, 128, 1, [49152] + [8192] * 15, 20000, 0, 1, 1, 0), (16, 8, 7, 256, 0, [32768] + [2048] * 15, 20000, 0, 1, 1, 0),
    (6, 8, 4, 128, 1, [131072] + [8192] * 5, 20000, 0, 1, 2, 5),
    (6, 8, 4, 128, 0, [131072] + [8192] * 5, 20000, 0, 1, 2, 5),
    (8, 8, 4, 128, 0, [131072] + [8192] * 7, 20000, 0, 1, 2, 4),             # 64 clusters of 4: layers of 33 and 31
    (4, 8, 4, 128, 0, [131072] + [8192] * 3, 20000, 0, 1, 4, 0),             # 32 in clusters of 8 would straddle the layers (15 and 17)
    (15, 5, 4, 128, 0, [65536] * 5 + [3000] * 10, 20000, 0, 1, 1, 3),        # 75 units: layers of 45 and 30 clusters of 3
    (1, 148, 4, 128, 0, [65536], 20000, 0, 1, 1, 0),                         # one sequence
    (17, 8, 4, 128, 0, [65536] + [4096] * 16, 20000, 0, 1, 1, 0),            # more sequences than are ranked
])
def test_two_per_sm_plan_on_given_device_limits(batch, heads, group, bits, score, lens, ppm, count, appends, plain, want):
    """The choice is host arithmetic over lengths, budget and the device's occupancy answers.  Where it is made, every unit has its place
    in the grid once, the longest have their SMs to themselves, and the next ones share theirs with the shortest."""
    B = _binding()
    cfg = B.make_config(batch, heads * group, heads, (max(lens) + 1024) // 64 * 64, bits, torch.bfloat16, score_mode=score)
    cs, units = B.plan_two_per_sm(cfg, WHOLE, HALF, 40000, plain, lens, ppm, count, bool(appends))
    assert cs == want
    if not cs:
        return
    n = batch * heads
    assert sorted(units) == list(range(n)) and WHOLE[cs] < n <= min(2 * WHOLE[cs], HALF[cs])
    first, pairs = WHOLE[cs], n - WHOLE[cs]
    length = [lens[u // heads] for u in units]
    ranked = sorted((lens[u // heads] for u in range(n)), reverse=True)
    assert sorted(length[pairs:first], reverse=True) == ranked[:first - pairs]
    for i in range(pairs):
        assert length[i] == ranked[first - pairs + i] and length[first + i] == ranked[n - 1 - i]


def test_two_per_sm_plan_refuses():
    B = _binding()
    lens = [65536] + [4096] * 15
    n_max = 66560

    def plan(cfg, whole=WHOLE, half=HALF, cap=40000, lens=lens):
        return B.plan_two_per_sm(cfg, whole, half, cap, 1, lens, 20000)[0]

    cfg = B.make_config(16, 32, 8, n_max, 128, torch.bfloat16)
    assert plan(cfg) == 2
    assert plan(cfg, cap=20000) == 0                                         # blocks that cannot hold half of n_max
    assert plan(cfg, half=[0] * 17) == 0 and plan(cfg, whole=[0] * 17) == 0
    assert plan(cfg, half=[min(v, 127) for v in HALF]) == 0                  # not all units resident
    assert plan(cfg, lens=[n_max + 1] + [0] * 15) == 0                       # no such length
    assert plan(B.make_config(16, 32, 8, n_max, 128, torch.float32)) == 0
    assert plan(B.make_config(16, 32, 8, n_max, 128, torch.bfloat16, eas_ppm=2000)) == 0


def test_fit_cluster_size_bounds_the_keys_of_a_block():
    """The sweep adds bytes over a block's keys in 32 bits: no size that gives a block more than 2^24 keys, whatever it would cost."""
    B = _binding()
    longest = B.make_config(1, 1, 1, 1 << 26, 128, torch.bfloat16)
    for units in (1, 40, 200):                               # (as cheap as a block per unit may look)
        cfg = B.make_config(units, 1, 1, 1 << 26, 128, torch.bfloat16)
        assert B.plan_fit_cluster_size(cfg, WHOLE) >= 4
    assert B.plan_fit_cluster_size(longest, WHOLE[:5] + [0] * 12) == 4
    assert B.plan_fit_cluster_size(longest, WHOLE[:4] + [0] * 13) == 0
    assert B.plan_fit_cluster_size(B.make_config(1, 1, 1, 1 << 24, 128, torch.bfloat16), WHOLE[:2] + [0] * 15) == 1
    assert B.plan_fit_cluster_size(B.make_config(1, 1, 1, (1 << 24) + 256, 128, torch.bfloat16), WHOLE[:2] + [0] * 15) == 0
    assert B.plan_fit_cluster_size(B.make_config(1, 32, 8, 32768, 128, torch.bfloat16), WHOLE) > 4
    assert B.plan_fit_cluster_size(longest, [0] * 17) == 0


def test_stream_where_torch_has_no_raw_one(monkeypatch):
    """The current stream comes from the public function where torch lacks the private ones."""
    B = _binding()

    class Stream:
        cuda_stream = 4711

    monkeypatch.setattr(torch.cuda, "current_stream", Stream)
    for name in ("_raw_stream", "_current_device"):
        with monkeypatch.context() as m:
            m.setattr(B, name, None)
            assert B._stream() == 4711


@pytest.mark.gpu
def test_stream_is_the_current_one():
    B = _binding()
    for s in (torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.default_stream()):
        with torch.cuda.stream(s):
            assert B._stream() == s.cuda_stream
