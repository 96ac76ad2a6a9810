"""Host-side checks that need no GPU: the C-ABI library builds, loads and exports every symbol the
header declares; size helpers; loud failure without a device; multi-rank aggregation (gloo)."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    from paper_2605_26632_b200 import binding

    lib = binding.load_library()
    header = open(os.path.join(ROOT, "include", "lynx.h")).read()
    declared = set(re.findall(r"LYNX_API\s+[\w\s\*]+?\b(lynx_\w+)\s*\(", header))
    assert declared, "no declarations parsed"
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_size_helpers():
    from paper_2605_26632_b200 import binding

    assert binding.values_bytes(4096, 12288) == 4096 * 6144 * 2
    assert binding.meta_bytes(4096, 12288) == 4096 * 12288 // 8
    assert binding.meta_bytes(200, 384) == 2 * 3 * 2048  # padded to 128 rows
    assert binding.meta_bytes(1, 128) == 2048
    lib = binding.load_library()
    assert lib.lynx_workspace_bytes(256, 512, 512) >= 256 * 256 * 2 + 2 * 4 * 2048 + 256 * 4


def test_compiled_calls_for_another_torch_or_other_sources_are_not_loaded(monkeypatch, tmp_path):
    """The extension reads tensors through inlined layouts: only a build for this interpreter, torch and header may be loaded.
    Where it cannot be made the layers take the general path, and the compiler is not run again for every context."""
    from paper_2605_26632_b200 import binding, build

    assert binding.load_calls() is binding._layer_calls() and os.path.samefile(binding.load_calls().__file__, build.calls_path())
    header = tmp_path / "lynx.h"
    header.write_text(open(build.HEADER).read() + "\n")
    for target, name, value in ((torch, "__version__", "0.0+other"), (torch.version, "git_version", "other"),
                                (build, "CALLS_DEPS", build.CALLS_SOURCES + [str(header)])):
        tried = []

        def no_compiler(cmd, path, verbose):
            tried.append(path)
            raise RuntimeError("no compiler")

        with monkeypatch.context() as mp:
            here = build.calls_path()
            mp.setattr(target, name, value)
            mp.setattr(build, "_run", no_compiler)
            mp.setattr(binding, "_calls", None)
            mp.setattr(binding, "_calls_failure", None)
            assert build.calls_path() != here
            for _ in range(2):
                with pytest.raises(RuntimeError):
                    binding.load_calls()
                with pytest.warns(UserWarning, match="compiled calls"):
                    assert binding._layer_calls() is binding._GeneralPathOnly
            assert tried == [build.calls_path()]


def test_fp8_two_row_tiles_are_planned_where_they_were_measured_faster():
    """(M, N, K) of layers timed with both kernels: two row tiles per W stage faster, or a single tile (192 wide) by 6 % and more."""
    from paper_2605_26632_b200 import binding

    plan = lambda m, n, k: binding.load_library().lynx_gemm_fp8_plan(148, m, n, k, None, None)
    for shape in [(4096, 3072, 12288), (16384, 3072, 12288), (4352, 9216, 3072), (8192, 8880, 1792), (1393, 10240, 3840), (270, 12744, 13824)]:
        assert plan(*shape) == 1, shape
    for shape in [(2994, 9216, 3072), (16384, 9216, 2048), (8192, 12288, 2304), (8321, 3840, 3840), (15102, 3072, 3072), (1401, 3160, 4864)]:
        assert plan(*shape) == 0, shape


def test_fp8_layers_let_the_next_launch_begin_only_where_their_prune_kernel_has_a_block_per_sm():
    """That kernel keeps whole rows in shared memory: at least two of them, 2048 elements or longer."""
    from paper_2605_26632_b200 import binding

    begins = binding.load_library().lynx_gemm_fp8_begins_next
    assert [begins(k) for k in (256, 1024, 1792, 2048, 2304, 12288, 57600, 57856, 65536)] == [0, 0, 0, 1, 1, 1, 1, 0, 0]
    assert begins(0) == -1 and begins(300) == -1


def test_no_accumulator_hand_back_is_outstanding_when_the_gemm_ends():
    """The MMA issuer's waits, against barriers that complete a phase per hand-back and an epilogue that hands back as
    late as it can: no buffer is filled before its contents were handed back, and when the issuer is through
    every hand-back has arrived (they are remote arrives on its CTA's shared memory)."""
    import random

    from paper_2605_26632_b200 import binding

    rng = random.Random(1)
    orders = [(b, n) for b in (1, 2) for n in range(8)]  # single-tile kernel: the buffers in turn
    orders += [(2, [0, 1] * d + [i % 2 for i in range(s)]) for d in range(4) for s in range(4)]  # doubles, then singles
    orders += [(2, [rng.randint(0, 1) for _ in range(rng.randint(1, 9))]) for _ in range(40)]
    for buffers, order in orders:
        waits = binding.gemm_accumulator_waits(buffers, order)
        if isinstance(order, int):
            n, uses = order, [i % buffers for i in range(order + buffers)]
        else:
            n, uses = len(order), order + list(range(buffers))
        assert len(waits) == len(uses)
        filled, back = [0] * buffers, [0] * buffers
        for i, (parity, a) in enumerate(zip(waits, uses)):
            while (back[a] & 1) == parity:  # the phase with this parity is not complete: the issuer waits
                assert back[a] < filled[a], ("waits for ever", buffers, order, i)
                back[a] += 1
            assert back[a] == filled[a], ("not handed back yet", buffers, order, i)
            if i < n:
                filled[a] += 1
        assert back == filled, (buffers, order)


def test_gemm_kernels_with_too_few_registers_are_refused():
    """The GEMM's warps take 72 and 216 registers out of what 384 threads were launched with: 168 is the least."""
    from paper_2605_26632_b200 import binding

    fit = binding.load_library().lynx_gemm_register_shares_fit
    assert fit(168) == 1 and fit(167) == 0 and fit(160) == 0 and fit(128) == 0
    # every launch of such a kernel goes through the check
    src = open(os.path.join(ROOT, "paper_2605_26632_b200", "csrc", "lynx_api.cu")).read()
    for launch in ("launch_gemm_cfg", "launch_gemm_rt2", "launch_gemm_fp8_cfg"):
        body = src[src.index(f"lynx_status {launch}(lynx_ctx"):]
        body = body[:body.index("cudaLaunchKernelEx")]
        assert "prepare_gemm_kernel(" in body and "allow_dynamic_smem(" not in body, launch


def test_waits_of_whole_warps_end_alike_for_every_lane():
    """A bounded wait may give up, and each lane sees that for itself.  What a whole warp does behind a wait (tensor-memory
    reads, shuffles, warp barriers) needs all lanes, so only code of a single lane (or of lanes that feed a group of slots each) calls the per-lane form."""
    csrc = os.path.join(ROOT, "paper_2605_26632_b200", "csrc")
    found = 0
    for name in sorted(os.listdir(csrc)):
        if name == "ptx.cuh":  # where both forms are defined
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        headers, start = [], 0  # for every open brace the text in front of it
        for i, ch in enumerate(text):
            if ch == "{":
                headers.append(text[start:i])
            elif ch == "}":
                headers.pop()
            if ch in "{};":
                start = i + 1
            if text.startswith("mbar_wait(", i) and not text[i - 1].isalnum() and text[i - 1] != "_":
                found += 1
                one_lane = any(re.search(r"if \([^)]*\b(lane|threadIdx\.x) (== 0|< NG\b)", h) for h in headers)
                assert one_lane, (name, text.count("\n", 0, i) + 1)
    assert found >= 5


def test_fp8_tile_is_never_wider_than_its_rounds_call_for():
    """A narrower tile does less per round: where it needs no more rounds over the CTA pairs it is the one to take."""
    import random

    from paper_2605_26632_b200 import binding

    tile = binding.load_library().lynx_gemm_fp8_tile
    rng = random.Random(2)
    cases = [(1024, 4608, 3072), (700, 6144, 2048), (4096, 3072, 12288), (64, 256, 512), (16384, 21504, 3072)]
    cases += [(rng.randint(1, 8192), 8 * rng.randint(1, 2688), 256 * rng.randint(1, 60)) for _ in range(400)]
    seen = set()
    for M, N, K in cases:
        for pairs in (74, 66):
            rounds = {w: -(-(-(-M // 256) * -(-N // w)) // pairs) for w in (128, 192, 240)}
            w = tile(2 * pairs, M, N, K)
            seen.add(w)
            assert all(rounds[v] > rounds[w] for v in rounds if v < w), (M, N, K, pairs, w)
    assert seen == {128, 192, 240}
    assert tile(148, 4096, 3072, 12288) == 240 and tile(148, 1024, 4608, 3072) == 128
    assert tile(148, 0, 8, 256) == -1


def test_phase0_plan_fits_the_slack_it_counts_on():
    """The down projection inside the GEMM launch: work that goes to the CTA pairs with a tile less than the others fits there
    as a whole, and the tile's time is the launched tile's.  2048 x 12288 x 3072 runs 192-wide tiles on 74 pairs: 20 pairs
    have a tile less, 8 row blocks in two K splits take 26 us of the 31 that a tile lasts, whole rows of K do not fit."""
    import random

    from paper_2605_26632_b200 import binding

    lib = binding.load_library()

    def plan(M, N, K, sms=148):
        s, f = ctypes.c_int(-1), ctypes.c_int(-1)
        return lib.lynx_gemm_phase0_plan(sms, M, N, K, ctypes.byref(s), ctypes.byref(f)), s.value, f.value

    assert plan(2048, 3072, 12288) == (192, 2, 1)
    rng = random.Random(3)
    for _ in range(300):
        M, N, K = rng.randint(1, 16384), 8 * rng.randint(1, 2688), 128 * rng.randint(1, 120)
        width, splits, fill = plan(M, N, K)
        if width == 0:
            continue
        assert width in (192, 240, 256) and 1 <= splits <= max(1, K // 256) and 0 <= fill <= 8
        rows, tiles = -(-M // 256), -(-M // 256) * -(-N // width)
        pairs = min(74, tiles)
        light = pairs - tiles % pairs if tiles % pairs else 0
        assert fill == 0 or light * fill >= rows * splits, (M, N, K)
    assert plan(0, 8, 128)[0] == -1


def test_two_row_tile_schedule_covers_every_tile_exactly_once():
    """Host logic of the GEMM's work distribution: for any number of row tiles, column tiles,
    CTA pairs and 512-row items, every 256 x 240 tile is computed exactly once, doubles pair the
    row tiles 2d / 2d + 1, consecutive single-tile items of a pair alternate accumulators, and
    the pairs' loads differ by at most one item of each kind."""
    from paper_2605_26632_b200 import binding

    import itertools
    import random

    rng = random.Random(0)
    cases = [(16, 13, 74, 74), (16, 13, 74, 0), (16, 13, 74, 104), (17, 13, 74, 80), (3, 5, 74, 5), (3, 5, 4, 2),
             (1, 7, 74, 0), (64, 13, 74, 300), (19, 5, 74, 45), (47, 5, 74, 115), (2, 1, 74, 1)]
    cases += [(rng.randint(1, 40), rng.randint(1, 30), rng.randint(1, 74), rng.randint(0, 700)) for _ in range(60)]
    for tm, tn, pairs, doubles in cases:
        dmax = (tm // 2) * tn
        d_eff = min(doubles, dmax)
        clusters = max(1, min(pairs, tm * tn - d_eff))
        seen = {}
        nd, ns = [], []
        for c in range(clusters):
            items = binding.gemm_schedule_items(tm, tn, clusters, doubles, c)
            singles = [it for it in items if it[2] == 1]
            assert [it[3] for it in singles] == list(range(len(singles)))  # ordinals 0, 1, 2, ...
            assert all(it[2] == 2 for it in items[:len(items) - len(singles)])  # doubles first
            for (m0, n, rows, _) in items:
                assert rows in (1, 2) and 0 <= n < tn
                if rows == 2:
                    assert m0 % 2 == 0 and m0 + 1 < tm
                for r in range(rows):
                    assert 0 <= m0 + r < tm
                    seen[(m0 + r, n)] = seen.get((m0 + r, n), 0) + 1
            nd.append(len(items) - len(singles))
            ns.append(len(singles))
        assert len(seen) == tm * tn and set(seen.values()) == {1}, (tm, tn, pairs, doubles)
        assert sum(nd) == d_eff
        assert max(nd) - min(nd) <= 1
        # a pair with one double fewer never has fewer singles than a pair with one double more
        light = [s_ for d_, s_ in zip(nd, ns) if d_ == min(nd)]
        heavy = [s_ for d_, s_ in zip(nd, ns) if d_ == max(nd)]
        if max(nd) != min(nd):
            assert min(light) >= max(heavy)
        assert max(light) - min(light) <= 1 and max(heavy) - min(heavy) <= 1


def test_gemm_plan_prefers_single_tiles_for_small_problems():
    from paper_2605_26632_b200 import binding

    use, d, c = binding.gemm_plan(148, 1024, 3072, 3072)
    assert d == 0 or not use  # 52 tiles on 74 pairs: pairing row tiles would only serialise them
    use, d, c = binding.gemm_plan(148, 4096, 3072, 12288)
    assert c == 74 and 0 <= d <= 8 * 13


def test_status_strings():
    from paper_2605_26632_b200 import binding

    assert binding.status_string(0) == "ok"
    assert "128" in binding.status_string(2)
    assert "sm_100" in binding.status_string(7)


@pytest.mark.skipif(torch.cuda.is_available(), reason="checks the no-GPU failure path")
def test_no_gpu_means_loud_failure_not_fallback():
    from paper_2605_26632_b200 import binding

    with pytest.raises(binding.LynxError):
        binding.Lynx(0)


def test_product_never_imports_the_oracle():
    pkg = os.path.join(ROOT, "paper_2605_26632_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                text = open(os.path.join(dirpath, f)).read()
                for needle in ("import oracle", "from oracle", "liblynx_oracle", "lynx_oracle.c", "oracle_"):
                    assert needle not in text, f"{f} reaches into the oracle ({needle})"
    for f in os.listdir(os.path.join(ROOT, "oracle")):
        if f.endswith((".py", ".c")):
            text = open(os.path.join(ROOT, "oracle", f)).read()
            assert "paper_2605_26632_b200" not in text and "liblynx.so" not in text


_WORKER = r"""
import os, sys
sys.path.insert(0, {root!r})
import torch.distributed as dist
import bench
rank = int(os.environ["RANK"]); world = int(os.environ["WORLD_SIZE"])
dist.init_process_group("gloo")
ms = bench.max_over_ranks(10.0 + 5.0 * rank, world, device="cpu")
assert ms == 15.0, ms
v = bench.aggregate_tflops(1e12, 10, ms, world)
assert abs(v - 1e12 * 10 * 2 / 15e-3 / 1e12) < 1e-9, v
dist.barrier(); dist.destroy_process_group()
print("ok", rank)
"""


def test_replica_aggregation_two_ranks_gloo(tmp_path):
    script = tmp_path / "worker.py"
    script.write_text(_WORKER.format(root=ROOT))
    env = dict(os.environ, MASTER_ADDR="127.0.0.1", MASTER_PORT="29611", WORLD_SIZE="2")
    procs = [subprocess.Popen([sys.executable, str(script)], env=dict(env, RANK=str(r)),
                              stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True) for r in range(2)]
    outs = [p.communicate(timeout=120)[0] for p in procs]
    for p, o in zip(procs, outs):
        assert p.returncode == 0, o


def test_bench_launches_its_own_ranks_when_started_plainly():
    """``python bench.py --gpus 2`` without torchrun starts two ranks itself (127.0.0.1 rendezvous);
    checked through the GPU-free launch check: gloo ranks, max-over-ranks and aggregation."""
    import json

    env = {k: v for k, v in os.environ.items() if k not in ("WORLD_SIZE", "RANK", "LOCAL_RANK")}
    res = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--gpus", "2", "--launch-check"],
                         env=env, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    line = [l for l in res.stdout.splitlines() if l.startswith("{")][-1]
    d = json.loads(line)
    assert d["launch_check"] and d["n_gpus"] == 2 and d["slowest_rank_ms"] == 15.0
    assert abs(d["aggregate_tflops"] - 1e12 * 10 * 2 / 15e-3 / 1e12) < 1e-6


def test_split_plan_is_not_chosen_where_it_was_measured_slower():
    """(M, N, K, low-rank steps) of layers timed with and without the split; where it is chosen no two-row-tile plan is."""
    import random

    from paper_2605_26632_b200 import binding

    for m, n, k, lora in [(1498, 256, 2304, 0), (169, 5520, 4608, 0), (774, 1104, 3328, 0), (206, 4320, 3072, 1), (266, 3072, 3072, 1),
                          (384, 3072, 3072, 2), (1274, 464, 2560, 2), (692, 480, 2560, 2), (696, 624, 3072, 1)]:
        assert binding.gemm_split_plan(False, m, n, k, lora) == (0, 1), (m, n, k, lora)
    for m, n, k, lora in [(256, 3072, 3072, 0), (64, 3072, 3072, 0), (429, 280, 2560, 0), (495, 416, 2048, 0), (209, 3656, 2304, 0), (131, 3072, 3072, 1),
                          (167, 3072, 3072, 2), (472, 3072, 12288, 1), (80, 3840, 3840, 1)]:
        assert binding.gemm_split_plan(False, m, n, k, lora)[0] > 0, (m, n, k, lora)
    assert binding.gemm_split_plan(True, 280, 1904, 4608) == binding.gemm_split_plan(True, 606, 1144, 5376) == (0, 1)
    assert binding.gemm_split_plan(True, 1858, 376, 4864)[0] > 0 and binding.gemm_split_plan(True, 76, 5744, 6144)[0] > 0
    rng = random.Random(7)
    for _ in range(5000):
        m, k, n, lora = rng.randint(1, 2047), 128 * rng.randint(1, 128), 8 * rng.randint(1, 2688), rng.choice([0, 0, 1, 2])
        if binding.gemm_split_plan(False, m, n, k, lora)[0]:
            assert not binding.gemm_plan(148, m, n, k, lora)[0], (m, n, k, lora)


def test_split_layers_let_the_next_launch_begin_only_before_a_short_prune_launch():
    from paper_2605_26632_b200 import binding

    begins = binding.load_library().lynx_gemm_split_begins_next
    for mode, early in ((binding.COMP_NONE, 1), (binding.COMP_ROW, 1), (binding.COMP_TENSOR, 0), (binding.COMP_GROUP, 0)):
        assert begins(mode, 256, 3072, 3072) == begins(mode, 442, 336, 2816) == begins(mode, 512, 256, 5120) == early
        assert begins(mode, 700, 424, 3072) == begins(mode, 1500, 256, 3072) == begins(mode, 513, 256, 5120) == 0
        assert begins(mode, 226, 3840, 3840) == 0  # 120 SMs are held
        assert begins(mode, 256, 512, 512) == 0  # K is not split


def test_split_plan_is_one_round_and_has_a_k_block_for_every_member():
    import random

    from paper_2605_26632_b200 import binding

    rows, width, ctas = {1: 256, 2: 256, 5: 128}, {1: 128, 2: 192, 5: 128}, {1: 2, 2: 2, 5: 1}
    held = {2: 148, 3: 135, 4: 132, 5: 130, 6: 132, 7: 105, 8: 120}
    rng, seen = random.Random(4), set()
    cases = [(2047, 256, 16384, 0, 0), (2048, 256, 16384, 0, 0), (1, 8, 128, 0, 0), (256, 3072, 12288, 0, 1)]
    cases += [(rng.randint(1, 2300), 8 * rng.randint(1, 1300), 256 * rng.randint(1, 64), rng.random() < 0.3, 0) for _ in range(2000)]
    for M, N, K, fp8, lora in cases:
        tile, s = binding.gemm_split_plan(fp8, M, N, K, lora)
        if tile == 0:
            continue
        seen.add((tile, bool(fp8)))
        members = ctas[tile] * s
        assert 2 <= members <= 8 and s >= 2 and s <= K // (256 if fp8 else 128) and M < 2048
        assert -(-M // rows[tile]) * -(-N // width[tile]) * members <= held[members], (M, N, K)
    assert seen == {(t, f) for t in (1, 2, 5) for f in (False, True)}
    assert binding.gemm_split_plan(False, 256, 3072, 12288) == (1, 2) and binding.gemm_split_plan(False, 4096, 3072, 12288)[0] == 0
