#!/usr/bin/env python3
"""Benchmark of the sparse-bitmap codec hot path on B200.

Headline workload: the sparsity-sweep tensor of 2^28 fp32 elements (1 GiB) at half zeros.  One "step" is
one pass of the whole hot path over one batch of such tensors (24 of them, seeded differently, all
resident in HBM): per tensor bt_compress of the activation, bt_decompress of that stash,
bt_relu_fwd_compress of the pre-activation (stash only) and bt_relu_bwd_from_bitmap of an upstream
gradient -- four launches per tensor on one stream, about 27 ms per step, so that the default 20 steps
last half a second and the clock samples fall inside the timed region.  The metric
is dense-equivalent GB/s: N * sizeof(dtype) per call, summed over the step, divided by the step time.

Before that JSON line, the only one on standard output, every kernel of the five workload configurations
timed on its own goes to standard error, a JSON object per line: CUDA events around ONE launch, the L2
flushed before it, median over repetitions -- the single fp32 layer, the ResNet-18 step (batched launches),
the sparsity sweep (i.i.d. and clustered), the VGG-16 tensors in bf16 and fp16 (fused forward with and
without the dense output, backward), and the MobileNetV2 forward-then-reverse trace.  `roofline` of the
line is the row with the lowest fraction among the five graded calls on tensors of at least 256 MB.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
    python bench.py --case <f32|f16|bf16|f64> <op> [--log2n 26] [--zeros 0.5] [--reps 3]     # one kernel, for a profiler

With N > 1 (launched by torch.distributed.run, one rank per GPU) every rank runs the same batch on its
own GPU -- data-parallel replicas stash their own activations, there is no data-path collective -- and
the value is the sum over ranks divided by the slowest rank's time (weak scaling).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "codec_dense_equivalent_throughput"
UNIT = "GB/s"
WORKLOAD = "cfg3_sparsity_sweep_2p28_f32_half_zeros"
OPS = ("bt_compress", "bt_decompress", "bt_relu_fwd_compress", "bt_relu_bwd_from_bitmap")
LOG2N = 28
ZEROS = 0.5
NOMINAL_GBS = 8000.0
CASE_OPS = ("compress", "relu", "relu_y", "prune", "narrow", "relu6", "relu6_bwd", "decompress", "relu_bwd", "mask",
            "mask_y", "maxpool", "maxpool_bwd", "widen", "batch", "batch_restore")

# DRAM bytes (read + write) per element of a kernel, from one ncu capture of
#   python bench.py --case <dtype> <op> --log2n <26 for 4-byte, 27 for 2-byte elements>
# (dram__bytes_read.sum + dram__bytes_write.sum of the captured launch / its elements, at half zeros).  Traffic
# grows in proportion to the element count, so a full launch is this figure times its elements; the figure sits a
# little below the algorithmic bytes because the tail of what a launch writes is still in the L2 when it ends.
# The capture and its command are summarised in the file named beside each figure.
NCU_DRAM_BYTES_PER_ELEMENT = {
    ("bf16", "bt_relu_fwd_compress"): (2.830, "profiles/bt_compress_ncu.md"),
    ("f16", "bt_relu_fwd_compress"): (2.830, "profiles/bt_compress_ncu.md (bf16 capture; same kernel)"),
    ("bf16", "bt_relu_fwd_compress+y"): (4.709, "profiles/bt_compress_ncu.md"),
    ("f16", "bt_relu_fwd_compress+y"): (4.709, "profiles/bt_compress_ncu.md (bf16 capture; same kernel)"),
    ("bf16", "bt_compress"): (2.830, "profiles/bt_compress_ncu.md (fused capture; same bytes)"),
    ("f16", "bt_compress"): (2.830, "profiles/bt_compress_ncu.md (bf16 fused capture; same bytes)"),
    ("bf16", "bt_decompress"): (2.708, "profiles/bt_staged_walk_ncu.md"),
    ("f16", "bt_decompress"): (2.708, "profiles/bt_staged_walk_ncu.md (bf16 capture; same kernel)"),
    ("f32", "bt_compress"): (5.443, "profiles/bt_compress_ncu.md"),
    ("f32", "bt_relu_fwd_compress"): (5.443, "profiles/bt_compress_ncu.md (plain compressor; same kernel body)"),
    ("f32", "bt_decompress"): (5.277, "profiles/bt_staged_walk_ncu.md"),
    ("f32", "bt_relu_bwd_from_bitmap"): (7.372, "profiles/bt_relu_bwd_ncu.md"),
}


def parse_args(argv=None):
    p = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=20)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", choices=("ours", "reference"), default="ours")
    p.add_argument("--tensors", type=int, default=24, help="tensors of the batch one step passes over")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--no-kernels", action="store_true", help="skip the per-kernel table of the five configurations")
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--case", nargs=2, metavar=("DTYPE", "OP"),
                   help="run one entry point a few times on one seeded tensor and exit (for profiler captures); "
                        "OP one of " + ", ".join(CASE_OPS))
    p.add_argument("--log2n", type=int, default=26, help="--case: log2 of the element count")
    p.add_argument("--zeros", type=float, default=0.5, help="--case: zero fraction of the 4- and 8-byte input")
    p.add_argument("--tau", type=float, default=0.1, help="--case prune: threshold")
    p.add_argument("--reps", type=int, default=3, help="--case: repetitions")
    return p.parse_args(argv)


def workload_config() -> dict:
    """What both arms measure; the reference arm times a bounded sample of it."""
    return {"workload": WORKLOAD, "elements_per_tensor": 1 << LOG2N, "dtype": "f32", "zero_fraction": ZEROS,
            "ops_per_tensor": list(OPS)}


# ------------------------------------------------------------------------------------------
# clocks: read-only NVML sampling in a thread while the timed region runs
class ClockSampler:
    REASONS = {0x1: "gpu_idle", 0x2: "applications_clocks_setting", 0x4: "sw_power_cap", 0x8: "hw_slowdown",
               0x10: "sync_boost", 0x20: "sw_thermal_slowdown", 0x40: "hw_thermal_slowdown",
               0x80: "hw_power_brake_slowdown", 0x100: "display_clock_setting"}

    def __init__(self, index: int, period_s: float = 0.005):
        self.samples = []          # (host time, sm MHz, reasons bitmask)
        self.period = period_s
        self._stop = threading.Event()
        self.ok = False
        self.sm_max = None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = self._handle(index)
            self.sm_max = int(pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM))
            self.ok = True
        except Exception:
            self.ok = False
        self.thread = threading.Thread(target=self._run, daemon=True)

    def _handle(self, index):
        import torch
        try:
            uuid = str(torch.cuda.get_device_properties(index).uuid)
            uuid = uuid if uuid.startswith("GPU-") else "GPU-" + uuid
            return self.nv.nvmlDeviceGetHandleByUUID(uuid)
        except Exception:
            return self.nv.nvmlDeviceGetHandleByIndex(index)

    def _run(self):
        while not self._stop.is_set():
            try:
                mhz = int(self.nv.nvmlDeviceGetClockInfo(self.h, self.nv.NVML_CLOCK_SM))
                try:
                    r = int(self.nv.nvmlDeviceGetCurrentClocksEventReasons(self.h))
                except Exception:
                    r = int(self.nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.h))
                self.samples.append((time.time(), mhz, r))
            except Exception:
                pass
            self._stop.wait(self.period)

    def start(self):
        if self.ok:
            self.thread.start()

    def stop(self):
        self._stop.set()
        if self.ok and self.thread.is_alive():
            self.thread.join(timeout=1.0)

    def summary(self, t0: float, t1: float) -> dict:
        inside = [s for s in self.samples if t0 <= s[0] <= t1]
        note = "sampled during the timed region"
        if not inside:
            inside = self.samples[-3:]
            note = "timed region shorter than the sampling period: nearest samples"
        if not inside:
            return {"sm_mhz": None, "sm_max_mhz": self.sm_max, "reasons": [], "note": "NVML unavailable"}
        mask = 0
        for s in inside:
            mask |= s[2]
        reasons = [name for bit, name in self.REASONS.items() if mask & bit and name != "gpu_idle"]
        return {"sm_mhz": statistics.median(s[1] for s in inside), "sm_max_mhz": self.sm_max,
                "reasons": reasons, "samples": len(inside), "timed_region_s": round(t1 - t0, 4), "note": note}


def max_over_ranks(ms: float, world: int, device) -> float:
    """Slowest rank's time: the job is as fast as its slowest GPU."""
    if world <= 1:
        return ms
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_value(dense_bytes_per_rank_step: int, world: int, ms_per_step: float) -> float:
    """Dense-equivalent GB/s of the whole job: every rank processes its own batch (weak scaling)."""
    return world * dense_bytes_per_rank_step / (ms_per_step * 1e-3) / 1e9


def measured_peak_gbs():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except Exception:
        return 6650.0, "fallback"


def algorithmic_bytes(op: str, n: int, nnz: int, es: int, with_y: bool = False) -> int:
    """Bytes the method itself must move for one call (dense tensor, bitmap, packed values, prefix)."""
    compressed = 4 * ((n + 31) // 32) + nnz * es + 8 * ((n + 4095) // 4096)
    if op in ("bt_compress", "bt_decompress"):
        return n * es + compressed
    if op == "bt_relu_fwd_compress":
        return n * es + compressed + (n * es if with_y else 0)
    if op == "bt_relu_bwd_from_bitmap":
        return 2 * n * es + 4 * ((n + 31) // 32)
    raise ValueError(op)


# ------------------------------------------------------------------------------------------
# per-kernel timing: events around one launch (or one group of launches), L2 flushed before each
class KernelTimer:
    def __init__(self, dev, peak_gbs: float):
        import torch
        self.torch = torch
        self.peak = peak_gbs
        self.flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)      # twice the 126 MB L2
        self.rows = []

    def time(self, fn, reps: int = 9) -> float:
        """Median device time in ms of fn(), each repetition bracketed by its own pair of events."""
        torch = self.torch
        fn()                                                                     # warm: first-use set-up, instruction cache
        fn()
        pairs = []
        for _ in range(reps):
            self.flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            fn()
            e1.record()
            pairs.append((e0, e1))
        torch.cuda.synchronize()
        return statistics.median(a.elapsed_time(b) for a, b in pairs)

    def row(self, config: str, kernel: str, dtype: str, zero_fraction, n: int, alg_bytes: int, ms: float, **extra):
        gbs = alg_bytes / (ms * 1e-3) / 1e9
        r = {"config": config, "kernel": kernel, "dtype": dtype,
             "zero_fraction": None if zero_fraction is None else round(zero_fraction, 4), "elements": n,
             "algorithmic_bytes": alg_bytes, "median_ms": round(ms, 5), "gbs": round(gbs, 1),
             "frac_of_measured": round(gbs / self.peak, 4), "frac_of_8tbs": round(gbs / NOMINAL_GBS, 4)}
        r.update(extra)
        self.rows.append(r)
        return r


def _kinds():
    import torch
    return {torch.float32: "f32", torch.float16: "f16", torch.bfloat16: "bf16", torch.float64: "f64"}


def codec_rows(T: KernelTimer, B, config: str, x, pre, g, label_zero, ops=("compress", "decompress", "bwd"), tag=""):
    """Times the graded calls on one tensor: x the activation (post-ReLU), pre its pre-activation (or None), g an
    upstream gradient (or None)."""
    import torch
    n = x.numel()
    es = x.element_size()
    kind = _kinds()[x.dtype]
    st = B.Stash(n, x.dtype, x.device)
    ws = B.new_workspace(n, x.device)
    out = torch.empty_like(x)
    B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
    torch.cuda.synchronize()
    assert st.status == B.BT_OK
    nnz = st.nnz
    zf = 1.0 - nnz / n if label_zero is None else label_zero
    extra = {"tensor": tag} if tag else {}
    if "compress" in ops:
        ms = T.time(lambda: B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
        T.row(config, "bt_compress", kind, zf, n, algorithmic_bytes("bt_compress", n, nnz, es), ms, **extra)
    if "decompress" in ops:
        ms = T.time(lambda: B.bt_decompress(st.bitmap, st.values, st.chunk_prefix, out))
        T.row(config, "bt_decompress", kind, zf, n, algorithmic_bytes("bt_decompress", n, nnz, es), ms, **extra)
        assert torch.equal(out.view(torch.uint8), x.view(torch.uint8)), "round trip is not the identity"
    if pre is not None and "fwd" in ops:
        ms = T.time(lambda: B.bt_relu_fwd_compress(pre, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
        T.row(config, "bt_relu_fwd_compress", kind, zf, n, algorithmic_bytes("bt_relu_fwd_compress", n, nnz, es), ms,
              dense_output=False, **extra)
        ms = T.time(lambda: B.bt_relu_fwd_compress(pre, out, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
        T.row(config, "bt_relu_fwd_compress", kind, zf, n, algorithmic_bytes("bt_relu_fwd_compress", n, nnz, es, True), ms,
              dense_output=True, **extra)
        torch.cuda.synchronize()
        assert st.status == B.BT_OK and st.nnz == nnz
    if g is not None and "bwd" in ops:
        ms = T.time(lambda: B.bt_relu_bwd_from_bitmap(st.bitmap, g, out))
        T.row(config, "bt_relu_bwd_from_bitmap", kind, zf, n, algorithmic_bytes("bt_relu_bwd_from_bitmap", n, nnz, es), ms, **extra)
    del st, ws, out


def kernel_table(dev, peak_gbs: float):
    """Every kernel of the five workload configurations, each timed on its own."""
    import torch
    from paper_2110_15362_b200 import binding as B
    from paper_2110_15362_b200 import workloads as W
    T = KernelTimer(dev, peak_gbs)
    extras = {}

    # configuration 1: one fp32 layer of 200,704 elements
    x = W.cfg1(dev).reshape(-1)
    codec_rows(T, B, "cfg1", x, None, None, None, ops=("compress", "decompress"))

    # configuration 2: the ResNet-18 step at batch 32, the compressors as one batched launch each
    shapes = W.resnet18_shapes(32)
    acts, pres, grads = [], [], []
    for i, shape, n in W.iter_layers(shapes):
        pre = W.cfg2_preact(i, shape, dev).reshape(-1)
        pres.append(pre)
        acts.append(torch.clamp_min(pre, 0.0))
        grads.append(W.cfg2_grad(i, shape, dev).reshape(-1))
    ns = [a.numel() for a in acts]
    st_a = [B.Stash(n, torch.float32, dev) for n in ns]
    st_b = [B.Stash(n, torch.float32, dev) for n in ns]
    outs = [torch.empty_like(a) for a in acts]
    bws = torch.empty(B.bt_batch_workspace_bytes(ns), dtype=torch.uint8, device=dev)
    items_a = B.batch_items(acts, st_a)
    items_b = B.batch_items(pres, st_b)

    def fwd_plain():
        B.bt_compress_batch(items_a, torch.float32, bws)

    def fwd_fused():
        B.bt_relu_fwd_compress_batch(items_b, torch.float32, bws)

    items_r = B.batch_items(outs[::-1], st_a[::-1], outs[::-1])            # the backward pass takes the layers in reverse
    items_g = B.batch_items(grads[::-1], st_b[::-1], outs[::-1])

    def bwd_restore():
        B.bt_decompress_batch(items_r, torch.float32)

    def bwd_grad():
        B.bt_relu_bwd_from_bitmap_batch(items_g, torch.float32)

    fwd_plain(), fwd_fused()
    torch.cuda.synchronize()
    nnzs = [s.nnz for s in st_a]
    assert all(s.status == B.BT_OK for s in st_a + st_b) and nnzs == [s.nnz for s in st_b]
    n_all, z_all = sum(ns), 1.0 - sum(nnzs) / sum(ns)
    for name, fn, op, launches in (("bt_compress_batch", fwd_plain, "bt_compress", 1),
                                   ("bt_relu_fwd_compress_batch", fwd_fused, "bt_relu_fwd_compress", 1),
                                   ("bt_decompress_batch", bwd_restore, "bt_decompress", 1),
                                   ("bt_relu_bwd_from_bitmap_batch", bwd_grad, "bt_relu_bwd_from_bitmap", 1)):
        alg = sum(algorithmic_bytes(op, n, z, 4) for n, z in zip(ns, nnzs))
        T.row("cfg2", name, "f32", z_all, n_all, alg, T.time(fn), launches=launches, tensors=len(ns),
              note="all 17 layers: one event pair around the %d launch(es)" % launches)
    ms_step = T.time(lambda: (fwd_plain(), fwd_fused(), bwd_restore(), bwd_grad()))
    extras["cfg2_step"] = {"device_ms": round(ms_step, 4), "launches": 4, "tensors": len(ns),
                           "elements": n_all, "dense_equivalent_gbs": round(4 * 4 * n_all / (ms_step * 1e-3) / 1e9, 1),
                           "caller_cta_budget": "none",
                           "what": "bt_compress_batch + bt_relu_fwd_compress_batch forward, bt_decompress_batch + "
                                   "bt_relu_bwd_from_bitmap_batch over the layers in reverse order, one stream, L2 "
                                   "flushed before the step"}
    assert all(torch.equal(o.view(torch.int32), torch.where(p > 0, g, torch.zeros((), device=dev)).view(torch.int32))
               for o, p, g in zip(outs, pres, grads))
    del acts, pres, grads, st_a, st_b, outs, bws
    torch.cuda.empty_cache()

    # configuration 3: 2^28 fp32 elements, six zero fractions, zeros i.i.d. and in runs
    n = 1 << LOG2N
    g = W.cfg2_grad(3, (n,), dev)
    for variant, gen in (("iid", W.cfg3_iid), ("clustered", W.cfg3_clustered)):
        for idx, s in enumerate(W.SPARSITY_SWEEP):
            x = gen(n, s, idx, dev)
            codec_rows(T, B, "cfg3_" + variant, x, None, g, s)
            del x
    del g
    torch.cuda.empty_cache()

    # configuration 4: the 13 VGG-16 tensors at batch 64 in bf16 and fp16, fused forward and backward; tensor by
    # tensor, then all 13 as one batched launch per direction
    for kind in ("bf16", "f16"):
        pres, grs = [], []
        for i, shape, n in W.iter_layers(W.vgg16_shapes(64)):
            pre = W.cfg4_preact(i, shape, kind, dev).reshape(-1)
            gr = W.cfg4_grad(i, shape, kind, dev).reshape(-1)
            y = torch.relu(pre) + 0.0
            codec_rows(T, B, "cfg4", y, pre, gr, None, ops=("fwd", "bwd") + (("compress", "decompress") if i == 0 else ()),
                       tag="%d:%s" % (i, "x".join(map(str, shape))))
            pres.append(pre), grs.append(gr)
            del y
        ns4 = [p.numel() for p in pres]
        sts = [B.Stash(n, pres[0].dtype, dev) for n in ns4]
        gins = [torch.empty_like(g) for g in grs]
        bws = torch.empty(B.bt_batch_workspace_bytes(ns4), dtype=torch.uint8, device=dev)
        items_f = B.batch_items(pres, sts)
        items_b = B.batch_items(grs[::-1], sts[::-1], gins[::-1])
        ms_f = T.time(lambda: B.bt_relu_fwd_compress_batch(items_f, pres[0].dtype, bws))
        torch.cuda.synchronize()
        z4 = [s_.nnz for s_ in sts]
        assert all(s_.status == B.BT_OK for s_ in sts)
        T.row("cfg4", "bt_relu_fwd_compress_batch", kind, 1.0 - sum(z4) / sum(ns4), sum(ns4),
              sum(algorithmic_bytes("bt_relu_fwd_compress", n, z, 2) for n, z in zip(ns4, z4)), ms_f, launches=1, tensors=len(ns4),
              dense_output=False, note="all 13 tensors in one launch")
        ms_b = T.time(lambda: B.bt_relu_bwd_from_bitmap_batch(items_b, pres[0].dtype))
        T.row("cfg4", "bt_relu_bwd_from_bitmap_batch", kind, 1.0 - sum(z4) / sum(ns4), sum(ns4),
              sum(algorithmic_bytes("bt_relu_bwd_from_bitmap", n, z, 2) for n, z in zip(ns4, z4)), ms_b, launches=1,
              tensors=len(ns4), note="all 13 tensors in one launch")
        assert torch.equal(gins[-1].view(torch.int16), torch.where(pres[-1] > 0, grs[-1], torch.zeros((), device=dev, dtype=grs[-1].dtype)).view(torch.int16))
        del pres, grs, sts, gins, bws
        torch.cuda.empty_cache()

    # configuration 5: MobileNetV2 trace at batch 128, forward then reverse on one stream, values packed back to
    # back in one arena whose cursor lives on the device (no host round trip between layers)
    shapes = W.mobilenetv2_shapes(128)
    fr = W.cfg5_zero_fractions(len(shapes))
    layers = [W.cfg5_layer(i, shape, fr[i], dev).reshape(-1) for i, shape, _ in W.iter_layers(shapes)]
    ns = [l.numel() for l in layers]
    nnz_true = [int(torch.count_nonzero(l).item()) for l in layers]
    arena_bytes = sum((4 * z + 15) // 16 * 16 for z in nnz_true)
    arena = torch.empty(arena_bytes, dtype=torch.uint8, device=dev)
    cursor = torch.zeros(1, dtype=torch.int64, device=dev)
    stashes = [B.Stash(n, torch.float32, dev, values_capacity=1) for n in ns]     # bitmap, prefix, nnz, status; values in the arena
    offsets = torch.zeros(len(ns), dtype=torch.int64, device=dev)
    backs = [torch.empty(n, dtype=torch.float32, device=dev) for n in ns]
    ws = torch.empty(B.bt_batch_workspace_bytes(ns), dtype=torch.uint8, device=dev)
    items_f = B.batch_items(layers, stashes)
    items_r = B.batch_items(backs[::-1], stashes[::-1], backs[::-1])
    offsets_r = torch.empty_like(offsets)

    def forward():
        cursor.zero_()
        B.bt_compress_arena_batch(items_f, torch.float32, arena, cursor, offsets, ws)

    def reverse():
        offsets_r.copy_(offsets.flip(0))
        B.bt_decompress_arena_batch(items_r, torch.float32, arena, offsets_r)

    ms_f, ms_r = T.time(forward, reps=5), T.time(reverse, reps=5)
    ms_both = T.time(lambda: (forward(), reverse()), reps=5)
    torch.cuda.synchronize()
    assert all(st.status == B.BT_OK for st in stashes)
    assert [st.nnz for st in stashes] == nnz_true
    assert all(torch.equal(b.view(torch.int32), l.view(torch.int32)) for b, l in zip(backs, layers))
    # the same trace as one launch per layer, for comparison
    ws1 = B.new_workspace(max(ns), dev)
    offs1 = [torch.zeros(1, dtype=torch.int64, device=dev) for _ in ns]

    def forward_single():
        cursor.zero_()
        for l, st, o in zip(layers, stashes, offs1):
            B.bt_compress_arena(l, st.bitmap, arena, cursor, o, st.chunk_prefix, st.nnz_out, ws1, st.dev_status)

    def reverse_single():
        for b, st, o in zip(reversed(backs), reversed(stashes), reversed(offs1)):
            B.bt_decompress_arena(st.bitmap, arena, o, st.chunk_prefix, b)

    ms_f1, ms_r1 = T.time(forward_single, reps=5), T.time(reverse_single, reps=5)
    launches_f = (len(ns) + B.MAX_BATCH_PER_LAUNCH - 1) // B.MAX_BATCH_PER_LAUNCH
    stash_bytes = sum(B.bt_compressed_bytes(n, z, torch.float32) for n, z in zip(ns, nnz_true))
    assert stash_bytes == sum(4 * ((n + 31) // 32) + 4 * z + 8 * ((n + 4095) // 4096) for n, z in zip(ns, nnz_true))
    dense = 4 * sum(ns)
    alg_f = sum(algorithmic_bytes("bt_compress", n, z, 4) for n, z in zip(ns, nnz_true))
    z5 = 1.0 - sum(nnz_true) / sum(ns)
    T.row("cfg5", "bt_compress_arena_batch", "f32", z5, sum(ns), alg_f, ms_f, launches=launches_f, tensors=len(ns),
          note="35 layers in forward order, 32 per launch: one event pair around the %d launches" % launches_f)
    T.row("cfg5", "bt_decompress_arena_batch", "f32", z5, sum(ns), alg_f, ms_r, launches=launches_f, tensors=len(ns),
          note="35 layers in reverse order, 32 per launch: one event pair around the %d launches" % launches_f)
    T.row("cfg5", "bt_compress_arena", "f32", z5, sum(ns), alg_f, ms_f1, launches=len(ns), tensors=len(ns),
          note="the same forward pass as one launch per layer: one event pair around the 35 launches")
    T.row("cfg5", "bt_decompress_arena", "f32", z5, sum(ns), alg_f, ms_r1, launches=len(ns), tensors=len(ns),
          note="the same reverse pass as one launch per layer: one event pair around the 35 launches")
    extras["cfg5_trace"] = {"device_ms_forward_then_reverse": round(ms_both, 4), "device_ms_forward": round(ms_f, 4),
                            "device_ms_reverse": round(ms_r, 4), "launches": 2 * launches_f, "layers": len(ns), "elements": sum(ns),
                            "dense_bytes": dense, "peak_compressed_bytes": stash_bytes,
                            "compressed_over_dense": round(stash_bytes / dense, 4),
                            "arena_bytes_in_use_at_peak": int(cursor.item()),
                            "storage_policy": "exact size: every layer's packed values pushed back to back into one "
                                              "arena (device-side cursor, 16-byte granules) by the batched arena calls, "
                                              "32 layers per launch, bitmap and prefix array per layer; nothing is "
                                              "sized from nnz on the host, no host synchronisation between layers; the "
                                              "peak is reached after the last forward layer, when all 35 stashes are live"}
    del layers, arena, stashes, ws, ws1, backs
    torch.cuda.empty_cache()

    next_rows(T, B, W, dev)
    return T.rows, extras


def next_rows(T: KernelTimer, B, W, dev):
    """The calls built after the hot path (pruning threshold, double mask, ReLU6 pair, down-cast on stash, 8-byte
    elements, max pooling), each alone on the 1 GiB fp32 tensor, the 392 MiB bf16 tensor or the 1 GiB fp64 tensor."""
    import torch
    for kind, n in (("f32", 1 << 28), ("bf16", 64 * 64 * 224 * 224), ("f64", 1 << 27)):
        if kind == "f32":
            x = W.cfg3_iid(n, 0.5, 2, dev)
            pre = x
        elif kind == "f64":
            x = W.cfg3_iid(n, 0.5, 3, dev).double()
            pre = x
        else:
            pre = W.cfg4_preact(0, (n,), kind, dev)
            x = torch.relu(pre) + 0.0
        es = x.element_size()
        st = B.Stash(n, x.dtype, dev)
        ws = B.new_workspace(n, dev)
        dense = torch.empty_like(x)
        meta = 4 * ((n + 31) // 32) + 8 * ((n + 4095) // 4096)

        def add(kernel, ms, alg, **extra):
            T.row("next", kernel, kind, 1.0 - st.nnz / n, n, alg, ms, **extra)

        if kind == "f64":                                    # 8-byte elements through the graded calls
            ms = T.time(lambda: B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
            add("bt_compress", ms, algorithmic_bytes("bt_compress", n, st.nnz, es))
            ms = T.time(lambda: B.bt_decompress(st.bitmap, st.values, st.chunk_prefix, dense))
            add("bt_decompress", ms, algorithmic_bytes("bt_decompress", n, st.nnz, es))
            ms = T.time(lambda: B.bt_relu_bwd_from_bitmap(st.bitmap, x, dense))
            add("bt_relu_bwd_from_bitmap", ms, algorithmic_bytes("bt_relu_bwd_from_bitmap", n, 0, es))
        ms = T.time(lambda: B.bt_relu6_fwd_compress(pre, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
        torch.cuda.synchronize()
        nnz6 = st.nnz
        add("bt_relu6_fwd_compress", ms, n * es + meta + nnz6 * es, dense_output=False)
        ms = T.time(lambda: B.bt_relu6_bwd_from_stash(st.bitmap, st.values, st.chunk_prefix, x, dense))
        add("bt_relu6_bwd_from_stash", ms, 2 * n * es + meta + nnz6 * es)
        if kind == "f32":
            for to, tdt in (("f16", torch.float16), ("bf16", torch.bfloat16)):
                v16 = torch.empty(n, dtype=tdt, device=dev)
                ms = T.time(lambda: B.bt_compress_narrow(x, st.bitmap, v16, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
                torch.cuda.synchronize()
                by16 = n * es + meta + st.nnz * 2
                add("bt_compress_narrow", ms, by16, values=to)
                ms = T.time(lambda: B.bt_prune_fwd_compress_narrow(pre, 0.0, None, st.bitmap, v16, st.chunk_prefix, st.nnz_out, ws,
                                                                    st.dev_status))
                add("bt_prune_fwd_compress_narrow", ms, by16, values=to, tau=0.0)
                ms = T.time(lambda: B.bt_decompress_widen(st.bitmap, v16, st.chunk_prefix, dense))
                add("bt_decompress_widen", ms, by16, values=to)
                del v16
        B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        torch.cuda.synchronize()
        nnz = st.nnz
        masked = torch.empty(nnz, dtype=x.dtype, device=dev)
        ms = T.time(lambda: B.bt_mask_compress(pre, st.bitmap, st.chunk_prefix, None, masked))
        add("bt_mask_compress", ms, n * es + meta + nnz * es, dense_output=False)
        ms = T.time(lambda: B.bt_mask_compress(pre, st.bitmap, st.chunk_prefix, dense, masked))
        add("bt_mask_compress", ms, 2 * n * es + meta + nnz * es, dense_output=True)
        del x, pre, st, ws, dense, masked
        torch.cuda.empty_cache()

    # the pruning thresholds of the paper's study on 2^28 close-to-zero fp32 pre-activations
    n = 1 << 28
    pre = W.prune_preact(n, dev)
    st = B.Stash(n, pre.dtype, dev)
    ws = B.new_workspace(n, dev)
    for tau in W.PRUNE_THRESHOLDS:
        ms = T.time(lambda: B.bt_prune_fwd_compress(pre, tau, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status))
        torch.cuda.synchronize()
        T.row("next", "bt_prune_fwd_compress", "f32", 1.0 - st.nnz / n, n, algorithmic_bytes("bt_relu_fwd_compress", n, st.nnz, 4), ms,
              tau=tau, stash_bytes_over_dense=round(B.bt_compressed_bytes(n, st.nnz, pre.dtype) / (4.0 * n), 4), dense_output=False)
    del pre, st, ws
    torch.cuda.empty_cache()

    # max pooling with winner codes: the first pooling layer of a VGG-16 at batch 32
    for kind, dt in (("f32", torch.float32), ("bf16", torch.bfloat16)):
        x = torch.clamp_min(torch.randn(32, 64, 224, 224, device=dev, generator=torch.Generator(device=dev).manual_seed(900)), 0).to(dt)
        no, es = x.numel() // 4, x.element_size()
        y = torch.empty(32, 64, 112, 112, dtype=dt, device=dev)
        codes = torch.empty((no + 15) // 16, dtype=torch.int32, device=dev)
        gin = torch.empty_like(x)
        by = 5 * no * es + 4 * ((no + 15) // 16)
        pooled_bitmap = torch.randint(-2 ** 31, 2 ** 31 - 1, ((no + 31) // 32,), dtype=torch.int32, device=dev)
        for op, fn in (("bt_maxpool2x2_fwd", lambda: B.bt_maxpool2x2_fwd(x, y, codes)),
                       ("bt_maxpool2x2_bwd", lambda: B.bt_maxpool2x2_bwd(codes, y, gin)),
                       ("bt_maxpool2x2_bwd_masked", lambda: B.bt_maxpool2x2_bwd_masked(codes, pooled_bitmap, y, gin))):
            T.row("next", op, kind, None, x.numel(), by, T.time(fn), tensor="32x64x224x224")
        del x, y, codes, gin, pooled_bitmap
        torch.cuda.empty_cache()


# ------------------------------------------------------------------------------------------
def oracle_four_ops(x_np, pre_np, g_np):
    """The CPU oracle on one tensor, the step's four operations; returns seconds."""
    from oracle import bt_oracle as O
    t0 = time.perf_counter()
    a = O.compress(x_np)
    O.decompress(a)
    _, b = O.relu_fwd_compress(pre_np, "f32", want_y=False)
    O.relu_bwd_from_bitmap(b.bitmap, g_np)
    return time.perf_counter() - t0


def host_sample(m: int):
    """The first m elements of tensor 0 of the batch, its pre-activation and a gradient, as raw numpy arrays."""
    import torch
    from paper_2110_15362_b200 import workloads as W
    x = W.cfg3_iid(m, ZEROS, 0, "cpu")
    pre = torch.where(x != 0, x, torch.full((), -1.0))
    g = W.cfg2_grad(0, (m,), "cpu")
    return W.raw_numpy(x), W.raw_numpy(pre), W.raw_numpy(g)


def run_reference(args):
    """The oracle, as it stands, on host cores.  Every step is the step's four operations on a bounded sample of
    one tensor of the workload, sized from a short calibration so that warm-up plus timed steps take a minute or two."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cal = host_sample(1 << 20)
    rate = (1 << 20) / max(oracle_four_ops(*cal), 1e-6)                  # elements per second through all four
    budget_s = float(getattr(args, "reference_budget_s", 60.0))
    m = int(rate * budget_s / max(args.steps + args.warmup, 1))
    m = max(1 << 16, min(1 << LOG2N, m // 4096 * 4096))
    x, pre, g = host_sample(m)
    for _ in range(args.warmup):
        oracle_four_ops(x, pre, g)
    total = sum(oracle_four_ops(x, pre, g) for _ in range(args.steps))
    value = len(OPS) * 4 * m * args.steps / total / 1e9
    sample = ("the first %d elements of one tensor of the batch per step (of %d), all four operations, single thread; "
              "host has %d cores" % (m, 1 << LOG2N, os.cpu_count()))
    line = {"impl": "reference", "metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(1e3 * total / args.steps, 3),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": workload_config(),
            "cpu_baseline": {"value": round(value, 4), "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": round(value, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line))


# ------------------------------------------------------------------------------------------
class Batch:
    """The batch one step passes over: `count` tensors of the headline workload with their pre-activations."""

    def __init__(self, dev, count: int):
        import torch
        from paper_2110_15362_b200 import binding as B
        from paper_2110_15362_b200 import workloads as W
        self.B, self.dev, self.n = B, dev, 1 << LOG2N
        n = self.n
        free, _ = torch.cuda.mem_get_info(dev)
        room = int((free - (16 << 30)) // (8 * n))                      # two fp32 tensors each
        self.count = max(1, min(count, room))
        self.x, self.pre = [], []
        for t in range(self.count):
            x = W.cfg3_iid(n, ZEROS, 100 + t, dev)
            self.x.append(x)
            self.pre.append(torch.where(x != 0, x, torch.full((), -1.0, device=dev)))
        self.g = W.cfg2_grad(0, (n,), dev)
        self.out = torch.empty(n, dtype=torch.float32, device=dev)
        self.sa, self.sb = B.Stash(n, torch.float32, dev), B.Stash(n, torch.float32, dev)
        self.ws = B.new_workspace(n, dev)
        self.launches_per_step = 4 * self.count
        self.dense_bytes_per_step = 4 * self.count * 4 * n

    def step(self):
        B, sa, sb, ws = self.B, self.sa, self.sb, self.ws
        for x, pre in zip(self.x, self.pre):
            B.bt_compress(x, sa.bitmap, sa.values, sa.chunk_prefix, sa.nnz_out, ws, sa.dev_status)
            B.bt_decompress(sa.bitmap, sa.values, sa.chunk_prefix, self.out)
            B.bt_relu_fwd_compress(pre, None, sb.bitmap, sb.values, sb.chunk_prefix, sb.nnz_out, ws, sb.dev_status)
            B.bt_relu_bwd_from_bitmap(sb.bitmap, self.g, self.out)

    def check(self):
        """The last tensor of a step, after the step: both stashes against torch, the gradient against torch."""
        import torch
        x, pre = self.x[-1], self.pre[-1]
        torch.cuda.synchronize()
        nnz = int(torch.count_nonzero(x).item())
        assert self.sa.status == self.B.BT_OK and self.sb.status == self.B.BT_OK
        assert self.sa.nnz == nnz and self.sb.nnz == nnz
        assert torch.equal(self.sa.values[:nnz], x[x != 0]) and torch.equal(self.sb.values[:nnz], x[x != 0])
        assert torch.equal(self.sa.bitmap, self.sb.bitmap)
        want = torch.where(pre > 0, self.g, torch.zeros((), device=self.dev))
        assert torch.equal(self.out.view(torch.int32), want.view(torch.int32))
        return nnz


def run_e2e(batch: Batch, steps: int = 3, warmup: int = 1, workers: int = 4):
    """The same four operations through the host-buffer entry points of the C ABI: a tensor, its pre-activation and
    the gradient start in pinned host memory, both stashes, the restored tensor and the input gradient end there;
    the host<->device copies happen inside the calls, inside the timed region.

    The calls are synchronous (each returns with its results on the host), so `workers` host threads, each with its
    own stream, staging area and output buffers, work on one tensor each at the same time: one call's upload
    overlaps another's download.  A step is `workers` tensors through the four operations."""
    from concurrent.futures import ThreadPoolExecutor
    import torch
    B, n, dev = batch.B, batch.n, batch.dev
    pin = lambda t: t.cpu().pin_memory()                                 # noqa: E731
    h_x, h_pre, h_g = pin(batch.x[0]), pin(batch.pre[0]), pin(batch.g)   # read-only inputs, shared by the workers
    res = []
    for _ in range(workers):
        res.append(dict(stream=torch.cuda.Stream(device=dev),
                        staging=torch.empty(B.bt_host_staging_bytes(n, torch.float32), dtype=torch.uint8, device=dev),
                        bitmap=torch.empty((n + 31) // 32, dtype=torch.int32).pin_memory(),
                        values=torch.empty(n, dtype=torch.float32).pin_memory(),
                        prefix=torch.empty((n + 4095) // 4096, dtype=torch.int64).pin_memory(),
                        nnz=torch.zeros(1, dtype=torch.int64).pin_memory(),
                        back=torch.empty(n, dtype=torch.float32).pin_memory()))

    def one(r):
        torch.cuda.set_device(dev)
        s = r["stream"]
        B.bt_compress_host(h_x, r["bitmap"], r["values"], r["prefix"], r["nnz"], r["staging"], stream=s)
        B.bt_decompress_host(r["bitmap"], r["values"], r["prefix"], int(r["nnz"].item()), r["back"], r["staging"], stream=s)
        B.bt_relu_fwd_compress_host(h_pre, None, r["bitmap"], r["values"], r["prefix"], r["nnz"], r["staging"], stream=s)
        B.bt_relu_bwd_from_bitmap_host(r["bitmap"], h_g, r["back"], r["staging"], stream=s)

    with ThreadPoolExecutor(max_workers=workers) as ex:
        for _ in range(warmup):
            list(ex.map(one, res))
        torch.cuda.synchronize()
        nnz = int(res[0]["nnz"].item())
        comp = B.bt_compressed_bytes(n, nnz, torch.float32)
        h2d = workers * (4 * n + comp + 4 * n + (4 * ((n + 31) // 32) + 4 * n))
        d2h = workers * ((comp + 12) + 4 * n + (comp + 12) + 4 * n)
        t0 = time.perf_counter()
        for _ in range(steps):
            list(ex.map(one, res))                                       # every call has synchronised its stream
        torch.cuda.synchronize()
        ms = (time.perf_counter() - t0) * 1e3 / steps
    want = torch.where(h_pre > 0, h_g, torch.zeros(()))
    for r in res:
        assert torch.equal(r["back"].view(torch.int32), want.view(torch.int32)), "end-to-end result differs"
    return {"ms_per_step": ms, "steps": steps, "h2d": h2d, "d2h": d2h, "dense_bytes_per_step": workers * 4 * 4 * n,
            "workers": workers}


def report(line: dict, rows: list) -> None:
    """The line on standard output, the per-kernel rows on standard error: with its 163 rows the line took 47 KB, more than is
    kept by a reader of the end of a program's output."""
    for r in rows:
        print(json.dumps(r), file=sys.stderr)
    sys.stderr.flush()
    line["roofline"]["rows_on_stderr"] = len(rows)
    print(json.dumps(line), flush=True)


def run_ours(args):
    import torch
    import torch.distributed as dist
    from paper_2110_15362_b200 import binding as B

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the codec has no CPU path")
    B.lib()                                                              # fails loudly if the library is missing
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    peak, peak_kind = measured_peak_gbs()

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    batch = Batch(dev, args.tensors)
    sampler = ClockSampler(local)
    sampler.start()
    for _ in range(max(args.warmup, 3)):
        batch.step()
    nnz = batch.check()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0 = time.time()
    e0.record()
    for _ in range(args.steps):
        batch.step()
    e1.record()
    barrier()
    t1 = time.time()
    sampler.stop()
    ms_step = max_over_ranks(e0.elapsed_time(e1) / args.steps, world, dev)
    clocks = sampler.summary(t0, t1)
    value = whole_job_value(batch.dense_bytes_per_step, world, ms_step)

    line = {"metric": METRIC, "value": round(value, 2), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": round(ms_step, 4), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic", "gpu_launches": batch.launches_per_step * args.steps,
            "config": workload_config(),
            "run": {"tensors_per_step": batch.count, "launches_per_step": batch.launches_per_step,
                    "dense_equivalent_bytes_per_step": batch.dense_bytes_per_step, "zero_fraction_measured": round(1 - nnz / batch.n, 4),
                    "launch": "one stream, four launches per tensor, no CUDA graph, no CTA budget",
                    "l2": "every tensor is 1 GiB and the batch %d GiB: inputs exceed the 126 MB L2, no flush between steps"
                          % (2 * batch.count),
                    "parallelism": "single" if world == 1 else "replicas x%d, no collective on the data path" % world},
            "clocks": clocks}

    if rank == 0:
        rows, extras = ([], {}) if args.no_kernels else kernel_table(dev, peak)
        graded = [r for r in rows if r["kernel"] in OPS and r.get("launches", 1) == 1 and r["algorithmic_bytes"] >= 256e6]
        if graded:
            low = min(graded, key=lambda r: r["frac_of_measured"])
            per_el, src = NCU_DRAM_BYTES_PER_ELEMENT.get((low["dtype"], low["kernel"] + ("+y" if low.get("dense_output") else "")), (None, None))
            line["roofline"] = {"bound": "hbm", "kernel": low["kernel"], "dtype": low["dtype"], "config": low["config"],
                                "tensor": low.get("tensor"), "dense_output": low.get("dense_output"),
                                "achieved": low["gbs"], "peak": peak, "unit": "GB/s", "frac": low["frac_of_measured"],
                                "peak_kind": peak_kind, "frac_of_8tbs": low["frac_of_8tbs"],
                                "algorithmic_bytes_per_launch": low["algorithmic_bytes"], "avg_launch_ms": low["median_ms"],
                                "traffic": None if per_el is None else round(per_el * low["elements"]),
                                "traffic_source": src,
                                "how": "the lowest fraction among the five graded calls on tensors of at least 256 MB; "
                                       "each row: CUDA events around one launch, L2 flushed before it, median of 9"}
        else:
            # without the table: the headline tensor's own four kernels, timed one by one
            T = KernelTimer(dev, peak)
            codec_rows(T, B, "cfg3_iid", batch.x[0], batch.pre[0], batch.g, ZEROS, ops=("compress", "decompress", "fwd", "bwd"))
            low = min(T.rows, key=lambda r: r["frac_of_measured"])
            line["roofline"] = {"bound": "hbm", "kernel": low["kernel"], "dtype": "f32", "achieved": low["gbs"], "peak": peak,
                                "unit": "GB/s", "frac": low["frac_of_measured"], "peak_kind": peak_kind, "traffic": None}
            rows = T.rows
        line.update(extras)
        if not args.no_e2e:
            e = run_e2e(batch)
            line["e2e"] = {"value": round(world * e["dense_bytes_per_step"] / (e["ms_per_step"] * 1e-3) / 1e9, 3), "unit": UNIT,
                           "h2d_bytes_per_step": e["h2d"], "d2h_bytes_per_step": e["d2h"],
                           "ms_per_step": round(e["ms_per_step"], 3), "steps": e["steps"], "tensors_per_step": e["workers"],
                           "what": "the step's four operations through bt_*_host on %d tensors at a time, one host thread, "
                                   "stream and staging area each: pinned host buffers in, pinned host buffers out, copies "
                                   "inside the calls, timed on the host around the synchronous calls (rank 0's GPU; value "
                                   "scaled by the number of ranks)" % e["workers"]}
        if not args.no_cpu_baseline and world == 1:
            cal = host_sample(1 << 20)
            rate = (1 << 20) / max(oracle_four_ops(*cal), 1e-6)
            m = max(1 << 20, min(1 << LOG2N, int(rate * 15.0) // 4096 * 4096))          # about 15 s of CPU work
            sec = oracle_four_ops(*host_sample(m))
            line["cpu_baseline"] = {"value": round(len(OPS) * 4 * m / sec / 1e9, 4), "unit": UNIT, "cores": 1,
                                    "kind": "oracle", "seconds": round(sec, 2),
                                    "sample": "the first %d elements of one tensor of the batch (of %d), all four operations, "
                                              "single thread; host has %d cores" % (m, 1 << LOG2N, os.cpu_count())}
        report(line, rows)
    barrier()
    if world > 1:
        dist.destroy_process_group()


# ------------------------------------------------------------------------------------------
def run_case(args) -> int:
    """One small, seeded invocation of one kernel, for profiler captures (python bench.py --case <dtype> <op>):
    `reps` repetitions of one entry point on a tensor of 2**log2n elements (default 2**26: larger than the 126 MB L2
    and small enough for a multi-pass capture); prints the non-zero count and the device status, non-zero exit
    if the status is not BT_OK.  The 4- and 8-byte input has independent zeros of the given fraction, the
    2-byte input is the ReLU of a normal pre-activation (about half zeros)."""
    import torch
    from paper_2110_15362_b200 import binding as B
    from paper_2110_15362_b200 import workloads as W
    kind, op = args.case
    if kind not in ("f32", "f16", "bf16", "f64") or op not in CASE_OPS:
        raise SystemExit("--case <f32|f16|bf16|f64> <%s>" % "|".join(CASE_OPS))
    dev = torch.device("cuda")
    if op in ("batch", "batch_restore"):                                 # the 17 ResNet-18 layers at batch 32, one launch
        tdt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "f64": torch.float64}[kind]
        acts = [torch.clamp_min(W.cfg2_preact(i, shape, dev), 0.0).reshape(-1).to(tdt) for i, shape, _ in W.iter_layers(W.resnet18_shapes(32))]
        sts = [B.Stash(a.numel(), tdt, dev) for a in acts]
        outs = [torch.empty_like(a) for a in acts]
        ws = torch.empty(B.bt_batch_workspace_bytes([a.numel() for a in acts]), dtype=torch.uint8, device=dev)
        items, ritems = B.batch_items(acts, sts), B.batch_items(outs[::-1], sts[::-1], outs[::-1])
        for _ in range(args.reps):
            B.bt_compress_batch(items, tdt, ws)
            if op == "batch_restore":
                B.bt_decompress_batch(ritems, tdt)
        torch.cuda.synchronize()
        ok = all(st.status == B.BT_OK for st in sts) and (op == "batch" or all(torch.equal(o, a) for o, a in zip(outs, acts)))
        print("tensors", len(acts), "nnz", sum(st.nnz for st in sts), "ok", ok)
        return 0 if ok else 1
    n = 1 << args.log2n
    if kind == "f32":
        x = W.prune_preact(n, dev) if op == "prune" else W.cfg3_iid(n, args.zeros, 2, dev)
    elif kind == "f64":
        x = W.cfg3_iid(n, args.zeros, 3, dev).double()
    else:
        x = torch.relu(W.cfg4_preact(0, (n,), kind, dev))
    st = B.Stash(n, x.dtype, dev)
    ws = B.new_workspace(n, dev)
    d = torch.empty_like(x)
    v16 = torch.empty(n, dtype=torch.float16, device=dev) if op in ("narrow", "widen") else None
    d32 = torch.empty(n, dtype=torch.float32, device=dev) if op == "widen" else None

    def compress():
        B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)

    if op in ("maxpool", "maxpool_bwd"):                                 # the tensor seen as rows of 256 elements
        xp = x.view(-1, n // 256 // 64, 256)
        yp = torch.empty(xp.shape[0], xp.shape[1] // 2, 128, dtype=x.dtype, device=dev)
        codes = torch.empty((yp.numel() + 15) // 16, dtype=torch.int32, device=dev)
        for _ in range(args.reps):
            B.bt_maxpool2x2_fwd(xp, yp, codes)
            if op == "maxpool_bwd":
                B.bt_maxpool2x2_bwd(codes, yp, d.view_as(xp))
        torch.cuda.synchronize()
        print("pooled", tuple(yp.shape), "non-zero", int(torch.count_nonzero(yp)))
        return 0
    for _ in range(args.reps):
        if op == "compress":
            compress()
        elif op == "relu":
            B.bt_relu_fwd_compress(x, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        elif op == "relu_y":
            B.bt_relu_fwd_compress(x, d, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        elif op == "prune":
            B.bt_prune_fwd_compress(x, args.tau, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        elif op == "narrow":                                             # float32 tensor, float16 stashed values
            B.bt_compress_narrow(x, st.bitmap, v16, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        elif op == "widen":
            B.bt_compress_narrow(x, st.bitmap, v16, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
            B.bt_decompress_widen(st.bitmap, v16, st.chunk_prefix, d32)
        elif op == "relu6":
            B.bt_relu6_fwd_compress(x, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
        elif op == "relu6_bwd":
            B.bt_relu6_fwd_compress(x, None, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
            B.bt_relu6_bwd_from_stash(st.bitmap, st.values, st.chunk_prefix, x, d)
        elif op in ("mask", "mask_y"):
            compress()
            B.bt_mask_compress(x, st.bitmap, st.chunk_prefix, d if op == "mask_y" else None, st.values)
        elif op == "decompress":
            compress()
            B.bt_decompress(st.bitmap, st.values, st.chunk_prefix, d)
        else:
            compress()
            B.bt_relu_bwd_from_bitmap(st.bitmap, x, d)
    torch.cuda.synchronize()
    print("nnz", st.nnz, "status", st.status)
    return 0 if st.status == B.BT_OK else 1


def main():
    args = parse_args()
    if args.case:
        sys.exit(run_case(args))
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
