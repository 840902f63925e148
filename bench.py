"""Throughput benchmark of the fused PIC decode synthesis on GB300.

One step = one pass of the whole hot path (dequantise, upsample, concatenate,
MLP, clamp) over one batch of synthetic input: by default the 64-image
throughput workload (64 independent 768x512 images, 7 levels x 1 channel,
7-64-64-3 ReLU, fp16 weights) decoded by one ``pic_decode_batch`` call.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload c5]
                    [--precision fp16_tc|fp32] [--impl ours|reference]
                    [--stage decode|izpr|idct|pipeline] [--chunk 64]

Prints one JSON line (rank 0).  ``value`` is decoded megapixels/s over all
ranks (weak scaling: each rank decodes its own batch; no collective on the
data path).  ``--impl reference`` times the fp64 CPU oracle on the host cores
on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2609_09020_gb300 import workloads as wk  # noqa: E402

METRIC = "decoded megapixels/s and images/s at 1 GB300; % of binding roofline"
UNIT = "MP/s"
SM_COUNT = 152
SM_MAX_MHZ = 2070.0
FP32_LANES_PER_SM = 128


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return {"hbm_gbs": d["hbm_gbs"], "bf16_tflops": d["bf16_tflops"],
                "bf16_tflops_sustained": d.get("bf16_tflops_sustained"), "source": "measured"}
    except (OSError, KeyError, ValueError):
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0,
                "source": "fallback"}


def fp32_peak_tflops():
    """FP32 CUDA-core peak: SMs x 128 FMA lanes x 2 FLOP x max SM clock."""
    return SM_COUNT * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12


def algorithmic(wl: wk.Workload, batch: int):
    """Per-launch algorithmic work: unpadded MLP FLOPs and the bytes the decode
    must move at least once (int32 latents, weights, steps, fp32 RGB)."""
    px = batch * wl.H * wl.W
    flops = 2.0 * wl.macs_per_pixel * px
    wbytes = 2 if wl.weight_dtype == "fp16" else 4
    nbytes = batch * (wl.n_latents * 4 + wl.n_params * wbytes + wl.L * 4 + 3 * wl.H * wl.W * 4)
    return flops, nbytes


# FP32-pipe operations of one GELU evaluation in the kernels (pic_gelu.cuh):
# six Horner steps, the saturating subtraction and the last multiply-add; the
# power of two runs on the special-function unit, the two comparisons beside
# the FP32 pipe.
GELU_OPS = 6 + 1 + 1
# Those of the rational function that the kernels evaluated before (z^2, the
# Horner steps of P (5) and Q (4), P * (1 / Q), the saturating fma and z * Phi).
GELU_FP32_OPS = 4 + 5 + 4


def march_tensor_macs_per_px(wl: wk.Workload) -> int:
    """MACs the tensor cores execute per pixel in the row-marching kernels (the
    ones staging "auto" picks): layer 0 (K = the hi and lo features and the
    constant 1, round16), hidden layers and the output layer (where it is not in
    fp32 on the CUDA cores) with the hi and lo halves of K.  Nets wider than 40
    run on N = 64 tiles, each bias that is no column of layer 0 as one K = 16
    step and the output layer as N = 16; narrower ones at their own width,
    biases free, the output layer as N = 8."""
    d0, width = wl.dims[0], max(wl.dims[1:-1])
    k1 = (4 * ((d0 + 1) // 2) + 15) // 16 * 16
    bias_column = d0 % 2 == 1 or 4 * ((d0 + 1) // 2) < k1
    n, bias, out = (64, 16, 16) if width > 40 else ((width + 7) // 8 * 8, 0, 8)
    mac = (k1 + (0 if bias_column else bias)) * n
    mac += (len(wl.dims) - 3) * (2 * n + bias) * n
    return mac + (2 * n * out if tc_output_on_tensor_cores(wl) else 0)


def executed_tensor_macs_per_px(wl: wk.Workload) -> int:
    """MACs the tensor cores execute per pixel in the per-tile kernels (staging
    "copies" and "tma"): layer 0 (K = round16(2 D0 + 1),
    N = round16 of the width), hidden layers and (for wide, shallow nets) the
    output layer (N = 16), with the hi and lo halves of K plus one K = 16 bias
    step each."""
    def r16(v):
        return (v + 15) // 16 * 16
    n_pad = r16(max(wl.dims[1:-1]))
    mac = r16(2 * wl.dims[0] + 1) * n_pad
    mac += (len(wl.dims) - 3) * (2 * n_pad + 16) * n_pad
    if tc_output_on_tensor_cores(wl):
        mac += (2 * n_pad + 16) * 16
    return mac


def tc_output_on_tensor_cores(wl: wk.Workload) -> bool:
    """The tensor-core kernels run the output layer as an MMA only for wide, shallow
    nets (width > 32 and fewer than 4 layers); else on the CUDA cores."""
    n_pad = (max(wl.dims[1:-1]) + 15) // 16 * 16
    return n_pad > 32 and len(wl.dims) - 1 < 4


def alu_ops_per_px(wl: wk.Workload, precision: str, gelu_ops: int = GELU_FP32_OPS) -> int:
    """Activation-inclusive CUDA-core work per pixel (FP32-pipe operations):
    every hidden activation (GELU at gelu_ops, GELU_OPS in the kernels; ReLU is
    folded into a conversion or runs beside the FP32 pipe), plus on the tensor
    path the hi/lo split of every hidden value that feeds an MMA (2 per value)
    and the output layer where it runs on the CUDA cores (one FMA per weight),
    plus on the fp32 path every MLP MAC."""
    hidden = list(wl.dims[1:-1])
    act = gelu_ops if wl.act == "gelu" else 0
    ops = act * sum(hidden)
    if precision == "fp16_tc":
        if tc_output_on_tensor_cores(wl):
            ops += 2 * sum(hidden)
        else:
            ops += 2 * sum(hidden[:-1]) + 3 * hidden[-1]
    else:
        ops += wl.macs_per_pixel
    return ops


def roofline_for(wl: wk.Workload, precision: str, B: int, ms: float, peaks: dict,
                 fp32_tflops: float, fp32_src: str, staging: str = "auto") -> dict:
    """The roofline of one decode launch of B images that took ms with the kernel
    that staging picks: the binding
    of (unpadded MLP FLOPs at the path's pipe peak, algorithmic bytes at the
    HBM peak), and beside it the activation-inclusive ALU bound."""
    flops, nbytes = algorithmic(wl, B)
    t_s = ms * 1e-3
    px = B * wl.H * wl.W
    if precision == "fp16_tc":
        peak_tf = peaks["bf16_tflops"]  # fp16 dense tensor rate = bf16 rate
        roof = {"bound": "tensor", "achieved": flops / t_s / 1e12, "peak": peak_tf,
                "unit": "TFLOP/s", "peak_source": f"bf16 dense burst, {peaks['source']}"}
    else:
        peak_tf = fp32_tflops
        roof = {"bound": "alu", "achieved": flops / t_s / 1e12, "peak": peak_tf,
                "unit": "TFLOP/s", "peak_source": fp32_src}
    t_pipe = flops / (peak_tf * 1e12)
    t_hbm = nbytes / (peaks["hbm_gbs"] * 1e9)
    if t_hbm > t_pipe:
        roof.update({"bound": "hbm", "achieved": nbytes / t_s / 1e9, "peak": peaks["hbm_gbs"],
                     "unit": "GB/s", "peak_source": f"copy bandwidth, {peaks['source']}"})
    roof["frac"] = roof["achieved"] / roof["peak"]
    roof["algorithmic_flops_per_launch"] = flops
    if precision == "fp16_tc":
        macs = march_tensor_macs_per_px if staging == "auto" else executed_tensor_macs_per_px
        roof["executed_tensor_flops_per_launch"] = 2.0 * macs(wl) * px
    roof["algorithmic_bytes_per_launch"] = nbytes
    roof["binding_time_us"] = max(t_pipe, t_hbm) * 1e6
    roof["avg_launch_us"] = ms * 1e3
    # activation-inclusive ALU bound (FP32 pipe at the measured FMA rate;
    # one operation = one lane-op, half an FMA's two FLOPs)
    ops = alu_ops_per_px(wl, precision, GELU_OPS)
    t_alu = ops * px / (fp32_tflops * 1e12 / 2)
    t_bind = max(t_pipe, t_hbm, t_alu)
    roof["alu_bound"] = {"ops_per_px": ops,
                         "gelu_evals_per_launch": px * sum(wl.dims[1:-1]) if wl.act == "gelu" else 0,
                         "t_alu_us": t_alu * 1e6, "binding_time_incl_alu_us": t_bind * 1e6,
                         "frac_incl_alu": t_bind / t_s}
    return roof


KERNEL_SOURCES = {
    "idct": ["k_idct.cu"],
    "izpr": ["k_izpr.cu"],
    "tc_march": ["k_tcmarch.cuh", "march.cuh", "tc_ptx.cuh", "pic_common.cuh", "pic_gelu.cuh", "pic_kernels.h"],
    "tc_strip": ["k_strip.cuh", "march.cuh", "tc_ptx.cuh", "pic_common.cuh", "pic_gelu.cuh", "pic_kernels.h"],
    "tc_tile": ["k_tc.cuh", "tc_ptx.cuh", "pic_common.cuh", "pic_gelu.cuh", "pic_kernels.h"],
    "fp32": ["k_fp32.cuh", "pic_common.cuh", "pic_gelu.cuh", "pic_kernels.h"],
}


def kernel_sources(kernel_name: str):
    """The source files that a decode kernel, by its name, is compiled from."""
    if kernel_name.startswith("tc"):
        if kernel_name.endswith(("_tile", "_tma", "_lo8")):
            return KERNEL_SOURCES["tc_tile"]
        dims = [int(d) for d in kernel_name.split("_")[1].split("x")]
        return KERNEL_SOURCES["tc_strip" if max(dims[1:-1]) <= 40 else "tc_march"]
    return KERNEL_SOURCES[next((k for k in ("idct", "izpr") if kernel_name.startswith(k)), "fp32")]


def kernel_source_hash(kernel_name: str) -> str:
    """Hash of the source files a decode kernel is compiled from."""
    files = kernel_sources(kernel_name)
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2609_09020_gb300", "csrc")
    for fn in files:
        with open(os.path.join(csrc, fn), "rb") as f:
            h.update(fn.encode() + f.read())
    return h.hexdigest()[:16]


def recorded_traffic(kernel_name: str, workload: str):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current kernel sources; else None."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        return None
    e = rec.get(f"{kernel_name}/{workload}")
    if not e or e.get("source_hash") != kernel_source_hash(kernel_name):
        return None
    return e.get("dram_bytes_per_launch")


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            time.sleep(0.3)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.lines = []
        if self.proc is not None:
            time.sleep(0.15)
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        mhz, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in getattr(self, "lines", []):
            f = [s.strip() for s in line.split(",")]
            if len(f) < 9:
                continue
            try:
                mhz.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not mhz:
            return {"sm_mhz": None, "sm_max_mhz": mx, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(mhz), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(mhz)}


def cpu_baseline(wl: wk.Workload, x: wk.Inputs, precision: str, budget_s: float,
                 single_thread: bool = True):
    """The fp64 oracle, as it stands, on the host cores: full images decoded
    one after another until about budget_s seconds have passed; then, with
    single_thread, the same on one thread for a third of that."""
    import oracle
    orc = oracle.load()
    cores = os.cpu_count() or 1
    w = x.weights_for(precision)
    n, t0 = 0, time.perf_counter()
    while True:
        b = n % x.latents.shape[0]
        orc.decode(x.latents[b], x.steps[b].astype(np.float64), w[b].astype(np.float64), wl.H,
                   wl.W, wl.L, wl.C, wl.dims, wl.act, nthreads=cores)
        n += 1
        el = time.perf_counter() - t0
        if el >= budget_s:
            break
    mp = n * wl.H * wl.W / 1e6
    r = {"value": mp / el, "unit": UNIT, "cores": cores, "kind": "oracle",
         "sample": f"{n} full {wl.W}x{wl.H} image(s) of workload {wl.name} in {el:.1f} s "
                   f"(fp64 C oracle, OpenMP over rows, {cores} threads)",
         "images_per_s": n / el}
    if not single_thread:
        return r
    # the same oracle on one thread, for a third of the budget
    n1, t1 = 0, time.perf_counter()
    while True:
        b = n1 % x.latents.shape[0]
        orc.decode(x.latents[b], x.steps[b].astype(np.float64), w[b].astype(np.float64), wl.H,
                   wl.W, wl.L, wl.C, wl.dims, wl.act, nthreads=1)
        n1 += 1
        el1 = time.perf_counter() - t1
        if el1 >= budget_s / 3:
            break
    r["single_thread"] = {"value": n1 * wl.H * wl.W / 1e6 / el1, "unit": UNIT,
                          "sample": f"{n1} full image(s) in {el1:.1f} s on one thread"}
    return r


# ---- the multi-process (weak-scaling) bookkeeping: each rank decodes its
# own batch, nothing is exchanged on the data path, the timing is the max
# over ranks and the rate counts every rank's pixels.
def shard_workload(wl: wk.Workload, rank: int) -> wk.Workload:
    """Rank r decodes its own batch: the workload's image seeds + 1000 r."""
    return wl.replace(seeds=tuple(s + 1000 * rank for s in wl.seeds)) if rank else wl


def max_over_ranks(v: float, world: int, device=None) -> float:
    """The largest of the ranks' values (a MAX all-reduce; v itself at N = 1)."""
    if world <= 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(px_per_rank: int, world: int, ms: float) -> float:
    """Decoded megapixels/s over all ranks for a step that took ms (the max)."""
    return world * px_per_rank / (ms * 1e-3) / 1e6


def workload_desc(wl: wk.Workload, precision: str):
    mlp = "-".join(str(d) for d in wl.dims) + " " + wl.act
    return {"workload": f"{wl.name}: {wl.B} x {wl.W}x{wl.H}, {wl.L} levels x {wl.C} ch, MLP {mlp}, "
                        f"{wl.weight_dtype} weights, {precision} path",
            "images": wl.B, "H": wl.H, "W": wl.W, "levels": wl.L, "channels": wl.C,
            "mlp": mlp, "precision": precision}


def run_reference(args, wl, precision, rank):
    if rank != 0:
        return
    x = wk.make_inputs(wl, batch=min(wl.B, 4))
    budget = args.ref_step_s
    for _ in range(args.warmup):
        cpu_baseline(wl, x, precision, 0.0, single_thread=False)
    vals, imgs, samples = [], [], []
    t0 = time.perf_counter()
    for _ in range(args.steps):
        r = cpu_baseline(wl, x, precision, budget, single_thread=False)
        vals.append(r["value"])
        imgs.append(r["images_per_s"])
        samples.append(r["sample"])
    el = time.perf_counter() - t0
    v = statistics.median(vals)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * el / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic (seeded, workload-shaped)",
            "config": {**workload_desc(wl, precision), "parallelism": "host cores"},
            "images_per_s": statistics.median(imgs),
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": os.cpu_count() or 1,
                             "kind": "oracle",
                             "sample": f"each step about {budget:g} s of whole images; last "
                                       f"step: {samples[-1]}"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# Stage benchmarks: the decoder's stages before the synthesis (Fig. 1: iZpR,
# then dequantisation + iDCT + un-patchify), alone and chained with it, on
# the 64-image workload's 524,288 patches.  One step = one pass over the
# whole batch.
STAGE_METRIC = {
    "izpr": ("inverse ZpR (Algorithm 1): 8x8 blocks/s at 1 GB300; % of HBM roofline", "Mblocks/s"),
    "idct": ("dequantise + 8x8 iDCT + un-patchify: 8x8 blocks/s at 1 GB300; % of HBM roofline",
             "Mblocks/s"),
    "pipeline": ("decoded megapixels/s from ZpR symbols (iZpR + iDCT + synthesis) at 1 GB300",
                 "MP/s"),
    "fuse": ("modulation fusion (App. A): per-image decoder weight blobs/s at 1 GB300", "images/s"),
    "huffman": ("Huffman decoding (image-specific tables, self-synchronising): symbols/s at 1 GB300; "
                "% of HBM roofline", "Msymbols/s"),
    "bitstream": ("decoded megapixels/s from Huffman-coded bitstreams (Huffman + iZpR + iDCT + "
                  "synthesis) at 1 GB300", "MP/s"),
}


def run_bitstream_stages(args):
    """Huffman decoding of the 64-image batch's ZpR streams (one table per
    image), alone ("huffman") or followed by iZpR, iDCT and the synthesis
    ("bitstream": the whole decoder after the header)."""
    import torch
    from paper_2609_09020_gb300 import build, pic
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    build.build()
    stage = args.stage
    wl = wk.WORKLOADS["c5"]
    B = wl.B
    h = wk.huffman_streams(wl)
    dx = wk.make_dct_inputs(wl)
    n_blk, eob, p = h["n_blocks"], h["eob"], h["p"]
    n_sym = int(h["sym_off"][-1])
    stream = torch.cuda.current_stream(dev)
    sp = stream.cuda_stream
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    words, word_off, n_bits = t(h["words"].view(np.int32)), t(h["word_off"]), t(h["n_bits"])
    tv, tl, sym_off = t(h["tab_value"]), t(h["tab_len"]), t(h["sym_off"])
    syms = torch.empty(n_sym, dtype=torch.int32, device=dev)
    hwb = pic.pic_huffman_workspace_bytes(words.numel(), B, p)
    hws = torch.empty(hwb, dtype=torch.uint8, device=dev)
    full = stage == "bitstream"
    if full:
        coeffs = torch.empty((B * n_blk, 64), dtype=torch.int32, device=dev)
        offsets = torch.empty(B * n_blk, dtype=torch.int64, device=dev)
        zwb = pic.pic_izpr_workspace_bytes(n_sym)
        zws = torch.empty(zwb, dtype=torch.uint8, device=dev)
        steps_t = t(dx.steps)
        lat = torch.empty((B, wl.n_latents), dtype=torch.float32, device=dev)
        wts = t(dx.weights_for("fp16_tc"))
        out = torch.empty((B, 3, wl.H, wl.W), dtype=torch.float32, device=dev)
        dec = pic.Decoder.for_workload(wl, "fp16_tc", max_batch=B, latent="fp32")
        dec.check_buffers(B, wl.H, wl.W, latents=lat, steps=None, weights=wts, out=out)

    def huff():
        rc = pic.pic_huffman_decode(words.data_ptr(), words.numel(), word_off.data_ptr(),
                                    n_bits.data_ptr(), B, tv.data_ptr(), tl.data_ptr(), tv.shape[1],
                                    p, sym_off.data_ptr(), syms.data_ptr(), hws.data_ptr(), hwb, sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_huffman_decode")

    def rest():
        rc = pic.pic_izpr_decode(syms.data_ptr(), n_sym, eob, B * n_blk, coeffs.data_ptr(),
                                 offsets.data_ptr(), zws.data_ptr(), zwb, sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_izpr_decode")
        rc = pic.pic_idct_unpatchify(coeffs.data_ptr(), steps_t.data_ptr(), B, wl.H, wl.W, wl.L,
                                     wl.C, lat.data_ptr(), sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_idct_unpatchify")
        dec.decode_batch(lat, None, wts, wl.H, wl.W, out, stream=stream, B=B, check=False)

    def one_step():
        huff()
        if full:
            rest()

    for _ in range(max(args.warmup, 3)):
        one_step()
    torch.cuda.synchronize()
    if pic.pic_huffman_status(hws.data_ptr(), sp) != pic.PIC_OK:
        raise RuntimeError("Huffman streams reported malformed")
    if not torch.equal(syms.cpu(), torch.from_numpy(h["symbols"])):
        raise RuntimeError("Huffman decode differs from the generated symbols")
    if full:
        if pic.pic_izpr_status(zws.data_ptr(), sp) != pic.PIC_OK:
            raise RuntimeError("ZpR streams reported malformed")
        dec.check(stream)
    with ClockSampler(0) as clk:
        ms = _event_time(one_step, args.steps, stream, torch)
    stage_ms = {"huffman": _event_time(huff, args.steps, stream, torch)}
    serial = None
    if full:
        dec.check(stream)
        stage_ms["izpr+idct+synthesis"] = ms - stage_ms["huffman"]
        # The paper's protocol (App. C): one image at a time, synchronised
        # before and after -- its whole decode after the header, per image.
        n_ser = min(B, 16)
        per = []
        for b in range(n_ser):
            w0, w1 = int(h["word_off"][b]), int(h["word_off"][b + 1])
            s0, s1 = int(h["sym_off"][b]), int(h["sym_off"][b + 1])
            one = {"words": t(h["words"][w0:w1].view(np.int32)),
                   "word_off": t(np.array([0, w1 - w0], np.int64)), "n_bits": t(h["n_bits"][b:b + 1]),
                   "tv": t(h["tab_value"][b:b + 1]), "tl": t(h["tab_len"][b:b + 1]),
                   "sym_off": t(np.array([0, s1 - s0], np.int64)), "steps": t(dx.steps[b:b + 1]),
                   "w": t(dx.weights_for("fp16_tc")[b:b + 1])}
            dec.check_buffers(1, wl.H, wl.W, latents=lat[:1], steps=None, weights=one["w"],
                              out=out[:1])
            hwb1 = pic.pic_huffman_workspace_bytes(one["words"].numel(), 1, p)
            hws1 = torch.empty(hwb1, dtype=torch.uint8, device=dev)

            def run_one():
                rc = pic.pic_huffman_decode(one["words"].data_ptr(), one["words"].numel(),
                                            one["word_off"].data_ptr(), one["n_bits"].data_ptr(), 1,
                                            one["tv"].data_ptr(), one["tl"].data_ptr(), one["tv"].shape[1],
                                            p, one["sym_off"].data_ptr(), syms.data_ptr(), hws1.data_ptr(),
                                            hwb1, sp)
                if rc != pic.PIC_OK:
                    raise pic.PicError(rc, "pic_huffman_decode")
                rc = pic.pic_izpr_decode(syms.data_ptr(), s1 - s0, eob, n_blk, coeffs.data_ptr(),
                                         offsets.data_ptr(), zws.data_ptr(), zwb, sp)
                if rc != pic.PIC_OK:
                    raise pic.PicError(rc, "pic_izpr_decode")
                rc = pic.pic_idct_unpatchify(coeffs.data_ptr(), one["steps"].data_ptr(), 1, wl.H, wl.W,
                                             wl.L, wl.C, lat.data_ptr(), sp)
                if rc != pic.PIC_OK:
                    raise pic.PicError(rc, "pic_idct_unpatchify")
                dec.decode_batch(lat[:1], None, one["w"], wl.H, wl.W, out[:1], stream=stream, B=1,
                                 check=False)

            run_one()  # warm this image's buffers
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            run_one()
            torch.cuda.synchronize(dev)
            per.append(time.perf_counter() - t0)
        dec.check(stream)
        serial = {"ms_per_image": 1e3 * float(np.mean(per)), "images": n_ser,
                  "note": "one image per call, synchronised before and after (the paper's protocol; "
                          "host clock): Huffman, iZpR, iDCT, synthesis"}
    peaks = load_peaks()
    hbytes = 4 * words.numel() + 8 * tv.numel() + 4 * n_sym + 24 * B
    t_h = stage_ms["huffman"] * 1e-3
    roof = {"bound": "hbm", "achieved": hbytes / t_h / 1e9, "peak": peaks["hbm_gbs"],
            "unit": "GB/s", "peak_source": f"copy bandwidth, {peaks['source']}",
            "kernel": "huff_decode (one call)", "avg_launch_us": t_h * 1e6,
            "traffic": None, "algorithmic_bytes_per_launch": hbytes}
    roof["frac"] = roof["achieved"] / roof["peak"]
    if full:
        value, unit = B * wl.H * wl.W / (ms * 1e-3) / 1e6, "MP/s"
        roof["note"] = "roofline of the Huffman stage; the synthesis dominates the step"
    else:
        value, unit = n_sym / (ms * 1e-3) / 1e6, "Msymbols/s"
    e2e = None
    if not args.no_e2e:
        src_h = torch.from_numpy(h["words"].view(np.int32)).pin_memory()
        res_d = out if full else syms
        res_h = torch.empty(res_d.shape, dtype=res_d.dtype).pin_memory()

        def e2e_step():
            words.copy_(src_h, non_blocking=True)
            one_step()
            res_h.copy_(res_d, non_blocking=True)
            torch.cuda.current_stream().synchronize()

        e2e_step()
        k = max(3, min(args.steps, 10))
        t0 = time.perf_counter()
        for _ in range(k):
            e2e_step()
        el = (time.perf_counter() - t0) / k
        units = B * wl.H * wl.W / 1e6 if full else n_sym / 1e6
        e2e = {"value": units / el, "unit": unit,
               "h2d_bytes_per_step": int(src_h.numel() * 4),
               "d2h_bytes_per_step": int(res_h.numel() * res_h.element_size()),
               "ms_per_step": 1e3 * el}
    cpu = None
    if not args.no_cpu_baseline:
        import oracle
        orc = oracle.load()
        n, t0 = 0, time.perf_counter()
        while time.perf_counter() - t0 < min(args.cpu_budget_s, 10.0):
            b = n % B
            m = int(np.count_nonzero(h["tab_len"][b]))
            orc.huffman_decode(h["words"][h["word_off"][b]:h["word_off"][b + 1]], h["n_bits"][b],
                               h["tab_value"][b, :m], h["tab_len"][b, :m],
                               int(h["sym_off"][b + 1] - h["sym_off"][b]))
            n += 1
        el = time.perf_counter() - t0
        per_img = n_sym / B
        cpu = {"value": n * per_img / el / 1e6, "unit": "Msymbols/s", "cores": 1, "kind": "oracle",
               "sample": f"{n} image stream(s) Huffman-decoded in {el:.1f} s (fp64-free C oracle, "
                         "bit by bit, one thread)"}
    line = {"metric": STAGE_METRIC[stage][0], "value": value, "unit": unit, "n_gpus": 1,
            "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int32 symbols" if not full else
            "int32 symbols; f32 iDCT; f16 operands (hi+lo), f32 accumulate",
            "data": "synthetic (seeded ZpR streams Huffman-coded with per-image tables)",
            "config": {"workload": f"{stage}: {B} x {wl.W}x{wl.H}, {n_sym} symbols, "
                                   f"{int(h['n_bits'].sum())} bits, p = {p}",
                       "images": B, "symbols": n_sym, "bits": int(h["n_bits"].sum()),
                       "bits_per_symbol": float(h["n_bits"].sum()) / n_sym,
                       "max_table": int(h["tab_value"].shape[1]),
                       "l2": "outputs larger than L2", "parallelism": "dp1"},
            "roofline": roof, "clocks": clk.summary(), "e2e": e2e,
            "gpu_launches": args.steps * (2 + (5 if full else 0)), "cpu_baseline": cpu,
            "stage": stage, "stage_ms": stage_ms}
    if full:
        line["images_per_s"] = B / (ms * 1e-3)
        line["serial_per_image"] = serial
    print(json.dumps(line), flush=True)


def run_fuse_stage(args):
    """64 images' decoder weights (7-64-64-3, fp16 blobs for the tensor path)
    from the shared g_s weights and each image's gamma, beta, mu, sigma."""
    import torch
    from paper_2609_09020_gb300 import build, pic
    torch.cuda.set_device(0)
    build.build()
    wl = wk.WORKLOADS["c5"]
    B, dims = wl.B, list(wl.dims)
    shared_h = wk.make_inputs(wl, batch=1).weights[0].astype(np.float32)
    cf = dims[-2]
    mod_h = wk.make_modulation(B, cf, 0)
    arch = pic.make_arch(wl.L, wl.C, dims, wl.act, "fp16_tc", max_H=wl.H, max_W=wl.W, max_batch=B)
    shared, mod = torch.from_numpy(shared_h).cuda(), torch.from_numpy(mod_h).cuda()
    out = torch.empty((B, shared_h.size), dtype=torch.float16, device="cuda")
    stream = torch.cuda.current_stream()

    def step():
        pic.fuse_modulation(arch, shared, mod, out=out, stream=stream)

    for _ in range(max(args.warmup, 3)):
        step()
    with ClockSampler(0) as clk:
        ms = _event_time(step, args.steps, stream, torch)
    peaks = load_peaks()
    nbytes = 4 * shared_h.size + 4 * mod_h.size + 2 * B * shared_h.size
    roof = {"bound": "hbm", "achieved": nbytes / (ms * 1e-3) / 1e9, "peak": peaks["hbm_gbs"],
            "unit": "GB/s", "peak_source": f"copy bandwidth, {peaks['source']}",
            "kernel": "fuse_kernel<half>", "avg_launch_us": ms * 1e3, "traffic": None,
            "algorithmic_bytes_per_launch": nbytes,
            "note": f"{nbytes / 1e6:.2f} MB per launch: launch-latency bound, far from any roofline"}
    roof["frac"] = roof["achieved"] / roof["peak"]
    e2e = None
    if not args.no_e2e:
        mod_p = torch.from_numpy(mod_h).pin_memory()
        out_p = torch.empty(out.shape, dtype=out.dtype).pin_memory()

        def e2e_step():
            mod.copy_(mod_p, non_blocking=True)
            step()
            out_p.copy_(out, non_blocking=True)
            torch.cuda.current_stream().synchronize()

        e2e_step()
        k = max(3, min(args.steps, 10))
        t0 = time.perf_counter()
        for _ in range(k):
            e2e_step()
        el = (time.perf_counter() - t0) / k
        e2e = {"value": B / el, "unit": "images/s", "h2d_bytes_per_step": int(mod_h.nbytes),
               "d2h_bytes_per_step": int(out_p.numel() * 2), "ms_per_step": 1e3 * el}
    cpu = None
    if not args.no_cpu_baseline:
        import oracle
        orc = oracle.load()
        off = sum(dims[k + 1] * (dims[k] + 1) for k in range(len(dims) - 2))
        w = shared_h[off:off + 3 * cf].astype(np.float64).reshape(3, cf)
        bb = shared_h[off + 3 * cf:].astype(np.float64)
        n, t0 = 0, time.perf_counter()
        while time.perf_counter() - t0 < min(args.cpu_budget_s, 5.0):
            g, be, mu, sd = mod_h[n % B].astype(np.float64)
            orc.fuse_modulation(w, bb, g, be, mu, sd)
            n += 1
        el = time.perf_counter() - t0
        cpu = {"value": n / el, "unit": "images/s", "cores": 1, "kind": "oracle",
               "sample": f"{n} fusions of one image's last layer in {el:.1f} s (fp64 C oracle, "
                         "one thread; the copy of the shared layers not included)"}
    line = {"metric": STAGE_METRIC["fuse"][0], "value": B / (ms * 1e-3), "unit": "images/s",
            "n_gpus": 1, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32 arithmetic, f16 out",
            "data": "synthetic (seeded weights; gamma, beta, mu, sigma stand-ins)",
            "config": {"workload": f"fuse: {B} images, MLP {'-'.join(map(str, dims))}",
                       "images": B, "params_per_image": int(shared_h.size),
                       "l2": "inputs smaller than L2; back-to-back calls", "parallelism": "dp1"},
            "roofline": roof, "clocks": clk.summary(), "e2e": e2e, "gpu_launches": args.steps,
            "cpu_baseline": cpu, "stage": "fuse"}
    print(json.dumps(line), flush=True)


def _event_time(fn, steps, stream, torch):
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record(stream)
    for _ in range(steps):
        fn()
    ev1.record(stream)
    torch.cuda.synchronize()
    return ev0.elapsed_time(ev1) / steps


def _stage_cpu(stage, wl, sym_h, counts, n_blk, eob, dx, budget_s):
    """The oracle, as it stands, on a bounded sample: whole images, one after
    another, until about budget_s seconds have passed."""
    import oracle
    orc = oracle.load()
    cores = os.cpu_count() or 1
    starts = np.r_[0, np.cumsum(counts)[:-1]]
    n, t0 = 0, time.perf_counter()
    while True:
        b = n % wl.B
        if stage == "izpr":
            orc.izpr(sym_h[starts[b]:starts[b] + counts[b]], eob, n_blk)
        elif stage == "idct":
            orc.unpatchify_idct(dx.coeffs[b], dx.steps[b].astype(np.float64), wl.H, wl.W, wl.L,
                                wl.C)
        else:
            c = orc.izpr(sym_h[starts[b]:starts[b] + counts[b]], eob, n_blk)
            y = orc.unpatchify_idct(c, dx.steps[b].astype(np.float64), wl.H, wl.W, wl.L, wl.C)
            orc.decode_values(y, dx.weights[b].astype(np.float64), wl.H, wl.W, wl.L, wl.C,
                              wl.dims, wl.act, nthreads=cores)
        n += 1
        el = time.perf_counter() - t0
        if el >= budget_s:
            break
    if stage == "pipeline":
        v, unit = n * wl.H * wl.W / 1e6 / el, "MP/s"
    else:
        v, unit = n * n_blk / 1e6 / el, "Mblocks/s"
    threads = cores if stage == "pipeline" else 1
    return {"value": v, "unit": unit, "cores": threads, "kind": "oracle",
            "sample": f"{n} whole image(s) of workload {wl.name} in {el:.1f} s "
                      f"({'fp64 C oracle, decode on ' + str(cores) + ' OpenMP threads' if stage == 'pipeline' else 'fp64 C oracle, one thread'})"}


def run_stage(args):
    import torch
    from paper_2609_09020_gb300 import build, pic
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    build.build()
    stage = args.stage
    wl = wk.WORKLOADS["c5"]
    B = wl.B
    sym_h, counts, n_blk, eob = wk.zpr_streams(wl)
    dx = wk.make_dct_inputs(wl)
    stream = torch.cuda.current_stream(dev)
    sp = stream.cuda_stream
    n_lat = wl.n_latents
    starts = np.r_[0, np.cumsum(counts)]
    chunk = max(1, min(args.chunk, B))
    peaks = load_peaks()

    sym = torch.from_numpy(sym_h).to(dev)
    coeffs_in = torch.from_numpy(dx.coeffs).to(dev)
    steps_t = torch.from_numpy(dx.steps).to(dev)
    w_host = np.ascontiguousarray(dx.weights_for("fp16_tc"))
    wts = torch.from_numpy(w_host).to(dev)
    rows = chunk if stage == "pipeline" else B
    coeffs = torch.empty((rows * n_blk, 64), dtype=torch.int32, device=dev)
    offsets = torch.empty(rows * n_blk, dtype=torch.int64, device=dev)
    lat = torch.empty((rows, n_lat), dtype=torch.float32, device=dev)
    out = torch.empty((B, 3, wl.H, wl.W), dtype=torch.float32, device=dev)
    wsb = pic.pic_izpr_workspace_bytes(int(counts.max()) * rows if stage == "pipeline"
                                       else sym.numel())
    ws = torch.empty(wsb, dtype=torch.uint8, device=dev)
    dec = pic.Decoder.for_workload(wl, "fp16_tc", max_batch=chunk, latent="fp32") \
        if stage == "pipeline" else None
    if dec is not None:
        dec.check_buffers(chunk, wl.H, wl.W, latents=lat, steps=None, weights=wts[:chunk],
                          out=out[:chunk])

    def izpr(s_ptr, n_sym, nb):
        rc = pic.pic_izpr_decode(s_ptr, n_sym, eob, nb, coeffs.data_ptr(), offsets.data_ptr(),
                                 ws.data_ptr(), wsb, sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_izpr_decode")

    def idct(c_ptr, s_ptr, nb_img):
        rc = pic.pic_idct_unpatchify(c_ptr, s_ptr, nb_img, wl.H, wl.W, wl.L, wl.C,
                                     lat.data_ptr(), sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_idct_unpatchify")

    def one_step():
        if stage == "izpr":
            izpr(sym.data_ptr(), sym.numel(), B * n_blk)
        elif stage == "idct":
            idct(coeffs_in.data_ptr(), steps_t.data_ptr(), B)
        else:
            for b0 in range(0, B, chunk):
                nb = min(chunk, B - b0)
                izpr(sym.data_ptr() + 4 * int(starts[b0]), int(starts[b0 + nb] - starts[b0]),
                     nb * n_blk)
                idct(coeffs.data_ptr(), steps_t.data_ptr() + 4 * b0 * wl.L, nb)
                dec.decode_batch(lat, None, wts[b0:b0 + nb], wl.H, wl.W, out[b0:b0 + nb],
                                 stream=stream, B=nb, check=False)

    for _ in range(max(args.warmup, 3)):
        one_step()
    torch.cuda.synchronize()
    if stage in ("izpr", "pipeline"):
        rc = pic.pic_izpr_status(ws.data_ptr(), sp)
        if rc != pic.PIC_OK:
            raise pic.PicError(rc, "pic_izpr_status")
    if dec is not None:
        dec.check(stream)
    with ClockSampler(0) as clk:
        ms = _event_time(one_step, args.steps, stream, torch)
    if dec is not None:
        dec.check(stream)

    # per-stage launch times (the same calls, timed one stage at a time)
    n_sym = sym.numel()
    stage_ms = {}
    if stage == "pipeline":
        def part(which):
            def f():
                for b0 in range(0, B, chunk):
                    nb = min(chunk, B - b0)
                    if which == "izpr":
                        izpr(sym.data_ptr() + 4 * int(starts[b0]),
                             int(starts[b0 + nb] - starts[b0]), nb * n_blk)
                    elif which == "idct":
                        idct(coeffs.data_ptr(), steps_t.data_ptr() + 4 * b0 * wl.L, nb)
                    else:
                        dec.decode_batch(lat, None, wts[b0:b0 + nb], wl.H, wl.W,
                                         out[b0:b0 + nb], stream=stream, B=nb, check=False)
            return f
        for which in ("izpr", "idct", "decode"):
            stage_ms[which] = _event_time(part(which), args.steps, stream, torch)

    blocks = B * n_blk
    n_chunks = (B + chunk - 1) // chunk
    if stage == "izpr":
        nbytes = 4 * n_sym + (256 + 8) * blocks
        value = blocks / (ms * 1e-3) / 1e6
        launches = 3
    elif stage == "idct":
        nbytes = 256 * blocks + 4 * B * n_lat + 4 * B * wl.L
        value = blocks / (ms * 1e-3) / 1e6
        launches = 1
    else:
        nbytes = (4 * n_sym + 2 * B * wl.n_params + 4 * B * wl.L + 12 * B * wl.H * wl.W)
        value = B * wl.H * wl.W / (ms * 1e-3) / 1e6
        launches = n_chunks * 5
    metric, unit = STAGE_METRIC[stage]
    if stage == "pipeline":
        flops = 2.0 * wl.macs_per_pixel * B * wl.H * wl.W
        t_dec = stage_ms["decode"] * 1e-3
        roof = {"bound": "tensor", "achieved": flops / t_dec / 1e12,
                "peak": peaks["bf16_tflops"], "unit": "TFLOP/s",
                "peak_source": f"bf16 dense burst, {peaks['source']}",
                "kernel": "tc05_7x64x64x3_relu_f32lat (the dominant stage)",
                "avg_launch_us": 1e3 * stage_ms["decode"] / n_chunks,
                "whole_step_hbm_gbs": nbytes / (ms * 1e-3) / 1e9}
    else:
        roof = {"bound": "hbm", "achieved": nbytes / (ms * 1e-3) / 1e9, "peak": peaks["hbm_gbs"],
                "unit": "GB/s", "peak_source": f"copy bandwidth, {peaks['source']}",
                "kernel": "izpr_count+izpr_expand (one call)"
                if stage == "izpr" else "idct_unpatchify_kernel",
                "avg_launch_us": ms * 1e3}
    roof["frac"] = roof["achieved"] / roof["peak"]
    roof["traffic"] = recorded_traffic("idct_unpatchify_kernel", "c5x64") if stage == "idct" \
        else None
    if stage == "izpr":
        roof["traffic_note"] = ("one call is 2 kernels; the stream is read twice "
                                "(profiles/izpr__c5x64_launches_and_full.md)")
    roof["algorithmic_bytes_per_launch"] = nbytes

    # end to end with host buffers: H2D of the step's input, the stage, D2H of its result
    e2e = None
    if not args.no_e2e:
        if stage == "izpr":
            src_h, dst_d = torch.from_numpy(sym_h).pin_memory(), sym
            res_d = coeffs
        elif stage == "idct":
            src_h, dst_d = torch.from_numpy(dx.coeffs).pin_memory(), coeffs_in
            res_d = lat
        else:
            src_h, dst_d = torch.from_numpy(sym_h).pin_memory(), sym
            res_d = out
        res_h = torch.empty(res_d.shape, dtype=res_d.dtype).pin_memory()

        def e2e_step():
            dst_d.copy_(src_h, non_blocking=True)
            one_step()
            res_h.copy_(res_d, non_blocking=True)
            torch.cuda.current_stream().synchronize()

        e2e_step()
        k = max(3, min(args.steps, 10))
        t0 = time.perf_counter()
        for _ in range(k):
            e2e_step()
        el = (time.perf_counter() - t0) / k
        units = blocks / 1e6 if stage != "pipeline" else B * wl.H * wl.W / 1e6
        e2e = {"value": units / el, "unit": unit,
               "h2d_bytes_per_step": int(src_h.numel() * src_h.element_size()),
               "d2h_bytes_per_step": int(res_h.numel() * res_h.element_size()),
               "ms_per_step": 1e3 * el}

    cpu = None if args.no_cpu_baseline else _stage_cpu(stage, wl, sym_h, counts, n_blk, eob, dx,
                                                       min(args.cpu_budget_s, 12.0))
    line = {"metric": metric, "value": value, "unit": unit, "n_gpus": 1, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": {"izpr": "int32", "idct": "int32 in, f32 arithmetic and out",
                      "pipeline": "int32 symbols; f32 iDCT; f16 operands (hi+lo), f32 accumulate"}[stage],
            "data": "synthetic (seeded DCT coefficients / ZpR streams shaped like the 64-image workload)",
            "config": {"workload": f"{stage}: {B} x {wl.W}x{wl.H}, {wl.L} levels x {wl.C} ch, "
                                   f"{n_blk} 8x8 patches per image",
                       "images": B, "patches": blocks, "symbols": int(n_sym),
                       "symbols_per_patch": n_sym / blocks, "eob": eob,
                       "chunk_images": chunk if stage == "pipeline" else None,
                       "l2": "inputs larger than L2 (no flush needed)",
                       "parallelism": "dp1"},
            "roofline": roof, "clocks": clk.summary(), "e2e": e2e, "gpu_launches": launches * args.steps,
            "cpu_baseline": cpu, "stage": stage}
    if stage_ms:
        line["stage_ms"] = stage_ms
    if stage == "pipeline":
        line["images_per_s"] = B / (ms * 1e-3)
    print(json.dumps(line), flush=True)
    if dec is not None:
        dec.close()


def fp32_peak(pic, dev):
    """The FP32 FMA rate (TFLOP/s) of this GPU from the library's FMA
    microbenchmark, else the formula; and a note saying which."""
    try:
        tf = pic.fma_peak_tflops(dev)
        return tf, (f"FP32 FMA microbenchmark, measured (formula: {fp32_peak_tflops():.1f} "
                    f"TFLOP/s = 152 SMs x 128 lanes x 2 FLOP x 2070 MHz)")
    except Exception as exc:  # report the formula instead of failing the bench
        return fp32_peak_tflops(), (f"FP32 FMA formula (152 SMs x 128 lanes x 2 FLOP x 2070 MHz; "
                                    f"microbenchmark failed: {exc})")


PER_CONFIG = ["c1", "c2", "c3", "c4", "c5"]
# extra tensor-path rows with the per-tile kernels' TMA staging, which the
# library's default (the row-marching kernels) does not pick
PER_CONFIG_STAGING = {"c5": "tma", "c3": "tma", "c4": "tma"}


def per_config_rows(pic, dev, stream, peaks, fp32_tf, fp32_src, reps=None):
    """Every workload on both decoder paths, one row each: the median over
    timed calls of one decode launch, each call preceded by a 256 MB write
    that flushes L2 (the small workloads' inputs fit in L2), CUDA events on
    the launching stream around the decode alone."""
    import torch
    flush = torch.empty(64 << 20, dtype=torch.float32, device=dev)  # 256 MB > L2
    rows = []
    for name in PER_CONFIG:
        wl = wk.WORKLOADS[name]
        x = wk.make_inputs(wl)
        B = x.latents.shape[0]
        lat = torch.from_numpy(x.latents).to(dev)
        st = torch.from_numpy(x.steps).to(dev)
        out = torch.empty((B, 3, wl.H, wl.W), dtype=torch.float32, device=dev)
        runs = [("fp16_tc", "auto"), ("fp32", "auto")]
        if name in PER_CONFIG_STAGING:
            runs.insert(1, ("fp16_tc", PER_CONFIG_STAGING[name]))
        for precision, staging in runs:
            w = torch.from_numpy(np.ascontiguousarray(x.weights_for(precision))).to(dev)
            dec = pic.Decoder.for_workload(wl, precision, max_batch=B, staging=staging)
            dec.check_buffers(B, wl.H, wl.W, latents=lat, steps=st, weights=w, out=out)
            for _ in range(3):
                dec.decode_batch(lat, st, w, wl.H, wl.W, out, stream=stream, B=B, check=False)
            torch.cuda.synchronize(dev)
            n = reps or (30 if wl.pixels > 5e6 else 60)
            times = []
            for _ in range(n):
                flush.fill_(1.0)
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                dec.decode_batch(lat, st, w, wl.H, wl.W, out, stream=stream, B=B, check=False)
                e1.record(stream)
                e1.synchronize()
                times.append(e0.elapsed_time(e1))
            dec.check(stream)
            ms = float(np.median(times))
            roof = roofline_for(wl, precision, B, ms, peaks, fp32_tf, fp32_src, staging)
            rows.append({"workload": name, "precision": precision, "staging": staging,
                         "kernel": dec.kernel_name,
                         "images": B, "ms": ms, "ms_p10": float(np.percentile(times, 10)),
                         "ms_p90": float(np.percentile(times, 90)), "calls": n,
                         "mp_per_s": B * wl.H * wl.W / (ms * 1e-3) / 1e6,
                         "images_per_s": B / (ms * 1e-3),
                         "roofline": {k: roof[k] for k in ("bound", "achieved", "peak", "unit",
                                                            "frac", "binding_time_us",
                                                            "alu_bound")}})
            dec.close()
            del w
        del lat, st, out
    # The floor of this timing method: a near-empty launch of the library's
    # FMA microbenchmark kernel (152 CTAs x 256 threads, 128 FMAs a thread)
    # timed the same way (L2 flushed, events around the launch alone).
    out = torch.empty(152, dtype=torch.float32, device=dev)
    lib = pic.load_library()
    sp = stream.cuda_stream
    for _ in range(3):
        lib.pic_fma_peak_launch(out.data_ptr(), 152, 1, sp)
    torch.cuda.synchronize(dev)
    floor = []
    for _ in range(60):
        flush.fill_(1.0)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        lib.pic_fma_peak_launch(out.data_ptr(), 152, 1, sp)
        e1.record(stream)
        e1.synchronize()
        floor.append(e0.elapsed_time(e1))
    del flush
    return {"rows": rows, "timing": "median of per-call CUDA events, L2 flushed (256 MB write) "
                                    "before every call, 3 warm-up calls per row",
            "launch_floor": {"ms": float(np.median(floor)),
                             "kernel": "FMA microbenchmark, 152 CTAs x 256 threads, 128 FMAs a "
                                       "thread, timed the same way"}}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--workload", default="c5", choices=sorted(wk.WORKLOADS))
    ap.add_argument("--precision", default=None, choices=["fp32", "fp16_tc"])
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-budget-s", type=float, default=12.0)
    ap.add_argument("--ref-step-s", type=float, default=5.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-per-config", action="store_true",
                    help="skip the rows of every workload on both paths")
    ap.add_argument("--no-protocols", action="store_true",
                    help="skip the per-call, CUDA-graph and serial-per-image rows")
    ap.add_argument("--stage", default="decode",
                    choices=["decode", "izpr", "idct", "pipeline", "fuse", "huffman",
                             "bitstream"],
                    help="decode (default): the synthesis; the others time the stages before "
                         "it, alone or chained, on one GPU")
    ap.add_argument("--chunk", type=int, default=64,
                    help="pipeline stage: images per iZpR/iDCT/decode round")
    args = ap.parse_args()
    if args.stage != "decode":
        if args.impl == "reference" or int(os.environ.get("WORLD_SIZE", "1")) > 1:
            print(json.dumps({"stage": args.stage, "unavailable":
                              "stage benchmarks run our arm on one GPU only"}))
            return
        if args.stage == "fuse":
            run_fuse_stage(args)
        elif args.stage in ("huffman", "bitstream"):
            run_bitstream_stages(args)
        else:
            run_stage(args)
        return

    wl = wk.WORKLOADS[args.workload]
    precision = args.precision or wl.precisions[-1]
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        if world > 1:
            import torch.distributed as dist
            dist.init_process_group("gloo")
        run_reference(args, wl, precision, rank)
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()
        return

    import torch
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    from paper_2609_09020_gb300 import build, pic
    if rank == 0:
        build.build()
    barrier()
    build.build()  # no-op once built

    # Each rank decodes its own batch: image seeds offset by rank (weak scaling).
    wl_r = shard_workload(wl, rank)
    x = wk.make_inputs(wl_r)
    B = x.latents.shape[0]
    dec = pic.Decoder.for_workload(wl, precision, max_batch=B)
    w_host = np.ascontiguousarray(x.weights_for(precision))
    lat = torch.from_numpy(x.latents).to(dev)
    steps_t = torch.from_numpy(x.steps).to(dev)
    wts = torch.from_numpy(w_host).to(dev)
    out = torch.empty((B, 3, wl.H, wl.W), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    dec.check_buffers(B, wl.H, wl.W, latents=lat, steps=steps_t, weights=wts, out=out)

    for _ in range(max(args.warmup, 3)):
        dec.decode_batch(lat, steps_t, wts, wl.H, wl.W, out, stream=stream, B=B, check=False)
    dec.check(stream)
    torch.cuda.synchronize(dev)

    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local_rank) as clk:
        barrier()
        torch.cuda.synchronize(dev)
        ev0.record(stream)
        for _ in range(args.steps):
            dec.decode_batch(lat, steps_t, wts, wl.H, wl.W, out, stream=stream, B=B, check=False)
        ev1.record(stream)
        torch.cuda.synchronize(dev)
        barrier()
    dec.check(stream)
    ms = max_over_ranks(ev0.elapsed_time(ev1) / args.steps, world, dev)

    # Extra rows (rank 0, outside the timed region above): per-call
    # percentiles, a CUDA-graph replay of the same calls, and the paper's
    # serial protocol (synchronise, decode one image, synchronise; App. C).
    protocols = None
    if rank == 0 and not args.no_protocols:
        for _ in range(20):  # warm-up calls
            dec.decode_batch(lat, steps_t, wts, wl.H, wl.W, out, stream=stream, B=B, check=False)
        call_ms = []
        for _ in range(200):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            dec.decode_batch(lat, steps_t, wts, wl.H, wl.W, out, stream=stream, B=B, check=False)
            e1.record(stream)
            e1.synchronize()
            call_ms.append(e0.elapsed_time(e1))
        q = np.percentile(call_ms, [10, 50, 90])
        graph = None
        try:
            g = torch.cuda.CUDAGraph()
            side = torch.cuda.Stream(dev)
            side.wait_stream(stream)
            with torch.cuda.stream(side):
                with torch.cuda.graph(g):
                    for _ in range(4):
                        dec.decode_batch(lat, steps_t, wts, wl.H, wl.W, out, B=B, check=False)
            stream.wait_stream(side)
            g.replay()
            torch.cuda.synchronize(dev)
            reps = 50  # 200 calls
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(reps):
                g.replay()
            e1.record(stream)
            torch.cuda.synchronize(dev)
            graph = {"ms_per_call": e0.elapsed_time(e1) / (4 * reps), "calls_per_graph": 4}
        except Exception as exc:  # graph capture unsupported here: report, don't fail the bench
            graph = {"unavailable": str(exc)[:200]}
        dec.check(stream)
        t_img = []
        n_ser = min(B, 16)
        w_img = [wts[b].clone() for b in range(n_ser)]  # each image's weights on its own (aligned)
        for b in range(n_ser):
            dec.check_buffers(1, wl.H, wl.W, latents=lat[b:b + 1], steps=steps_t[b:b + 1],
                              weights=w_img[b], out=out[b:b + 1])
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            dec.decode_batch(lat[b:b + 1], steps_t[b:b + 1], w_img[b], wl.H, wl.W, out[b:b + 1],
                             stream=stream, B=1, check=False)
            torch.cuda.synchronize(dev)
            t_img.append(time.perf_counter() - t0)
        protocols = {
            "per_call_ms": {"p10": float(q[0]), "median": float(q[1]), "p90": float(q[2]),
                            "calls": len(call_ms)},
            "cuda_graph": graph,
            "serial_per_image": {"ms_per_image": 1e3 * float(np.mean(t_img)),
                                 "images_per_s": 1.0 / float(np.mean(t_img)), "images": len(t_img),
                                 "note": "synchronise, decode one image, synchronise (the paper's "
                                         "timing protocol; host clock)"}}
    px_total = world * B * wl.H * wl.W
    value = whole_job_rate(B * wl.H * wl.W, world, ms)
    images_per_s = world * B / (ms * 1e-3)

    # End to end through the C ABI with host buffers (pinned): H2D of the
    # inputs, the decode, D2H of the RGB planes, every step.
    e2e = None
    if not args.no_e2e:
        lat_h = torch.from_numpy(x.latents).pin_memory()
        st_h = torch.from_numpy(x.steps).pin_memory()
        w_h = torch.from_numpy(w_host).pin_memory()
        out_h = torch.empty((B, 3, wl.H, wl.W), dtype=torch.float32).pin_memory()
        sp = stream.cuda_stream
        ptrs = (lat_h.data_ptr(), st_h.data_ptr(), w_h.data_ptr(), out_h.data_ptr())

        def host_call():
            rc = pic.pic_decode_batch_host(dec.handle, B, ptrs[0], ptrs[1], ptrs[2], wl.H, wl.W,
                                           ptrs[3], sp)
            if rc != pic.PIC_OK:
                raise pic.PicError(rc, "pic_decode_batch_host")

        for _ in range(3):  # warm-up: staging allocation, first DMA of the pinned pages
            host_call()
        e_steps = max(3, min(args.steps, 10))
        barrier()
        t0 = time.perf_counter()
        for _ in range(e_steps):
            host_call()
        el = max_over_ranks(time.perf_counter() - t0, world, dev)
        h2d = lat_h.numel() * 4 + st_h.numel() * 4 + w_h.numel() * w_h.element_size()
        e2e = {"value": px_total * e_steps / el / 1e6, "unit": UNIT,
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(out_h.numel() * 4),
               "ms_per_step": 1e3 * el / e_steps}

    # The same end to end with the uint8 HWC output (a quarter of the fp32
    # RGB return over the host link), through its own handle.
    e2e_u8 = None
    if not args.no_e2e:
        dec8 = pic.Decoder.for_workload(wl, precision, max_batch=B, output="u8_hwc")
        out8_h = torch.empty((B, wl.H, wl.W, 3), dtype=torch.uint8).pin_memory()
        p8 = out8_h.data_ptr()

        def host_call_u8():
            rc = pic.pic_decode_batch_host(dec8.handle, B, ptrs[0], ptrs[1], ptrs[2], wl.H, wl.W,
                                           p8, sp)
            if rc != pic.PIC_OK:
                raise pic.PicError(rc, "pic_decode_batch_host")

        for _ in range(3):
            host_call_u8()
        barrier()
        t0 = time.perf_counter()
        for _ in range(e_steps):
            host_call_u8()
        el8 = max_over_ranks(time.perf_counter() - t0, world, dev)
        dec8.check(stream)
        e2e_u8 = {"value": px_total * e_steps / el8 / 1e6, "unit": UNIT,
                  "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(out8_h.numel()),
                  "ms_per_step": 1e3 * el8 / e_steps, "output": "uint8 [B][H][W][3]"}
        dec8.close()

    peaks = load_peaks()
    flops, nbytes = algorithmic(wl, B)
    kname = dec.kernel_name
    fp32_tf, fp32_src = fp32_peak(pic, dev)
    roof = roofline_for(wl, precision, B, ms, peaks, fp32_tf, fp32_src)
    roof["traffic"] = recorded_traffic(kname, wl.name)
    roof["kernel"] = kname

    per_config = None
    if rank == 0 and not args.no_per_config:
        per_config = per_config_rows(pic, dev, stream, peaks, fp32_tf, fp32_src)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(wl, x, precision, args.cpu_budget_s)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f16 operands (hi+lo split), f32 accumulate" if precision == "fp16_tc"
                else "f32",
                "data": "synthetic (seeded Laplacian int latents, N(0,1/fan_in) weights)",
                "config": {**workload_desc(wl, precision), "parallelism": f"dp{world}",
                           "l2": "inputs larger than L2 (no flush needed)"
                           if nbytes > 129e6 else "inputs smaller than L2; back-to-back calls",
                           "batch_per_gpu": B},
                "images_per_s": images_per_s,
                "roofline": roof, "clocks": clk.summary(), "e2e": e2e,
                "gpu_launches": args.steps, "cpu_baseline": cpu}
        if e2e_u8 is not None:
            line["e2e_u8"] = e2e_u8
        if per_config is not None:
            line["per_config"] = per_config
        if protocols is not None:
            line["protocols"] = protocols
        print(json.dumps(line), flush=True)
    dec.close()
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
