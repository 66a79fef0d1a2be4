#!/usr/bin/env python
"""Benchmark: whole-network forward of the synthetic pruned ResNet-50 (batch 1 per GPU).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--workload resnet50|vgg16|mobilenet_v2|mobilenet_v1|inception_v3|single] [--batch B]

One step = one pass of the whole hot path (every layer of the network) over one
batch.  Prints ONE JSON line on rank 0.  Multi-GPU runs are independent replicas
(images shard over ranks; no data-path collective); launch them with torchrun.
"""
import argparse
import json
import os
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "pruned ResNet-50 batch-1 latency (ms), images/sec, fraction of sparse roofline"


def build_model(name):
    from workloads import models
    if name == "resnet50":
        return models.resnet50(), "resnet50_v1.5_224_conv12.5pct_fc10pct_stem_dense"
    if name == "vgg16":
        return models.vgg16(), "vgg16_int8_224_conv8pct_fc4pct"
    if name == "mobilenet_v2":
        return models.mobilenet_v2(), "mobilenet_v2_1.0_224_pointwise25pct"
    if name == "inception_v3":
        return models.inception_v3(), "inception_v3_299_conv12.5pct_fc10pct_stem_dense"
    if name == "mobilenet_v1":
        return models.mobilenet_v1(), "mobilenet_v1_1.0_224_pointwise25pct"
    if name == "resnet50_int8":
        return models.resnet50_int8(), "resnet50_v1.5_int8_224_conv12.5pct_fc10pct"
    if name == "single":
        return models.single_layer(), "conv3x3_64to64_56x56_10pct"
    raise SystemExit("unknown workload " + name)


class ClockSampler:
    """nvidia-smi clock / throttle-reason samples taken while the timed region runs."""
    FIELDS = ("uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.uuid = uuid
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.out = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                                          "-lms", "20"], stdout=self.out, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def run_until(self, samples, load, limit_s=5.0):
        """Runs load() until that many samples have been written (nvidia-smi takes longer to start than a short timed region lasts)."""
        end = time.time() + limit_s
        while self.proc is not None and time.time() < end and self.proc.poll() is None:
            load()
            with open(self.path) as f:
                if sum(self.uuid is None or self.uuid in line for line in f) >= samples:
                    return

    def stop(self):
        res = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        if self.proc is None:
            return res
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.out.close()
        sm, reasons, smax = [], set(), None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            f = [v.strip() for v in line.split(",")]
            if len(f) < 9 or (self.uuid and self.uuid not in f[0]):
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.path)
        if sm:
            sm.sort()
            res.update(sm_mhz=sm[len(sm) // 2], sm_max_mhz=smax, reasons=sorted(reasons), samples=len(sm))
        return res


def oracle_sample_plan(model, budget_s, full_s):
    """Ops of the bounded sample one reference step runs, and the share of the network's
    dense multiply-adds it covers (the oracle's cost is proportional to dense MACs)."""
    macs = []
    for op in model.ops:
        if op.kind in ("conv", "fc"):
            macs.append(float(op.w.size) * op.out_hw[0] * op.out_hw[1])
        else:
            macs.append(0.0)
    total = sum(macs)
    if budget_s >= full_s:
        return list(range(len(model.ops))), 1.0
    order = sorted((i for i in range(len(model.ops)) if macs[i] > 0), key=lambda i: macs[i])
    picked, acc = [], 0.0
    for i in order:
        if picked and (acc + macs[i]) / total * full_s > budget_s:
            break
        picked.append(i)
        acc += macs[i]
    return sorted(picked), acc / total


def run_reference(args):
    """Reference arm: the CPU oracle, as it stands, on the host cores."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from oracle import forward as oracle_forward
    from oracle import ref
    from workloads import models
    model, wname = build_model(args.workload)
    x = models.make_input(model, args.batch)
    cores = ref.num_threads()
    t0 = time.perf_counter()
    _, slots = oracle_forward.forward(model, x)
    full_s = time.perf_counter() - t0
    steps, warm = args.steps, args.warmup
    budget = 150.0 / max(1, steps + warm)
    picked, share = oracle_sample_plan(model, budget, full_s)

    def one_step():
        for i in picked:
            op = model.ops[i]
            oracle_forward.run_op(op, slots[op.src], slots[op.res] if op.res >= 0 else None)

    for _ in range(warm):
        one_step()
    t0 = time.perf_counter()
    for _ in range(steps):
        one_step()
    dt = (time.perf_counter() - t0) / max(1, steps)
    value = args.batch * share / dt
    sample = ("whole network, %d image(s) per step" % args.batch if share >= 1.0 else
              "%d of %d layers per step (%.2f%% of the network's dense multiply-adds), scaled to whole images"
              % (len(picked), len(model.ops), 100 * share))
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "images/s", "n_gpus": args.gpus,
            "steps": steps, "warmup": warm, "ms_per_step": dt * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64" if model.dtype == "f32" else "int32", "data": "synthetic",
            "config": {"workload": wname, "batch_per_gpu": args.batch, "full_forward_s": full_s},
            "cpu_baseline": {"value": value, "unit": "images/s", "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "images/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line))


def pack(model, batch, dev, x, flush, no_autotune, PackedModel):
    """The packed network, and how its schedules were chosen: timed layer by layer at pack time, or by the packer's own rules where
    the whole network measured faster that way (layers timed one by one do not show how far a kernel overlaps its neighbours)."""
    import torch
    best = None
    for timed in ((False,) if no_autotune else (True, False)):
        pm = PackedModel(model, batch, dev, autotune=timed)
        y = pm.new_output()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(25)]
        for a, b in ev:
            flush.zero_()
            a.record()
            pm.forward(x, y)
            b.record()
        torch.cuda.synchronize()
        ms = sorted(a.elapsed_time(b) for a, b in ev[5:])[10]
        if best is None or ms < best[0]:
            best = (ms, pm, "timed at pack time" if timed else "model")
    return best[1], best[2]


def run_ours(args):
    import torch
    from paper_1905_00571_b200 import dist, roofline
    from paper_1905_00571_b200.network import PackedModel
    from workloads import models

    rank, world, local = dist.init()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device; there is no CPU fallback")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    model, wname = build_model(args.workload)
    batch = args.batch
    x_np = models.make_input(model, batch, seed=1000 + rank)
    x_host = torch.from_numpy(x_np).pin_memory()
    x = x_host.to(dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)   # larger than the 126 MB L2
    stream = torch.cuda.current_stream()
    pm, schedules = pack(model, batch, dev, x, flush, args.no_autotune, PackedModel)
    y_host = torch.empty(pm.out_shape, dtype=pm.out_dtype).pin_memory()
    y = pm.new_output()
    n_ops = len(model.ops)
    K, W = args.steps, args.warmup

    for _ in range(max(W, 3)):
        flush.zero_()
        pm.forward(x, y)
    torch.cuda.synchronize()

    props = torch.cuda.get_device_properties(local)
    uuid = str(getattr(props, "uuid", "")) or None
    sampler = ClockSampler(uuid)

    # ---- timed region 1: inputs resident in HBM, L2 flushed between iterations ----
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    dist.barrier()
    torch.cuda.synchronize()
    sampler.start()

    def load():   # untimed
        for _ in range(50):
            pm.forward(x, y)
        torch.cuda.synchronize()

    sampler.run_until(1, load)   # sampling, and at the clocks of the load, before the first timed step
    dist.barrier()
    torch.cuda.profiler.start()   # lets a profiler started with --profile-from-start off see only the timed steps
    for a, b in ev:
        flush.zero_()
        a.record(stream)
        pm.forward(x, y)
        b.record(stream)
    torch.cuda.synchronize()
    torch.cuda.profiler.stop()
    dist.barrier()
    cold_ms = sum(a.elapsed_time(b) for a, b in ev) / K

    # ---- timed region 2: back-to-back graph replays (weights and activations stay in L2) ----
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record(stream)
    for _ in range(K):
        pm.forward(x, y)
    b.record(stream)
    torch.cuda.synchronize()
    warm_ms = a.elapsed_time(b) / K

    # ---- end to end: host buffers through the C ABI, copies inside the timed region ----
    for _ in range(3):
        pm.forward_host(x_host, y_host)
    dist.barrier()
    torch.cuda.synchronize()
    a.record(stream)
    for _ in range(K):
        flush.zero_()
        pm.forward_host(x_host, y_host)
    b.record(stream)
    torch.cuda.synchronize()
    e2e_total_ms = a.elapsed_time(b)
    # the flush is not part of a step: time it alone and take it out
    a.record(stream)
    for _ in range(K):
        flush.zero_()
    b.record(stream)
    torch.cuda.synchronize()
    e2e_ms = max(1e-6, (e2e_total_ms - a.elapsed_time(b)) / K)
    sampler.run_until(5, load)   # the timed regions may be shorter than the sampling period
    clocks = sampler.stop()

    cold_ms = dist.max_over_ranks(cold_ms, dev)
    warm_ms = dist.max_over_ranks(warm_ms, dev)
    e2e_ms = dist.max_over_ranks(e2e_ms, dev)
    images = dist.sum_over_ranks(batch, dev)

    # ---- per-layer device times -> kernel families -> roofline of the dominant one ----
    # every op is replayed as a CUDA graph of 20 back-to-back launches between CUDA events on the
    # launching stream (operands stay in L2, as they do inside a batch-1 forward)
    reps = 3
    per = [0.0] * n_ops
    for _ in range(reps):
        t = pm.layer_times(x, y, flush_l2=False, reps=20)
        per = [p + v / reps for p, v in zip(per, t)]
    peaks = roofline.measured_peaks()
    from paper_1905_00571_b200 import binding as B
    r_alu_derived = roofline.alu_peak_tflops(peaks["sm_max_mhz"])
    # the plain ALUs' multiply-add rate measured on this device (a kernel of nothing but FFMA / IMAD chains):
    # the compute-side denominator of every fraction below
    ffma_tflops = max(B.cadnn_measure_alu_peak("f32") for _ in range(2)) / 1e12
    imad_tops = max(B.cadnn_measure_alu_peak("s8") for _ in range(2)) / 1e12
    r_alu = imad_tops if model.dtype == "s8" else ffma_tflops
    rows_nom = roofline.network_roofline(model, batch, r_alu, roofline.HBM_NOMINAL_GBS)
    rows_meas = roofline.network_roofline(model, batch, r_alu, peaks["hbm_gbs"])
    fam = {}
    for r, ms in zip(rows_nom, per):
        f = fam.setdefault(r["family"], {"ms": 0.0, "flops": 0.0, "bytes": 0.0, "launches": 0, "t_roof_us": 0.0})
        f["ms"] += ms
        f["flops"] += r["flops"]
        f["bytes"] += r["wbytes"] + r["abytes"]
        f["launches"] += 1
        f["t_roof_us"] += r["t_roof_us"]
    top = max(fam, key=lambda k: fam[k]["ms"])
    ft = fam[top]
    alu_bound = sum(1 for r in rows_nom if r["family"] == top and r["t_alu_us"] >= r["t_mem_us"]) * 2 >= ft["launches"]
    if alu_bound:
        achieved = ft["flops"] / (ft["ms"] * 1e-3) / 1e12
        roof = {"bound": "alu", "achieved": achieved, "peak": r_alu, "unit": "TFLOP/s", "frac": achieved / r_alu,
                "traffic": None, "peak_source": "measured: %s chains on this device" % ("IMAD" if model.dtype == "s8" else "FFMA"),
                "frac_of_derived_peak": achieved / r_alu_derived}
    else:
        achieved = ft["bytes"] / (ft["ms"] * 1e-3) / 1e9
        roof = {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": achieved / peaks["hbm_gbs"], "traffic": None, "peak_source": peaks["source"]}
    roof.update(kernel=top, launches_per_step=ft["launches"], avg_launch_us=ft["ms"] * 1e3 / ft["launches"])
    planar = B.cadnn_net_layout(pm.net)["planar"]
    roof["traffic"] = recorded_traffic(args.workload, batch, top, planar)
    roof["algorithmic_bytes_per_launch"] = ft["bytes"] / ft["launches"]
    if top.startswith("sconv"):   # CUDA kernels behind the family in this net's layout
        roof["cuda_kernels"] = (["sconv_planar_kernel", "sconv_planar_tma_kernel", "sconv_planar_staged_kernel"]
                                if planar else ["tcconv_kernel", "sconv_kernel"])   # with and without a dense image
    t_roof_nom = sum(r["t_roof_us"] for r in rows_nom)
    t_roof_meas = sum(r["t_roof_us"] for r in rows_meas)
    k3 = [(r, ms) for r, ms in zip(rows_nom, per) if r["family"] == "sconv_kxk" and r["nnz"] and r["name"] not in ("conv1", "stem")]
    sparse = {"t_roof_us_8TBs": t_roof_nom, "t_roof_us_measured_hbm": t_roof_meas,
              "frac_cold": t_roof_nom / (cold_ms * 1e3), "frac_warm": t_roof_nom / (warm_ms * 1e3),
              "frac_kernel_sum": t_roof_nom / (sum(per) * 1e3),
              "frac_3x3_layers": (sum(r["t_roof_us"] for r, _ in k3) / (sum(ms for _, ms in k3) * 1e3)) if k3 else None,
              "alu_peak_tflops": r_alu, "alu_peak_source": "measured",
              "alu_peak_ffma_tflops_measured": ffma_tflops, "alu_peak_imad_tops_measured": imad_tops,
              "alu_peak_tflops_derived": r_alu_derived,
              "frac_warm_of_derived_peak": sum(r["t_roof_us"] for r in roofline.network_roofline(model, batch, r_alu_derived, roofline.HBM_NOMINAL_GBS)) / (warm_ms * 1e3),
              "families": {k: {"ms": v["ms"], "launches": v["launches"], "t_roof_us": v["t_roof_us"]} for k, v in fam.items()}}

    # the throughput regime beside the latency-limited batch-1 number: kernel-only fraction of the pruned 3x3
    # layers at batch 32 (schedules timed at pack time like the batch-1 ones; per-layer times as above)
    if rank == 0 and world == 1 and args.workload == "resnet50" and not args.no_batch32:
        pm32 = PackedModel(model, 32, dev, autotune=not args.no_autotune)
        x32 = torch.from_numpy(models.make_input(model, 32, seed=7)).to(dev)
        y32 = pm32.new_output()
        pm32.forward(x32, y32)
        torch.cuda.synchronize()
        t32 = pm32.layer_times(x32, y32, flush_l2=False, reps=5)
        rows32 = roofline.network_roofline(model, 32, r_alu, roofline.HBM_NOMINAL_GBS)
        k32 = [(r, ms) for r, ms in zip(rows32, t32) if r["family"] == "sconv_kxk" and r["nnz"] and r["name"] not in ("conv1", "stem")]
        sparse["frac_3x3_layers_batch32_kernel_only"] = sum(r["t_roof_us"] for r, _ in k32) / (sum(ms for _, ms in k32) * 1e3)
        sparse["frac_network_batch32_kernel_sum"] = sum(r["t_roof_us"] for r in rows32) / (sum(t32) * 1e3)
        del pm32, x32, y32

    line = None
    if rank == 0:
        cpu_base = None
        if world == 1:
            from oracle import forward as oracle_forward
            from oracle import ref
            t0 = time.perf_counter()
            reps_cpu = 0
            while reps_cpu < 1 or (time.perf_counter() - t0 < 10.0 and reps_cpu < 20):
                oracle_forward.forward(model, x_np)
                reps_cpu += 1
            dt = (time.perf_counter() - t0) / reps_cpu
            cores = ref.num_threads()
            cpu_base = {"value": batch / dt, "unit": "images/s", "cores": cores, "kind": "oracle",
                        "sample": "%d whole-network forward(s) of %d image(s), %.2f s each" % (reps_cpu, batch, dt)}
            if not args.no_one_thread:
                ref.set_threads(1)
                t0 = time.perf_counter()
                oracle_forward.forward(model, x_np)
                dt1 = time.perf_counter() - t0
                ref.set_threads(cores)
                cpu_base["one_thread"] = {"value": batch / dt1, "unit": "images/s", "cores": 1,
                                          "sample": "1 whole-network forward of %d image(s), %.2f s" % (batch, dt1)}
        value = images / (cold_ms * 1e-3)
        line = {"metric": METRIC, "value": value, "unit": "images/s", "n_gpus": world, "steps": K, "warmup": W,
                "ms_per_step": cold_ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f32" if model.dtype == "f32" else "s8", "data": "synthetic",
                "config": {"workload": wname, "batch_per_gpu": batch, "parallelism": "replicas x%d" % world,
                           "l2": "flushed between iterations (256 MiB write)", "launch": "CUDA graph replay",
                           "schedules": schedules},
                "latency_ms": cold_ms, "latency_ms_warm_l2": warm_ms, "images_per_s_warm_l2": images / (warm_ms * 1e-3),
                "sparse_roofline": sparse, "roofline": roof, "cpu_baseline": cpu_base,
                "e2e": {"value": images / (e2e_ms * 1e-3), "unit": "images/s", "ms_per_step": e2e_ms,
                        "h2d_bytes_per_step": int(x_host.numel() * x_host.element_size()),
                        "d2h_bytes_per_step": int(y_host.numel() * y_host.element_size())},
                "gpu_launches": K * pm.launches_per_forward(), "clocks": clocks,
                "paper_context": "26 ms (title) / 21 ms (text) ResNet-50 on a Snapdragon 835 / Adreno 540 phone"}
        print(json.dumps(line))
    dist.finalize()
    return line


# DRAM bytes per launch (dram__bytes_read.sum + dram__bytes_write.sum) of the dominant kernel family, from one ncu
# pass over this command (summary and command line: profiles/resnet50_batch1_launch_list.md), valid for the kernel
# sources whose digest is recorded with it.  The family's layers run in the dense tensor-core kernel (NHWC networks),
# which serves 1x1 and k x k layers alike: the figure is the mean over the 52 conv launches of a step behind the stem.
TRAFFIC = {"workload": "resnet50", "batch": 1, "family": "sconv_1x1", "planar": False, "dram_bytes_per_launch": 4410143,
           "digest": "1d40905414a3c903"}


def kernel_sources_digest():
    import hashlib
    here = os.path.dirname(os.path.abspath(__file__))
    h = hashlib.sha256()
    for sub in ("paper_1905_00571_b200/csrc", "include"):
        d = os.path.join(here, sub)
        for name in sorted(os.listdir(d)):
            if name.endswith((".cu", ".h")):
                with open(os.path.join(d, name), "rb") as f:
                    h.update(name.encode() + b"\0" + f.read())
    return h.hexdigest()[:16]


def recorded_traffic(workload, batch, family, planar):
    t = TRAFFIC
    if t["dram_bytes_per_launch"] is None or (t["workload"], t["batch"], t["family"], t["planar"]) != (workload, batch, family, planar):
        return None
    return t["dram_bytes_per_launch"] if t["digest"] == kernel_sources_digest() else None


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None)
    ap.add_argument("--warmup", type=int, default=None)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="resnet50")
    ap.add_argument("--batch", type=int, default=1)
    ap.add_argument("--no-autotune", action="store_true", help="use the packer's time model instead of timing schedules")
    ap.add_argument("--no-one-thread", action="store_true", help="skip the 1-thread run of the CPU baseline")
    ap.add_argument("--no-batch32", action="store_true", help="skip the batch-32 kernel-only fraction of the 3x3 layers")
    args = ap.parse_args()
    if args.impl == "reference":
        args.steps = 5 if args.steps is None else args.steps
        args.warmup = 1 if args.warmup is None else args.warmup
        run_reference(args)
    else:
        args.steps = 2000 if args.steps is None else args.steps
        args.warmup = 10 if args.warmup is None else args.warmup
        run_ours(args)


if __name__ == "__main__":
    main()
