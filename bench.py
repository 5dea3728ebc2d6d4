#!/usr/bin/env python
"""Benchmark of the predictive-delta-coding hot path (encode then decode of one synthetic batch).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload llama2-7b] [--impl own|reference]

A step = one pass of the whole path over one batch: top-K softmax, fused predict + quantise + rANS
encode of every (stream, position), then the decode of the same batch.  The metric is KV tokens per
second (a KV token = one token position of one session across all 2*L*H streams) that were both
encoded and decoded.  With N > 1 (torchrun) every rank runs its own batch (streams shard with no
exchange): weak scaling, value = tokens of all ranks / slowest rank's time; `--shard layers` instead
gives rank r the layers [r L/N, (r+1) L/N) of ONE batch (strong scaling: each rank holds only its
slice of T and of the KV tensor, the union of the ranks' chunks is the single-GPU result).

The default run (no --workload, one GPU) prints the headline line for `llama2-7b` and, in its
`configs` object, one compact record per benchmark configuration (tiny, llama2-7b, 70b-longctx top-K
and dense, the dedup pipeline, the append path with its perplexity x step sweep).
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "KV tokens/s encoded+decoded per B200"
UNIT = "KV tokens/s"


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        return float(json.load(open(p))["hbm_gbs"]), "measured"
    return 6650.0, "fallback"


def tensor_peak():
    """Sustained dense bf16 TFLOP/s (the contraction is timed inside a long step)."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        return float(json.load(open(p)).get("bf16_tflops_sustained", 1400.0)), "measured sustained bf16"
    return 1400.0, "fallback"


def parse_over(pairs):
    over = {}
    for kvs in pairs:
        k, v = kvs.split("=")
        over[k] = float(v) if "." in v else int(v)
    return over


# Issue-slot use of the fused kernels (smsp__issue_active) from an ncu capture; quoted beside the roofline fraction, not part of it.
NCU_ISSUE_SLOT_USE = {"encode_kernel": 0.727, "decode_kernel": 0.722}


def fused_roofline(vecs, K, d, t_bytes, kv_bytes, payload, ek, dk, sm_mhz, sms, peak, peak_kind, traffic_per_vector=None):
    """Roofline record of the fused predict + quantise + code kernels (the slower of the two).
    Two ceilings apply to a launch: HBM on the COMPULSORY bytes (KV once, bitstream once, every
    table once) and the plain fp32 ALUs on the mixture's K*d fused multiply-adds per vector; the
    fraction reported is the larger of the two (the ceiling the kernel is closer to), `bound` says
    which.  The gathered-row accounting of the benchmark definition (K*d*2 bytes per vector) is
    kept apart: those rows come from L1 / L2, so it is not an HBM utilisation."""
    dom_enc = ek >= dk
    ms = ek if dom_enc else dk
    name = "encode_kernel" if dom_enc else "decode_kernel"
    sec = ms / 1e3
    bytes_c = kv_bytes + t_bytes + payload
    hbm_frac = bytes_c / sec / 1e9 / peak
    fma = vecs * K * d
    flop_peak = 2.0 * sms * 128 * sm_mhz * 1e6 / 1e12            # TFLOP/s of the fp32 FMA pipes at the sampled clock
    flop_ach = 2.0 * fma / sec / 1e12
    alu_frac = flop_ach / flop_peak
    bytes_ns = kv_bytes + vecs * K * d * 2 + payload
    r = {"kernel": name, "ms_per_launch": ms, "encode_kernel_ms": ek, "decode_kernel_ms": dk,
         "hbm_compulsory": {"bytes_per_launch": bytes_c, "achieved": bytes_c / sec / 1e9, "peak": peak, "unit": "GB/s",
                            "frac": hbm_frac, "peak_kind": peak_kind},
         "fp32_fma": {"achieved": flop_ach, "peak": flop_peak, "unit": "TFLOP/s", "frac": alu_frac,
                      "peak_kind": "SMs x 128 lanes x 2 flop x sampled SM clock (%d x %.0f MHz)" % (sms, sm_mhz)},
         "issue_slot_use_ncu": NCU_ISSUE_SLOT_USE.get(name),
         "busiest_units_ncu": "issue slots 72-73 %, heavy half of the FMA pipe 67 / 65 %, L1 data pipe 60 / 62 % (ncu capture, "
                              "encode / decode): no single unit saturated",
         "gathered_row_bytes_frac": bytes_ns / sec / 1e9 / peak,
         "gathered_row_note": "KV + K*d*2 B of gathered rows per vector + bitstream over the HBM copy peak; the rows are "
                           "L1 / L2 hits, so this is an on-chip gather rate, not an HBM utilisation",
         "traffic": None if traffic_per_vector is None else traffic_per_vector[name] * vecs}
    if alu_frac >= hbm_frac:
        r.update(bound="alu", achieved=flop_ach, peak=flop_peak, unit="TFLOP/s", frac=alu_frac)
    else:
        r.update(bound="hbm", achieved=bytes_c / sec / 1e9, peak=peak, unit="GB/s", frac=hbm_frac)
    return r


class ClockSampler:
    """nvidia-smi sampling of SM clock and throttle reasons while the timed region runs."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        cmd = ["nvidia-smi", "-i", uuid, "--query-gpu=" + self.Q, "--format=csv,noheader,nounits", "-lms", "200"]
        try:
            self.p = subprocess.Popen(cmd, stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        self.f.flush()
        rows = [r.strip().split(",") for r in open(self.f.name) if r.strip()]
        os.unlink(self.f.name)
        sm, mx, power, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                sm.append(float(r[0])); mx.append(float(r[1])); power.append(float(r[2]))
            except (ValueError, IndexError):
                continue
            for nme, v in zip(names, r[3:7]):
                if v.strip().lower().startswith("active"):
                    reasons.add(nme)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "power_w_max": max(power) if power else None, "samples": len(sm), "reasons": sorted(reasons)}


# DRAM bytes per vector of the fused kernels and the launch that forms their variance terms (2.2 of them), from the ncu
# capture summarised in profiles/gather_one_block_and_variance.md (dram__bytes_read.sum + dram__bytes_write.sum over 4.19 M
# vectors; traffic grows in proportion to the vectors).  Valid for the default workload and chunk size only.
NCU_DRAM_BYTES_PER_VECTOR = {"encode_kernel": 655.7, "decode_kernel": 418.4}
NCU_TRAFFIC_NOTE = ("dram__bytes_read + dram__bytes_write of a 4-layer ncu capture "
                    "scaled by the vectors of a launch")


def max_over_ranks(ms, dist, device):
    """Slowest rank's time (the job's time); identity without a process group."""
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    if dist is not None:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t[0])


def job_value(world, tokens_per_rank_step, ms_per_step):
    """Whole-job KV tokens/s: every rank codes its own batch (weak scaling)."""
    return world * tokens_per_rank_step / (ms_per_step / 1e3)


def oracle_sample_rate(w, positions, layers, workers=1):
    """Times the CPU oracle (encode + decode) on a slice of the workload: `positions` positions of
    session 0, `layers` layers, all heads, cut along the head axis over `workers` processes (1 = the
    single-threaded oracle in this process).  Returns KV tokens/s (vectors / W / seconds)."""
    import oracle
    cfg = w["cfg"]
    H, d, V, K = cfg["H"], cfg["d"], cfg["V"], cfg["K"]
    Tn = w["T"][:layers].cpu().numpy()
    kvn = w["kv"][:layers, :, :1, :, :positions].cpu().numpy()
    lgn = w["logits"][:1, :positions].cpu().numpy()
    tkn = w["tokens"][:1, :positions].cpu().numpy()
    ocfg = oracle.Config(layers, H, d, V, K, cfg["delta"], 0.0, cfg["chunk_pos"], 0)
    r = oracle.roundtrip_parallel(ocfg, Tn, kvn, lgn, tkn, workers=workers)
    assert r["rc"] == 0 and r["max_err"] <= cfg["delta"] / 2 + 1e-3
    W_full = 2 * cfg["L"] * H
    vecs = positions * 2 * layers * H
    return dict(value=vecs / W_full / r["seconds"], encode=vecs / W_full / r["encode_s"], decode=vecs / W_full / r["decode_s"],
                seconds=r["seconds"], bytes=r["payload_bytes"], vectors=vecs, workers=r["workers"],
                bits_per_component=8.0 * r["payload_bytes"] / (vecs * d),
                ideal_bits_per_component=r["ideal_bits"] / (vecs * d),                # sum of -log2(f/M) + raw bits
                token_bits_per_position=r["token_bits"] / positions)                  # sum of -log2 P(x_i | x_<i)


def cpu_baseline(w):
    """The oracle as it stands on the host's cores: single-threaded, then one process per slice of
    heads on every core this process may use.  Bounded samples of the same workload."""
    import oracle
    cfg = w["cfg"]
    L, n, H, W = cfg["L"], cfg["n"], cfg["H"], 2 * cfg["L"] * cfg["H"]
    layers, pos = min(L, 2), min(n, 256)
    one = oracle_sample_rate(w, pos, layers, workers=1)
    cores = oracle.host_cores()
    many = oracle_sample_rate(w, pos, layers, workers=cores) if cores > 1 and H > 1 else one
    return {"value": many["value"], "unit": UNIT, "cores": many["workers"], "kind": "oracle",
            "host_cores": cores, "cpu_count": os.cpu_count(),
            "sample": f"session 0, first {pos} positions, {layers} of {L} layers, all heads ({one['vectors']} vectors; "
                      f"{many['seconds']:.1f} s encode+decode with one process per slice of heads on {many['workers']} cores, "
                      f"{one['seconds']:.1f} s single-threaded); rate scaled by W={W} vectors per KV token",
            "single_core": {"value": one["value"], "encode": one["encode"], "decode": one["decode"], "seconds": one["seconds"]},
            "encode": many["encode"], "decode": many["decode"],
            "sample_bits_per_component": one["bits_per_component"],
            "sample_ideal_bits_per_component": one["ideal_bits_per_component"],
            "sample_token_bits_per_position": one["token_bits_per_position"]}


def shard_layers(L, world, rank):
    """Layers [lo, hi) that rank codes under --shard layers (contiguous, sizes differ by at most one)."""
    return L * rank // world, L * (rank + 1) // world


def shard_slots(S, L, H, mc, world, rank):
    """(session, table, chunk) index slots of the single-GPU run that this rank produces under
    --shard layers: table = (layer*2 + kv)*H + head for the rank's own layers."""
    lo, hi = shard_layers(L, world, rank)
    return {(s, t, c) for s in range(S) for t in range(lo * 2 * H, hi * 2 * H) for c in range(mc)}


def run_codec(args, torch, plc, workloads, dev, name, over, steps, warmup, dist=None, world=1, rank=0,
              variant="topk", d_model=4096, adaptive_b0=0, zero_rate=0.0, sigma_floor=0.0, shard=None,
              want_e2e=False, want_cpu=False, e2e_steps=4, e2e_groups=4, w=None, layers=None):
    """Times `steps` passes (encode then decode) of workload `name` after `warmup` untimed ones and
    returns (line, workload).  `w` reuses a workload already built; `layers` = (lo, hi) restricts the
    run to a slice of its layers (views, nothing is copied)."""
    import math
    linear = variant == "linear"
    dense = variant == "dense"
    if w is None:
        o = dict(over)
        if linear:
            o["dm"] = d_model
        seed = 20260415 + (0 if shard else 1000 * rank)           # a sharded job codes ONE batch: same inputs on every rank
        w = workloads.build(name, dev, seed=seed, **o)
    cfg = dict(w["cfg"])
    T, kv = w["T"], w["kv"]
    if shard == "layers":
        layers = shard_layers(cfg["L"], world, rank)
    if layers is not None:
        lo, hi = layers
        T, kv = T[lo:hi], kv[lo:hi]
        cfg["L"] = hi - lo
    S, n, L, H, d, V, K = cfg["S"], cfg["n"], cfg["L"], cfg["H"], cfg["d"], cfg["V"], cfg["K"]
    W = 2 * L * H
    adaptive = (adaptive_b0, 4, math.log2(cfg["pp"])) if adaptive_b0 > 0 else None
    tok = w["tokens"] if adaptive else None
    if linear:
        ctx = plc.Context.linear(w["E"], w["A"], w["c"], cfg["delta"], chunk_pos=cfg["chunk_pos"], out_dtype=plc.OUT_F16,
                                 zero_rate_D=zero_rate, sigma_floor=sigma_floor)
    else:
        ctx = plc.Context(T, K, cfg["delta"], chunk_pos=cfg["chunk_pos"], out_dtype=plc.OUT_F16,
                          variant=plc.PRED_DENSE if dense else plc.PRED_TOPK, adaptive=adaptive, zero_rate_D=zero_rate,
                          sigma_floor=sigma_floor)
        ctx.reserve(S * n)
    ctx.set_profiling(True)
    mc = ctx.max_chunks(n)
    kv_bytes = kv.numel() * 2
    st = plc.StreamSet(S * W, mc, int(0.70 * kv_bytes) + S * W * mc * 160 + (1 << 20), dev)
    out = torch.empty_like(kv)
    tokens_per_step = S * n
    count = plc.DebugBuffers(None, None, None, None, 1)               # statistics only: ideal code length of what is coded

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    for i in range(max(warmup, 1)):
        st.total_bytes.zero_()
        if i == 0:
            ctx.stats(reset=True)
        ctx.encode(kv, w["logits"], st, tokens=tok, debug=count if i == 0 else None)
        if i == 0:
            first = ctx.stats(reset=True)                             # one pass with the ideal-length counter on
        ctx.decode(st, w["logits"], out, tokens=tok)
    barrier()
    assert ctx.sync_status() == plc.OK, "device status after warm-up"
    ctx.stats(reset=True)

    uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    sampler = ClockSampler(uuid)
    launches0 = plc.launch_count()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3 * steps)]
    for which in range(3):
        ctx.kernel_ms(which, reset=True)                              # the log of profiled launches starts empty
    barrier()
    t_start = torch.cuda.Event(enable_timing=True); t_end = torch.cuda.Event(enable_timing=True)
    t_start.record()
    gemm_k = None
    for i in range(steps):
        st.total_bytes.zero_()
        ev[3 * i].record()
        ctx.encode(kv, w["logits"], st, tokens=tok)
        ev[3 * i + 1].record()
        ctx.decode(st, w["logits"], out, tokens=tok)
        ev[3 * i + 2].record()
    t_end.record()
    barrier()
    # the library's own events around every fused-kernel launch of the region, read after it
    ek, n_ek = ctx.kernel_ms(0)
    dk, n_dk = ctx.kernel_ms(1)
    if dense or linear:
        gemm_k = ctx.kernel_ms(2)
    launches = plc.launch_count() - launches0
    clocks = sampler.stop()
    total_ms = t_start.elapsed_time(t_end)
    enc_ms = [ev[3 * i].elapsed_time(ev[3 * i + 1]) for i in range(steps)]
    dec_ms = [ev[3 * i + 1].elapsed_time(ev[3 * i + 2]) for i in range(steps)]
    assert ctx.sync_status() == plc.OK, "device status after the timed region"
    stats = ctx.stats()
    payload_per_step = stats.payload_bytes / steps
    chunks_per_step = stats.n_chunks / steps
    sched = ctx.last_schedule() if variant == "topk" else None

    ms_per_step = max_over_ranks(total_ms, dist, dev) / steps
    if shard:
        value = tokens_per_step / (ms_per_step / 1e3)               # one batch, cut across the ranks (strong scaling)
    else:
        value = job_value(world, tokens_per_step, ms_per_step)

    # spot check of the decoded batch (outside the timed region)
    sel = torch.randint(0, n, (64,), device=dev)
    err = float((out[:, :, :, :, sel].float() - kv[:, :, :, :, sel].float()).abs().max())
    if not zero_rate:      # skipped positions are bounded in expectation only
        assert err <= cfg["delta"] * (2.0 ** (adaptive_b0 - 1) if adaptive else 1.0) / 2 + 1e-3 + 8 * 2 ** -11, err

    peak, peak_kind = measured_peaks()
    vecs = S * n * W
    ek_last, dk_last = ek, dk
    sm_mhz = clocks.get("sm_mhz") or 1965.0
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    default_kernels = name == "llama2-7b" and not over and variant == "topk" and not adaptive and not zero_rate and \
        not sigma_floor and layers is None
    roofline = fused_roofline(vecs, K, d, 0 if linear else T.numel() * 2, kv_bytes, payload_per_step, ek, dk, sm_mhz, sms, peak,
                              peak_kind, NCU_DRAM_BYTES_PER_VECTOR if default_kernels else None)
    if roofline["traffic"] is not None:
        roofline["traffic_note"] = NCU_TRAFFIC_NOTE
    if dense or linear:
        gm, n_gemm = gemm_k
        per_launch = 2.0 * L * steps / n_gemm                          # layers one contraction covers (small batches: several)
        tpeak, tkind = tensor_peak()
        if dense:      # 2 * rows * V * (2H*d) flop per layer and direction
            flop = 2.0 * S * n * V * (2 * H * d) * per_launch
        else:          # per layer: rows x (2H*d) x d_model
            flop = 2.0 * S * n * d_model * (2 * H * d) * per_launch
        roofline = {"kernel": "dense_gemm_kernel", "bound": "tensor", "achieved": flop / (gm / 1e3) / 1e12, "peak": tpeak,
                    "unit": "TFLOP/s", "frac": flop / (gm / 1e3) / 1e12 / tpeak, "traffic": None, "peak_kind": tkind,
                    "ms_per_launch": gm, "flop_per_launch": flop, "launches_per_step": n_gemm // steps,
                    "coder_kernels_ms_per_launch": {"encode": ek_last, "decode": dk_last}}
        if linear:
            roofline["flop_per_step_all_contractions"] = 2 * (L * flop / per_launch + 2.0 * S * n * V * d_model +
                                                              2.0 * S * n * V * 256 * ((W + 255) // 256))
    e2e = None
    if want_e2e and not linear:
        del out, st
        torch.cuda.empty_cache()

        def make_ctx(Tslice):
            return plc.Context(Tslice, K, cfg["delta"], chunk_pos=cfg["chunk_pos"], out_dtype=plc.OUT_F16,
                               variant=plc.PRED_DENSE if dense else plc.PRED_TOPK, adaptive=adaptive,
                               zero_rate_D=zero_rate, sigma_floor=sigma_floor)
        e2e = run_e2e(torch, plc, make_ctx, dict(cfg=cfg, T=T, kv=kv, logits=w["logits"]), dev, world, dist, tokens_per_step,
                      tok, e2e_groups if variant == "topk" else 1, e2e_steps, adaptive_b0, bool(shard))

    cpu = None
    if want_cpu and rank == 0 and not linear:
        cpu = cpu_baseline(dict(cfg=cfg, T=T, kv=kv, logits=w["logits"], tokens=w["tokens"]))

    coded_bits = 8.0 * first.payload_bytes
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps, "warmup": warmup,
        "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "strong" if shard else "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": name, "S": S, "n": n, "L": L, "H": H, "d": d, "V": V, "K": K,
                   "delta": cfg["delta"], "chunk_pos": cfg["chunk_pos"], "perplexity": cfg["pp"],
                   "kv_dtype": "f16", "decode_out": "f16", "variant": variant, "adaptive_b0": adaptive_b0,
                   "zero_rate_D": zero_rate, "sigma_floor": sigma_floor,
                   "shard": ("layers %d..%d of %d on rank 0, the other ranks alike" % (*shard_layers(w["cfg"]["L"], world, 0), w["cfg"]["L"])) if shard else None,
                   "layer_subset": list(layers) if layers is not None and not shard else None,
                   "work_queues": None if sched is None else {"queues": sched[0], "sms_per_queue": sched[1]},
                   "l2": "inputs larger than L2 (KV+logits %.1f GB per step)" % ((kv_bytes + w["logits"].numel() * 2) / 1e9)},
        "encode_tokens_s": tokens_per_step / (statistics.mean(enc_ms) / 1e3),
        "decode_tokens_s": tokens_per_step / (statistics.mean(dec_ms) / 1e3),
        "encode_ms": statistics.mean(enc_ms), "decode_ms": statistics.mean(dec_ms),
        "bits_per_token": 8 * (payload_per_step + 12 * chunks_per_step) / tokens_per_step,
        "bits_per_component": 8 * payload_per_step / (vecs * d),
        "ideal_bits_per_component": first.ideal_bits / (vecs * d),
        "ideal_note": "sum of -log2(f / 2^15) + raw bit-plane bits over every component coded in one pass (counted by "
                      "the encode kernel): the -log2 P code length under the coder's model; coded / ideal = %.5f" %
                      (coded_bits / max(first.ideal_bits, 1.0)),
        "paper_bound_bits_per_token": "3.3-4.3 at perplexity 10-20 (Cor. 1: theory for the token stream, not this synthetic KV)",
        "escapes_per_step": stats.n_escapes / steps,
        "skipped_vector_fraction": stats.skipped_vectors / max(stats.coded_vectors, 1),
        "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": launches, "clocks": clocks,
    }
    return line, w


def compact(line, keep=("value", "unit", "ms_per_step", "steps", "warmup", "encode_ms", "decode_ms", "bits_per_token",
                        "bits_per_component", "ideal_bits_per_component", "clocks", "gpu_launches", "latency_ms", "stage_ms",
                        "sweep", "shared_fraction", "relative_storage_vs_no_dedup", "covered_tokens_s", "extrapolated_full",
                        "logp2_stage")):
    """One configuration's record inside the headline line: the figures, its own roofline and clocks."""
    r = {k: line[k] for k in keep if k in line}
    r["config"] = {k: v for k, v in line["config"].items() if v is not None}
    rf = line["roofline"]
    r["roofline"] = {k: rf[k] for k in ("kernel", "bound", "achieved", "peak", "unit", "frac", "ms_per_launch", "accounting",
                                        "encode_kernel_ms", "decode_kernel_ms") if k in rf}
    for sub in ("hbm_compulsory", "fp32_fma"):
        if sub in rf:
            r["roofline"][sub + "_frac"] = rf[sub]["frac"]
    return r


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="own", choices=["own", "reference"])
    ap.add_argument("--workload", default=None,
                    help="tiny | llama2-7b | 70b-longctx | dedup | append; default: llama2-7b as the headline plus, on one "
                         "GPU, a compact record of every benchmark configuration (see --no-configs)")
    ap.add_argument("--no-configs", action="store_true", help="default run: headline only")
    ap.add_argument("--chunk-pos", type=int, default=None)
    ap.add_argument("--e2e-steps", type=int, default=4)
    ap.add_argument("--e2e-groups", type=int, default=4, help="layer groups (streams) of the host-buffer step")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--set", action="append", default=[], help="override a workload field, e.g. --set L=4")
    ap.add_argument("--adaptive", type=int, default=0,
                    help="b0 > 0: surprisal-adaptive step (Def. 7) with hbar = log2(perplexity), cap b0 + 4")
    ap.add_argument("--variant", default="topk", choices=["topk", "dense", "linear"],
                    help="prediction: top-K gather (default), full-vocabulary bf16 tensor-core contraction, or the "
                         "linear-embedding model of Sec. 7.1 (two chained contractions; see --d-model)")
    ap.add_argument("--d-model", type=int, default=4096, help="embedding width of --variant linear")
    ap.add_argument("--rotq", type=int, default=0,
                    help="bits > 0: rotated fixed-rate quantiser on the residual (Prop. 3 step 3) instead of the entropy coder")
    ap.add_argument("--sigma-floor", type=float, default=0.0,
                    help="standard deviation added in quadrature to the mixture's before the scale class is taken")
    ap.add_argument("--zero-rate", type=float, default=0.0,
                    help="D > 0: zero-rate rule (Thm. 3), positions with mixture variance <= D carry no symbols")
    ap.add_argument("--topk-only", action="store_true",
                    help="time the top-K softmax call alone on synthetic logits (V and K of --workload; rows chosen so "
                         "that the input is about 1 GB, larger than L2), with and without the selection")
    ap.add_argument("--shard", default=None, choices=["layers"],
                    help="with --gpus N: cut ONE batch across the ranks by layer (strong scaling) instead of one batch per rank")
    args = ap.parse_args()

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    all_configs = args.workload is None and not args.no_configs and world == 1 and args.variant == "topk" and \
        not (args.set or args.adaptive or args.rotq or args.zero_rate or args.sigma_floor or args.chunk_pos or args.shard)
    if args.workload is None:
        args.workload = "llama2-7b"

    import torch
    from paper_2604_15356_b200 import workloads

    if args.impl == "reference":
        if rank != 0:
            return 0
        return reference_arm(args, workloads)

    import paper_2604_15356_b200 as plc
    plc.build()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    if args.topk_only:
        print(json.dumps(topk_arm(args, torch, plc, workloads, dev)))
        return 0
    if args.workload == "append":
        print(json.dumps(append_arm(args, torch, plc, workloads, dev)))
        return 0
    if args.workload == "dedup":
        print(json.dumps(dedup_arm(args, torch, plc, workloads, dev)))
        return 0
    if args.rotq > 0:
        return rotq_arm(args, torch, plc, workloads, dev)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    over = parse_over(args.set)
    if args.chunk_pos:
        over["chunk_pos"] = args.chunk_pos
    line, w = run_codec(args, torch, plc, workloads, dev, args.workload, over, args.steps, args.warmup, dist, world, rank,
                        variant=args.variant, d_model=args.d_model, adaptive_b0=args.adaptive, zero_rate=args.zero_rate,
                        sigma_floor=args.sigma_floor, shard=args.shard, want_e2e=not args.no_e2e,
                        want_cpu=world == 1 and not args.no_cpu_baseline, e2e_steps=args.e2e_steps, e2e_groups=args.e2e_groups)
    if all_configs:
        del w
        torch.cuda.empty_cache()
        line["configs"] = every_config(args, torch, plc, workloads, dev, line)
    if rank == 0:
        print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


def every_config(args, torch, plc, workloads, dev, headline):
    """One compact record per benchmark configuration, measured in this same process after the
    headline (inputs regenerated per configuration; device memory is released in between)."""
    import gc
    out = {"llama2-7b": compact(headline)}

    def free():
        gc.collect()
        torch.cuda.empty_cache()

    t0 = time.perf_counter()
    line, w = run_codec(args, torch, plc, workloads, dev, "tiny", {}, 20, 5)
    out["tiny"] = compact(line)
    out["tiny"]["note"] = "1024 vectors: two kernel launches of a few microseconds of work each; launch-latency bound"
    del w; free()
    # 70B long context: top-K over all 80 layers, then the full-vocabulary contraction on 4 of the 80 layers
    line, w = run_codec(args, torch, plc, workloads, dev, "70b-longctx", {}, 3, 3)
    out["70b-longctx topk"] = compact(line)
    Lfull, sub = w["cfg"]["L"], 4
    line, _ = run_codec(args, torch, plc, workloads, dev, "70b-longctx", {}, 2, 3, variant="dense", w=w, layers=(0, sub))
    r = compact(line)
    r["extrapolated_full"] = {"layers": Lfull, "ms_per_step": line["ms_per_step"] * Lfull / sub,
                              "value": line["value"] * sub / Lfull,
                              "note": "the layers are independent launches of the same shapes: time scales by %d / %d" % (Lfull, sub)}
    out["70b-longctx dense (4 of 80 layers)"] = r
    del w; free()
    a = argparse.Namespace(**vars(args)); a.steps, a.warmup, a.set = 2, 1, []
    out["dedup"] = compact(dedup_arm(a, torch, plc, workloads, dev))
    free()
    a = argparse.Namespace(**vars(args)); a.steps, a.set = 17, []
    out["append"] = compact(append_arm(a, torch, plc, workloads, dev, sweep=True))
    free()
    out["seconds_for_the_other_configs"] = time.perf_counter() - t0
    return out


def append_run(torch, plc, synth, dev, cfg, T, nsteps, seed, pp=None, delta=None, zero_clock=True):
    """One run of the append path: B sessions grow by one token per plc_append_step for nsteps steps
    (the first chunk's steps are warm-up).  Returns latencies (ms, sorted), seal-step latencies, stats."""
    B, L, H, d, V, K, CP = cfg["S"], cfg["L"], cfg["H"], cfg["d"], cfg["V"], cfg["K"], cfg["chunk_pos"]
    pp = cfg["pp"] if pp is None else pp
    delta = cfg["delta"] if delta is None else delta
    W = 2 * L * H
    table = synth.markov_table(V, pp, seed, device=dev)
    tokens = synth.sample_tokens(table, B, nsteps, seed + 1)
    logits = synth.position_logits(table, tokens)                       # [B][nsteps][V]
    del table
    ctx = plc.Context(T, K, delta, chunk_pos=CP)
    sb = ctx.new_session_batch(B, nsteps // CP + 1, int(nsteps * B * W * d * 1.45) + (1 << 20))
    g = torch.Generator(device=dev); g.manual_seed(seed + 3)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nsteps)]
    launches0 = plc.launch_count()
    for i in range(nsteps):
        tok = tokens[:, i].to(torch.int64)
        kv_step = (T[:, :, :, tok, :].permute(0, 1, 3, 2, 4).float() +
                   cfg["sigma"] * torch.randn(L, 2, B, H, d, device=dev, generator=g)).to(torch.float16).contiguous()
        lg = logits[:, i, :].contiguous()
        torch.cuda.synchronize()
        ev[i][0].record()
        ctx.append_step(sb, kv_step, lg)
        ev[i][1].record()
    torch.cuda.synchronize()
    assert ctx.sync_status() == plc.OK
    lat = sorted(a.elapsed_time(b) for a, b in ev[CP:])                 # first chunk = warm-up
    seal = sorted(ev[i][0].elapsed_time(ev[i][1]) for i in range(CP, nsteps) if (i + 1) % CP == 0)
    st = ctx.stats()
    return dict(lat=lat, seal=seal, stats=st, launches=plc.launch_count() - launches0, W=W,
                bits_per_token=8 * (st.payload_bytes + 12 * st.n_chunks) / max(st.coded_vectors / W, 1),
                bits_per_component=8 * st.payload_bytes / max(st.coded_vectors * d, 1))


def append_arm(args, torch, plc, workloads, dev, sweep=False):
    """Decode-time append: B sessions grow by one token per plc_append_step; per-step latency.
    `--steps` counts groups of chunk_pos append steps (one chunk seal per group); the first group is
    warm-up.  With sweep=True the perplexity x step grid of the streaming configuration is added
    (p50 / p99 latency and bits per component of every cell)."""
    from paper_2604_15356_b200 import synth
    cfg = dict(workloads.CONFIGS["append"]); cfg.update(parse_over(args.set))
    B, L, H, d, V, K, CP = cfg["S"], cfg["L"], cfg["H"], cfg["d"], cfg["V"], cfg["K"], cfg["chunk_pos"]
    nsteps = CP * max(args.steps, 2)
    seed = 20260419
    T = synth.make_tables(L, H, V, d, seed + 2, device=dev)
    uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    sampler = ClockSampler(uuid)
    r = append_run(torch, plc, synth, dev, cfg, T, nsteps, seed)
    clocks = sampler.stop()
    lat, seal, W = r["lat"], r["seal"], r["W"]
    mean_ms = sum(lat) / len(lat)
    peak, kind = measured_peaks()
    gathered = B * W * K * d * 2
    p50 = lat[len(lat) // 2]
    line = {"metric": METRIC, "value": B / (mean_ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": nsteps - CP, "warmup": CP,
            "ms_per_step": mean_ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "append", "B": B, "L": L, "H": H, "d": d, "V": V, "K": K, "delta": cfg["delta"],
                       "chunk_pos": CP, "perplexity": cfg["pp"], "encode_only": True,
                       "l2": "random rows of a %.1f GB table set, larger than L2" % (T.numel() * 2 / 1e9)},
            "latency_ms": {"p50": p50, "p99": lat[int(len(lat) * 0.99)], "max": lat[-1],
                           "seal_steps_mean": sum(seal) / max(len(seal), 1)},
            "bits_per_token": r["bits_per_token"], "bits_per_component": r["bits_per_component"],
            "roofline": {"kernel": "append_quantise_kernel", "bound": "hbm", "achieved": gathered / (p50 / 1e3) / 1e9,
                         "peak": peak, "unit": "GB/s", "frac": gathered / (p50 / 1e3) / 1e9 / peak,
                         "traffic": None, "peak_kind": kind, "ms_per_launch": p50,
                         "accounting": "random 256-byte T rows per step (B*W*K*d*2 bytes, tables far larger than L2: every "
                                       "row is an HBM read) over the median whole-step time"},
            "gpu_launches": r["launches"], "clocks": clocks}
    if sweep:
        grid = {}
        for pp in (4.0, 12.0, 20.0, 50.0):
            for delta in (0.005, 0.02, 0.08):
                rr = append_run(torch, plc, synth, dev, cfg, T, CP * 9, seed + int(pp), pp=pp, delta=delta)
                l2 = rr["lat"]
                grid["pp=%g delta=%g" % (pp, delta)] = {"p50_ms": l2[len(l2) // 2], "p99_ms": l2[int(len(l2) * 0.99)],
                                                         "bits_per_component": rr["bits_per_component"],
                                                         "bits_per_token": rr["bits_per_token"]}
        line["sweep"] = grid
    return line


def dedup_arm(args, torch, plc, workloads, dev):
    """Prefix dedup followed by delta coding of the tails, at the shapes of `llama3-8b-dedup`: S
    sessions whose system prefixes come from a seeded 8-leaf prefix trie.  One step = log2 P of every
    token (top-K softmax kernel), batched LCP / trie metric / parents (plc_prefix_dedup), clusters
    (plc_prefix_clusters), then encode and decode of the non-shared tails, the sessions taken in
    batches of Sb (the logits of all sessions do not fit in memory at once).  Only library calls are
    timed (CUDA events around them); the synthetic inputs of a batch are generated between them.
    `--steps` repeats the whole pipeline; the first `--warmup` repetitions are not counted."""
    from paper_2604_15356_b200 import synth
    cfg = dict(workloads.CONFIGS["llama3-8b-dedup"]); cfg.update(parse_over(args.set))
    S, n, L, H, d, V, K, CP = cfg["S"], cfg["n"], cfg["L"], cfg["H"], cfg["d"], cfg["V"], cfg["K"], cfg["chunk_pos"]
    Sb = int(cfg.get("Sb", 8))
    assert S % Sb == 0
    W = 2 * L * H
    seed = 20260417
    table = synth.markov_table(V, cfg["pp"], seed, alpha=cfg["alpha"], max_states=cfg.get("max_states", 4096), device=dev)
    seg_lo, seg_hi = int(cfg.get("seg_lo", 128)), int(cfg.get("seg_hi", 1024))
    tokens, keys, leaf, plen = synth.trie_sessions(table, S, n, seed + 1, seg_lo, seg_hi)
    T = synth.make_tables(L, H, V, d, seed + 2, device=dev)
    ctx = plc.Context(T, K, cfg["delta"], chunk_pos=CP, out_dtype=plc.OUT_F16)
    ctx.reserve(Sb * n)
    mc = ctx.max_chunks(n)
    kv = torch.empty(L, 2, Sb, H, n, d, dtype=torch.float16, device=dev)
    out = torch.empty_like(kv)
    st = plc.StreamSet(Sb * W, mc, int(0.70 * kv.numel() * 2) + (1 << 20), dev)
    lens = torch.full((S,), n, dtype=torch.int32, device=dev)
    logp2 = torch.empty(S, n, dtype=torch.float32, device=dev)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    reps, stats_keep = [], None
    launches0 = plc.launch_count()
    sampler = ClockSampler("GPU-" + str(torch.cuda.get_device_properties(dev).uuid))
    for rep in range(args.warmup + args.steps):
        t = {"logp2": 0.0, "dedup": 0.0, "encode": 0.0, "decode": 0.0}
        spans = []

        def timed(key, fn):
            a, b = ev(), ev()
            a.record(); r = fn(); b.record()
            spans.append((key, a, b))
            return r
        for b0 in range(0, S, Sb):                                     # stage 1: edge weights of the trie
            lg = synth.position_logits(table, tokens[b0:b0 + Sb])
            o = timed("logp2", lambda: ctx.topk_softmax(lg, tokens[b0:b0 + Sb].reshape(-1), want=("logp2",)))
            logp2[b0:b0 + Sb] = o["logp2"].view(Sb, n)
            del lg
        lcp, dT, parent, shared = timed("dedup", lambda: ctx.prefix_dedup(tokens, lens, logp2))
        cl, ce, be = timed("dedup", lambda: ctx.prefix_clusters(lcp, dT, float(cfg.get("cluster_bits", 64.0))))
        ctx.stats(reset=True)
        worst = 0.0
        for b0 in range(0, S, Sb):                                     # stage 2: tails only
            tb = tokens[b0:b0 + Sb]
            lg = synth.position_logits(table, tb)
            synth.make_kv(T, tb, cfg["sigma"], seed + 3, keys=keys[b0:b0 + Sb], out=kv)
            pb, pe = shared[b0:b0 + Sb].contiguous(), lens[b0:b0 + Sb].contiguous()
            st.total_bytes.zero_()
            timed("encode", lambda: ctx.encode(kv, lg, st, pb, pe))
            out.zero_()
            timed("decode", lambda: ctx.decode(st, lg, out, pb, pe))
            torch.cuda.synchronize()
            assert ctx.sync_status() == plc.OK
            for s_ in range(Sb):                                       # decoded tails against the input
                m = int(pb[s_])
                if m < n:
                    worst = max(worst, float((out[:, :, s_, :, m:].float() - kv[:, :, s_, :, m:].float()).abs().max()))
            del lg
        torch.cuda.synchronize()
        for key, a, b in spans:
            t[key] += a.elapsed_time(b)
        assert worst <= cfg["delta"] / 2 + 1e-3 + 8 * 2 ** -11, worst
        if rep >= args.warmup:
            reps.append(t)
            stats_keep = ctx.stats()
    launches = plc.launch_count() - launches0
    clocks = sampler.stop()
    mean = {k: sum(r[k] for r in reps) / len(reps) for k in reps[0]}
    total_ms = sum(mean.values())
    sh = shared.cpu().numpy().astype("int64")
    coded = int((n - sh).sum())
    peak, kind = measured_peaks()
    logits_bytes = 2.0 * S * n * V
    row_bytes = stats_keep.coded_vectors * (K * d * 2.0 + 2.0 * d) + stats_keep.payload_bytes
    line = {"metric": METRIC, "value": coded / (total_ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "encode_ms": mean["encode"], "decode_ms": mean["decode"],
            "config": {"workload": "dedup (llama3-8b-dedup shapes)", "S": S, "n": n, "L": L, "H": H, "d": d, "V": V, "K": K,
                       "delta": cfg["delta"], "chunk_pos": CP, "perplexity": cfg["pp"], "session_batch": Sb,
                       "prefix_trie": "15 segments of U[%d,%d] tokens, 8 leaves" % (seg_lo, seg_hi),
                       "value_counts": "coded (non-shared) token positions; shared prefixes cost no bits and no time"},
            "stage_ms": mean,
            "covered_tokens_s": S * n / (total_ms / 1e3),
            "shared_fraction": float(sh.sum()) / (S * n), "mean_shared_len": float(sh.mean()),
            "sessions_with_parent": int((parent.cpu().numpy() >= 0).sum()),
            "clusters_at_%g_bits" % float(cfg.get("cluster_bits", 64.0)): int(len(set(cl.cpu().numpy().tolist()))),
            "bits_per_token": 8 * (stats_keep.payload_bytes + 12 * stats_keep.n_chunks) / max(coded, 1),
            "bits_per_component": 8 * stats_keep.payload_bytes / max(stats_keep.coded_vectors * d, 1),
            "relative_storage_vs_no_dedup": coded / float(S * n),
            # dominant kernels: the fused encode / decode, whose K*d*2 B of candidate rows per vector are HBM reads
            # here (tables in flight far beyond L2, candidates spread over the vocabulary)
            "roofline": {"kernel": "decode_kernel" if mean["decode"] >= mean["encode"] else "encode_kernel", "bound": "hbm",
                         "achieved": row_bytes / (max(mean["encode"], mean["decode"]) / 1e3) / 1e9, "peak": peak, "unit": "GB/s",
                         "frac": row_bytes / (max(mean["encode"], mean["decode"]) / 1e3) / 1e9 / peak, "traffic": None,
                         "peak_kind": kind, "ms_per_launch": max(mean["encode"], mean["decode"]) / (S // Sb),
                         "accounting": "K*d*2 B of random T rows + 2*d B of KV per coded vector + the coded bytes, over the slower "
                                       "of encode / decode (top-K of the coded positions included)"},
            "logp2_stage": {"kernel": "topk_stream_kernel", "bound": "hbm", "achieved": logits_bytes / (mean["logp2"] / 1e3) / 1e9,
                            "peak": peak, "unit": "GB/s", "frac": logits_bytes / (mean["logp2"] / 1e3) / 1e9 / peak,
                            "ms_per_launch": mean["logp2"] / (S // Sb),
                            "accounting": "logits read once (2*S*n*V bytes) over the summed log2 P launches; the encode and "
                                          "decode calls scan the logits of the coded positions once more each"},
            "gpu_launches": launches, "clocks": clocks}
    return line


def topk_arm(args, torch, plc, workloads, dev):
    """The top-K softmax call by itself: N rows of V seeded logits (N*V*2 bytes of about 1 GB, so every call
    reads its input from HBM), once with the K largest, their weights, lse, Z_k and log2 P asked for, once
    with lse / log2 P only.  CUDA events around 100 x `--steps` calls after `--warmup`."""
    shapes = {"dedup": (128256, 64), "tiny": (256, 16)}
    V, K = shapes.get(args.workload, (32000, 64))
    over = parse_over(args.set)
    V, K = int(over.get("V", V)), int(over.get("K", K))
    N = max(1, int(over.get("N", (1 << 30) // (2 * V))))
    g = torch.Generator(device=dev); g.manual_seed(20260415)
    logits = (torch.randn(N, V, device=dev, generator=g) * 3.0).to(torch.float16)
    tokens = torch.randint(0, V, (N,), device=dev, dtype=torch.int32, generator=g)
    ctx = plc.Context(torch.zeros(1, 2, 1, V, 32, dtype=torch.float16, device=dev), K, 0.02)
    peak, kind = measured_peaks()
    uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    sampler = ClockSampler(uuid)
    launches0 = plc.launch_count()
    out = {}
    for name, want in (("with_selection", ("idx", "w", "lse", "zk", "logp2")), ("lse_logp2_only", ("lse", "logp2"))):
        for _ in range(max(args.warmup, 3)):
            ctx.topk_softmax(logits, tokens, want=want)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        calls = 100 * args.steps                       # long enough for the clock sampler to see the region
        e0.record()
        for _ in range(calls):
            ctx.topk_softmax(logits, tokens, want=want)
        e1.record(); torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / calls
        gbs = N * V * 2 / (ms / 1e3) / 1e9
        out[name] = {"ms_per_call": ms, "achieved": gbs, "unit": "GB/s", "frac": gbs / peak}
    assert ctx.sync_status() == plc.OK
    clocks = sampler.stop()
    sel = out["with_selection"]
    return {"metric": "logits rows/s through the top-K softmax call", "value": N / (sel["ms_per_call"] / 1e3), "unit": "rows/s",
            "n_gpus": 1, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": sel["ms_per_call"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "top-K softmax alone", "rows": N, "V": V, "K": K, "l2": "input of %.2f GB, larger than L2" % (N * V * 2 / 1e9)},
            "roofline": {"kernel": "topk_stream_kernel" if K <= 128 else "topk_softmax_kernel", "bound": "hbm",
                         "achieved": sel["achieved"], "peak": peak, "unit": "GB/s", "frac": sel["frac"], "traffic": None,
                         "peak_kind": kind, "accounting": "the logits once (rows * V * 2 bytes) over the whole call (all its kernels)"},
            "modes": out, "gpu_launches": plc.launch_count() - launches0, "clocks": clocks}


def rotq_arm(args, torch, plc, workloads, dev):
    """Predict, rotate and quantise the residual to `--rotq` bits per component (fixed-size records),
    then decode; same workloads, same prediction kernels, no entropy coder."""
    w = workloads.build(args.workload, dev, seed=20260415, **parse_over(args.set))
    cfg = w["cfg"]
    S, n, L, H, d, V, K = cfg["S"], cfg["n"], cfg["L"], cfg["H"], cfg["d"], cfg["V"], cfg["K"]
    W = 2 * L * H
    ctx = plc.Context(w["T"], K, cfg["delta"], chunk_pos=cfg["chunk_pos"], out_dtype=plc.OUT_F16)
    ctx.reserve(S * n)
    g = torch.Generator().manual_seed(7)
    params = ctx.rotq_params(args.rotq, torch.randint(0, 2, (d,), generator=g).tolist())
    rb = ctx.rotq_record_bytes(args.rotq)
    records = torch.empty(S * W * n * rb, dtype=torch.uint8, device=dev)
    out = torch.empty_like(w["kv"])
    for _ in range(max(args.warmup, 1)):
        ctx.encode_rotq(w["kv"], w["logits"], params, records)
        ctx.decode_rotq(records, w["logits"], params, out)
    torch.cuda.synchronize()
    assert ctx.sync_status() == plc.OK
    uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    sampler = ClockSampler(uuid)
    launches0 = plc.launch_count()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * args.steps + 1)]
    ev[0].record()
    for i in range(args.steps):
        ctx.encode_rotq(w["kv"], w["logits"], params, records)
        ev[2 * i + 1].record()
        ctx.decode_rotq(records, w["logits"], params, out)
        ev[2 * i + 2].record()
    torch.cuda.synchronize()
    clocks = sampler.stop()
    launches = plc.launch_count() - launches0
    enc = statistics.mean(ev[2 * i].elapsed_time(ev[2 * i + 1]) for i in range(args.steps))
    dec = statistics.mean(ev[2 * i + 1].elapsed_time(ev[2 * i + 2]) for i in range(args.steps))
    ms = ev[0].elapsed_time(ev[-1]) / args.steps
    diff = out.float() - w["kv"].float()
    rms = float(diff.pow(2).mean().sqrt())
    peak, kind = measured_peaks()
    vecs = S * n * W
    sec = max(enc, dec) / 1e3                                   # per call, top-K included
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    sm_mhz = clocks.get("sm_mhz") or clocks.get("sm_max_mhz") or 1965.0
    flop_peak = 2.0 * sms * 128 * sm_mhz * 1e6 / 1e12
    flop_ach = 2.0 * vecs * K * d / sec / 1e12
    bytes_c = w["kv"].numel() * 2 + w["T"].numel() * 2 + vecs * rb
    line = {"metric": METRIC, "value": S * n / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": args.workload, "S": S, "n": n, "L": L, "H": H, "d": d, "V": V, "K": K, "quantiser": "rotated, %d bits" % args.rotq,
                       "chunk_pos": cfg["chunk_pos"], "l2": "inputs larger than L2"},
            "encode_ms": enc, "decode_ms": dec, "bits_per_component": 8.0 * rb / d, "bits_per_token": 8.0 * rb * W,
            "rms_error": rms, "max_error": float(diff.abs().max()),
            "roofline": {"kernel": "rotq_kernel", "bound": "alu", "achieved": flop_ach, "peak": flop_peak, "unit": "TFLOP/s",
                         "frac": flop_ach / flop_peak, "traffic": None,
                         "peak_kind": "SMs x 128 lanes x 2 flop x sampled SM clock (%d x %.0f MHz); the mixture's K*d FMAs per vector" % (sms, sm_mhz),
                         "hbm_compulsory": {"bytes_per_launch": bytes_c, "achieved": bytes_c / sec / 1e9, "peak": peak, "unit": "GB/s",
                                            "frac": bytes_c / sec / 1e9 / peak, "peak_kind": kind},
                         "accounting": "per call (top-K included); same gather and prediction as the fused kernels, no entropy coder"},
            "gpu_launches": launches, "clocks": clocks}
    print(json.dumps(line))
    return 0


def run_e2e(torch, plc, make_ctx, w, dev, world, dist, tokens_per_step, tok=None, groups=4, e2e_steps=2, adaptive_b0=0,
            sharded=False):
    """Same step with HOST buffers: pinned inputs are copied in, the coded bytes and index are
    copied out and back in, the decoded KV is copied out -- all inside the timed region.  The
    layers are cut into groups, each with its own context and CUDA stream, so that the copies of
    one group overlap the kernels and the opposite-direction copies of the others; consecutive steps
    are not joined (a step's output copies run beside the next step's input copies), only the end of
    the timed region is."""
    cfg = w["cfg"]
    S, n, L, H, d = cfg["S"], cfg["n"], cfg["L"], cfg["H"], cfg["d"]
    G = groups if L % groups == 0 else 1
    Lg = L // G
    kv_h = w["kv"].cpu().pin_memory()
    lg_h = w["logits"].cpu().pin_memory()
    kvo_h = torch.empty_like(kv_h).pin_memory()
    kv_d, out_d = torch.empty_like(w["kv"]), torch.empty_like(w["kv"])
    lg_d = [torch.empty_like(w["logits"]), torch.empty_like(w["logits"])]   # steps alternate between two logits buffers
    ctxs, sts, pay_h, off_h, nby_h, tot_h, streams = [], [], [], [], [], [], []
    for g in range(G):
        c = make_ctx(w["T"][g * Lg:(g + 1) * Lg])
        c.reserve(S * n)
        ctxs.append(c)
        st = plc.StreamSet(S * c.W, c.max_chunks(n), int(0.70 * kv_h.numel() * 2 / G) + (1 << 20), dev)
        sts.append(st)
        pay_h.append(torch.empty(st.payload.numel(), dtype=torch.uint8).pin_memory())
        off_h.append(torch.empty_like(st.chunk_offset, device="cpu").pin_memory())
        nby_h.append(torch.empty_like(st.chunk_bytes, device="cpu").pin_memory())
        tot_h.append(torch.zeros(1, dtype=torch.int64).pin_memory())
        streams.append(torch.cuda.Stream(device=dev))
    copy_stream = torch.cuda.Stream(device=dev)
    ev_lg = [torch.cuda.Event(), torch.cuda.Event()]
    done = [[torch.cuda.Event() for _ in range(G)] for _ in range(2)]

    def step(i):
        """Step i.  Nothing joins the groups between steps: a group goes on to the next step's input copy
        as soon as its own output copy is queued, so one group's device-to-host copy of decoded KV runs
        beside another group's host-to-device copy of the next step's input."""
        b = i & 1
        with torch.cuda.stream(copy_stream):
            for g in range(G):
                copy_stream.wait_event(done[b][g])            # step i - 2 is through with this logits buffer
            lg_d[b].copy_(lg_h, non_blocking=True)
            ev_lg[b].record(copy_stream)
        for g in range(G):
            lo, hi = g * Lg, (g + 1) * Lg
            with torch.cuda.stream(streams[g]):
                streams[g].wait_event(ev_lg[b])
                kv_d[lo:hi].copy_(kv_h[lo:hi], non_blocking=True)
                sts[g].total_bytes.zero_()
                ctxs[g].encode(kv_d[lo:hi], lg_d[b], sts[g], tokens=tok)
                tot_h[g].copy_(sts[g].total_bytes, non_blocking=True)
        used_all = 0
        for g in range(G):
            lo, hi = g * Lg, (g + 1) * Lg
            streams[g].synchronize()                          # the byte count decides how much to copy out
            used = int(tot_h[g][0]); used_all += used
            st = sts[g]
            with torch.cuda.stream(streams[g]):
                pay_h[g][:used].copy_(st.payload[:used], non_blocking=True)
                off_h[g].copy_(st.chunk_offset, non_blocking=True); nby_h[g].copy_(st.chunk_bytes, non_blocking=True)
                st.payload[:used].copy_(pay_h[g][:used], non_blocking=True)
                st.chunk_offset.copy_(off_h[g], non_blocking=True); st.chunk_bytes.copy_(nby_h[g], non_blocking=True)
                ctxs[g].decode(st, lg_d[b], out_d[lo:hi], tokens=tok)
                kvo_h[lo:hi].copy_(out_d[lo:hi], non_blocking=True)
                done[b][g].record(streams[g])
        return used_all

    def join():
        main = torch.cuda.current_stream()
        for g in range(G):
            main.wait_stream(streams[g])

    used = step(0)
    join()
    torch.cuda.synchronize()
    for c in ctxs:
        assert c.sync_status() == plc.OK
    err = float((kvo_h[:, :, :, :, :64].float() - kv_h[:, :, :, :, :64].float()).abs().max())
    assert err <= cfg["delta"] * (2.0 ** (adaptive_b0 - 1) if adaptive_b0 > 0 else 1.0) / 2 + 1e-3 + 8 * 2 ** -11, err
    kvo_h.zero_()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    for i in range(e2e_steps):
        used = step(i + 1)
    join()
    t1.record()
    torch.cuda.synchronize()
    for c in ctxs:
        assert c.sync_status() == plc.OK
    err = float((kvo_h[:, :, :, :, -64:].float() - kv_h[:, :, :, :, -64:].float()).abs().max())     # the last timed step's output
    assert err <= cfg["delta"] * (2.0 ** (adaptive_b0 - 1) if adaptive_b0 > 0 else 1.0) / 2 + 1e-3 + 8 * 2 ** -11, err
    ms = max_over_ranks(t0.elapsed_time(t1) / e2e_steps, dist, dev)
    idx_bytes = sum(o.numel() * 8 + b.numel() * 4 for o, b in zip(off_h, nby_h))
    return {"value": tokens_per_step / (ms / 1e3) if sharded else job_value(world, tokens_per_step, ms), "unit": UNIT,
            "ms_per_step": ms,
            "h2d_bytes_per_step": kv_h.numel() * 2 + lg_h.numel() * 2 + used + idx_bytes,
            "d2h_bytes_per_step": used + idx_bytes + 8 * G + kvo_h.numel() * 2, "steps": e2e_steps,
            "layer_groups": G}


def reference_arm(args, workloads):
    """The reference arm is the CPU oracle as it stands, on a bounded sample of the same workload."""
    cfg = dict(workloads.CONFIGS[args.workload])
    layers, pos = 1, min(cfg["n"], 64)
    # the sample is built on the CPU at the sample's own size (same recipe)
    w = workloads.build(args.workload, "cpu", seed=20260415, S=1, n=pos, L=layers, max_states=64)
    w["cfg"]["L"] = cfg["L"]                                  # the rate is scaled to the full number of streams
    import oracle
    cores = oracle.host_cores()
    for _ in range(min(args.warmup, 1)):
        oracle_sample_rate(w, pos, layers)
    rates = []
    t0 = time.perf_counter()
    for _ in range(args.steps):
        rates.append(oracle_sample_rate(w, pos, layers, workers=cores if cfg["H"] > 1 else 1))
    dt = (time.perf_counter() - t0) / max(args.steps, 1)
    value = statistics.mean(r["value"] for r in rates)
    W = 2 * cfg["L"] * cfg["H"]
    sample = (f"1 session, {pos} positions, {layers} of {cfg['L']} layers, all heads "
              f"({rates[0]['vectors']} vectors per step); rate scaled by W={W} vectors per KV token")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "sample": sample},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": rates[0]["workers"], "host_cores": cores,
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line))
    return 0


if __name__ == "__main__":
    sys.exit(main())
