"""Benchmark: ray-segments/s of the column-density trace at 512^3, Nside 1.

Workload: 512^3 uniform leaf grid (134,217,728 leaves, Morton keys), lognormal
density (P(k) ~ k^-4, sigma 2), 4 FP32 species; sources = every leaf centre;
12 HEALPix Nside-1 directions (1.61e9 rays); F32-Kahan columns (25.8 GB).
A step is one full trace of that workload.  Inputs (3.4 GB tree, 3.2 GB
sources) and output are far larger than L2, so no flush is needed between
steps.  Also reported: the FP64 form, the adjoint / forward time ratio, an
end-to-end number with host buffers, and the CPU oracle on a sample.

python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

FP32_OPS_PER_SEGMENT = 4 * 4  # a Kahan step for each of 4 species
BYTES_PER_SEGMENT = 8 + 1 + 4 * 4  # key + level + 4 FP32 densities (algorithmic)
NSIDE = 1
LEVEL = 9
E2E_CHUNK = 1 << 23  # sources per pipeline chunk of the host-buffer call (16 chunks at 512^3)
METRIC = "ray-segments/s at 512^3 Nside=1 (FP32-Kahan vs FP64 @1e-5 rel); adjoint/fwd time"


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=5)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--level", type=int, default=LEVEL, help="uniform grid level (9 = 512^3)")
    p.add_argument("--no-extras", action="store_true", help="skip FP64 form, adjoint, e2e, CPU baseline")
    p.add_argument("--cpu-seconds", type=float, default=12.0, help="target CPU time of the oracle sample")
    p.add_argument("--amr-base", type=int, default=128, help="base size of the amr128 workload's cloud")
    p.add_argument("--workload", default="uniform512",
                   choices=["uniform512", "amr128", "batched64", "adjoint_amr64", "dualgrid256", "angular128",
                            "search", "adjoint_uniform"],
                   help="uniform512 is the benchmark; the others run one secondary workload alone")
    return p.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            m = json.load(f)
        return float(m["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# The sources the bench kernel (the forward trace) is compiled and launched
# from: its device code, its translation unit and the launch code (the
# launch shape, the ray order and the density check live in rt_api.cu and
# rt_octree.cu).
FORWARD_SOURCES = ("paper_2605_09882_gb300/csrc/rt_device.cuh", "paper_2605_09882_gb300/csrc/rt_kernels.cuh",
                   "paper_2605_09882_gb300/csrc/rt_internal.h", "paper_2605_09882_gb300/csrc/rt_forward.cu",
                   "paper_2605_09882_gb300/csrc/rt_beam.cu",
                   "paper_2605_09882_gb300/csrc/rt_api.cu", "paper_2605_09882_gb300/csrc/rt_octree.cu")


def kernel_source_sha() -> str:
    h = hashlib.sha256()
    for n in FORWARD_SOURCES:
        with open(os.path.join(ROOT, n), "rb") as f:
            h.update(n.encode() + f.read())
    return h.hexdigest()[:16]


def kernel_profile(name="trace_f32k_uniform512"):
    """Per-segment counters of a trace kernel from a committed ncu summary
    (warp instructions and DRAM bytes per segment), if it was taken from the
    current kernel sources (else None)."""
    path = os.path.join(ROOT, "profiles", name + ".json")
    try:
        with open(path) as f:
            m = json.load(f)
        if m.get("kernel_source_sha") == kernel_source_sha():
            return {"warp_inst_per_segment": float(m["warp_inst_per_segment"]),
                    "dram_bytes_per_segment": float(m["dram_bytes_per_segment"]),
                    "issue_active_pct": m.get("issue_active_pct"), "lts_hit_pct": m.get("lts_hit_pct"),
                    "warp_exec_efficiency": m.get("warp_exec_efficiency")}
    except Exception:
        pass
    return None


def profiled_traffic(segments=None):
    """DRAM bytes of one launch of `segments` segments from the committed
    summary (scaled per segment), or None when the sources changed since."""
    p = kernel_profile()
    if p is None or segments is None:
        return None
    return p["dram_bytes_per_segment"] * segments


class Clocks:
    """nvidia-smi samples during the timed region."""

    def __init__(self, index: int):
        self.path = tempfile.mktemp(suffix=".csv")
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.f = open(self.path, "w")
            self.p = subprocess.Popen(["nvidia-smi", f"--id={index}", f"--query-gpu={q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None

    def stop(self):
        if not self.p:
            return None
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except Exception:
            self.p.kill()
        self.f.close()
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx = max(mx, float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def trace_roofline(seg_per_launch, launch_s, clk, hbm_gbs, hbm_kind, dev):
    """The bound of the trace kernel: the FP32 pipe.  A segment takes 16 FP32
    operations at 4 species (a Kahan step is a fused multiply-add, an addition and two
    subtractions), and an SM does 128 a cycle: the peak is SMs x 128 x the SM
    clock (the median sampled under load).  Beside it: the issue rate (segments/s x
    warp instructions per segment, ncu, 256^3 capture of the same sources,
    against four warp instructions a cycle and SM), the effective HBM fraction
    of the 25 algorithmic bytes per segment (above 1 because L2 serves the
    re-reads) and the fraction of HBM bandwidth the measured DRAM traffic uses."""
    import torch
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    mhz = (clk or {}).get("sm_mhz") or 2070.0
    issue_peak = sms * 4 * mhz * 1e6
    prof = kernel_profile()
    seg_rate = seg_per_launch / launch_s
    eff = BYTES_PER_SEGMENT * seg_rate / 1e9
    fma_peak = sms * 128 * mhz * 1e6
    r = {"bound": "fp32", "achieved": seg_rate * FP32_OPS_PER_SEGMENT, "peak": fma_peak, "unit": "FP32 operations/s",
         "frac": seg_rate * FP32_OPS_PER_SEGMENT / fma_peak,
         "traffic": None, "peak_kind": f"derived: {sms} SMs x 128 x {mhz:.0f} MHz (median under load)",
         "fp32_ops_per_segment": FP32_OPS_PER_SEGMENT,
         "issue": {"achieved": None, "peak": issue_peak, "unit": "warp-instructions/s", "frac": None},
         "warp_inst_per_segment": None, "dram_frac": None,
         "effective_hbm": {"bytes_per_segment": BYTES_PER_SEGMENT, "achieved": eff, "peak": hbm_gbs, "unit": "GB/s",
                           "frac": eff / hbm_gbs, "peak_kind": hbm_kind},
         "kernel": "k_beam<S=4> (F32K forward, cube, sources at one offset: step tables)",
         "profile": "profiles/trace_f32k_uniform512.md (256^3 capture, per segment)"}
    if prof is not None:
        r["warp_inst_per_segment"] = prof["warp_inst_per_segment"]
        r["issue"]["achieved"] = seg_rate * prof["warp_inst_per_segment"]
        r["issue"]["frac"] = r["issue"]["achieved"] / issue_peak
        r["traffic"] = prof["dram_bytes_per_segment"] * seg_per_launch
        r["dram_frac"] = r["traffic"] / launch_s / (hbm_gbs * 1e9)
        r["ncu"] = {"issue_active_pct": prof["issue_active_pct"], "lts_hit_pct": prof["lts_hit_pct"],
                    "warp_exec_efficiency": prof["warp_exec_efficiency"],
                    "dram_gbs": r["traffic"] / launch_s / 1e9}
    return r


# ------------------------------------------------------------------ oracle

def oracle_sample(keys_h, lev_h, dens_h64, n_leaves, seconds, seed=5, level=LEVEL):
    """Times the oracle on a random sample of sources sized to ~`seconds`."""
    import oracle
    import synth
    rng = np.random.default_rng(seed)
    dirs = oracle.healpix(NSIDE)
    nth = os.cpu_count() or 1

    def centres(idx):
        cl = synth.Cloud(keys_h[idx], lev_h[idx], np.zeros((len(idx), 1)), (1 << 21,) * 3)
        return synth.leaf_centres(cl)

    def run(n):
        idx = np.sort(rng.choice(n_leaves, size=n, replace=False))
        src = centres(idx)
        t0 = time.perf_counter()
        cols, _, nseg = oracle.trace(keys_h, lev_h, dens_h64, src, dirs, nthreads=nth)
        dt = time.perf_counter() - t0
        return idx, cols, int(nseg.sum()), dt

    _, _, seg0, dt0 = run(256)
    rate = seg0 / max(dt0, 1e-6)
    n = int(min(max(256, 256 * seconds / max(dt0, 1e-3)), 400_000))
    idx, cols, seg, dt = run(n)
    return {"idx": idx, "cols": cols, "segments": seg, "seconds": dt, "threads": nth, "n_src": n,
            "rate_small": rate}


def cpu_model():
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith(("model name", "cpu part")):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    return "unknown"


# ------------------------------------------------------- other workloads

def timed(fn, stream, reps=1):
    import torch
    fn()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(reps):
        fn()
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / 1e3 / reps


def amr_leg(rt, dev, stream, check_sources=400, reps=3, base=128):
    """AMR workload: 128^3 base (sigma 1.5), field on 512^3, 2 levels above p90,
    4 FP32 species, 1M mass-weighted sources, Nside 2, F32-Kahan; plus an
    oracle spot check of a few hundred sources.  (base: another base size,
    for profiling a smaller cloud of the same recipe.)"""
    import torch
    from synth import torchgen
    keys, lev, dens, ntot, ext = torchgen.amr_cloud(base, 2, 90.0, 1.5, 2, device=dev)
    src = torchgen.mass_weighted_sources(keys, lev, ntot, 1_000_000, 102)
    tree = rt.Octree(keys, lev, extent=ext)
    out = torch.empty((src.shape[0], 48, 4), dtype=torch.float32, device=dev)
    tree.reset_stats()
    t = timed(lambda: rt.trace_columns(tree, src, 2, dens, "f32k", out=out), stream, reps=reps)
    st = tree.stats()
    assert st["status"] == 0, st
    segs = st["segments"] / (reps + 1)
    res = {"workload": "%d^3 base AMR (2 levels above p90, %d leaves), 4 FP32 species, 1M mass-weighted "
                       "sources, Nside 2, F32-Kahan" % (base, keys.numel()),
           "value": segs / t, "unit": "ray-segments/s", "ms_per_step": t * 1e3,
           "segments_per_step": int(segs), "exit_fallbacks_per_step": st["exit_fallbacks"] / (reps + 1),
           "lookup_fallbacks_per_step": st["lookup_fallbacks"] / (reps + 1)}
    import oracle
    idx = torch.arange(0, src.shape[0], src.shape[0] // check_sources, device=dev)[:check_sources]
    want, _, _ = oracle.trace(keys.cpu().numpy().view(np.uint64), lev.cpu().numpy(),
                              dens.cpu().numpy().astype(np.float64), src[idx].cpu().numpy(),
                              oracle.healpix(2), extent=ext)
    got = out[idx].double().cpu().numpy()
    err = np.abs(got - want) / np.maximum(np.abs(want), 1e-300)
    res["parity_sample"] = {"n_src": int(idx.numel()), "max_rel": float(err.max())}
    # its bound: instruction issue, warp instructions per segment from the
    # committed capture of the same kernel on the 64^3-base cloud of this recipe
    prof = kernel_profile("trace_f32k_amr64")
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    peak = sms * 4 * 2070e6
    res["roofline"] = {"bound": "issue", "unit": "warp-instructions/s", "peak": peak,
                       "peak_kind": f"derived: {sms} SMs x 4 schedulers x 2070 MHz",
                       "warp_inst_per_segment": prof["warp_inst_per_segment"] if prof else None,
                       "achieved": segs / t * prof["warp_inst_per_segment"] if prof else None,
                       "frac": segs / t * prof["warp_inst_per_segment"] / peak if prof else None,
                       "ncu": {"issue_active_pct": prof["issue_active_pct"], "lts_hit_pct": prof["lts_hit_pct"],
                               "warp_exec_efficiency": prof["warp_exec_efficiency"]} if prof else None,
                       "profile": "profiles/trace_f32k_amr64.md"}
    # Alg. 1's chunked contribution grid: 8 Morton-range chunks, densities
    # streamed from page-locked host memory, rays carried between chunks
    d_host = dens.cpu().pin_memory()
    tree.reset_stats()
    tc = timed(lambda: rt.trace_columns_chunked(tree, src, 2, d_host, 8, "f32k", out=out), stream, reps=1)
    stc = tree.stats()
    assert stc["status"] == 0, stc
    res["chunked8_host"] = {"value": stc["segments"] / 2 / tc, "unit": "ray-segments/s", "ms_per_step": tc * 1e3,
                            "what": "8 chunks, densities streamed from page-locked host memory"}
    tree.close()
    return res


def batched_leg(rt, dev, stream, cache, reps=3):
    """64 independent clouds (base in {16,24,32,48,64,96}^3, 0-3 levels above
    p80, 2 FP32 species, leaf-centre sources, Nside 1 or 2) in one launch,
    launch shape from the autotuner."""
    from synth import torchgen
    clouds = []
    for k, l, d, ext, src, nside in torchgen.batched_clouds(dev):
        clouds.append((rt.Octree(k, l, extent=ext), src, nside, d))
    batch = rt.Batch(clouds, "f32k")
    best, rate = batch.autotune(cache)
    batch.reset_stats()
    t = timed(lambda: batch.launch(), stream, reps=reps)
    st = batch.stats()
    assert st["status"] == 0, st
    segs = st["segments"] / (reps + 1)
    res = {"workload": "64 clouds of uneven size and depth, %d rays, one persistent launch (CUDA graph)"
                       % (st["rays"] // (reps + 1)),
           "value": segs / t, "unit": "ray-segments/s", "ms_per_step": t * 1e3,
           "autotuned": {"threads": best[0], "blocks_per_sm": best[1], "groups_per_pop": best[2]}}
    batch.close()
    rt.set_launch(0, 0, 0)
    for c in clouds:
        c[0].close()
    return res


def adjoint_leg(rt, dev, stream, reps=3):
    """Differentiable workload: 64^3 base refined once above p85, one species,
    leaf-centre sources, Nside 2: forward (F32-Kahan) and adjoint times."""
    import torch
    from synth import torchgen
    k, l, d, n, ext = torchgen.amr_cloud(64, 1, 85.0, 1.5, 4, fracs=(1.0,), device=dev)
    tree = rt.Octree(k, l, extent=ext)
    src = torchgen.leaf_centres(k, l)
    out = torch.empty((src.shape[0], 48, 1), dtype=torch.float32, device=dev)
    tf = timed(lambda: rt.trace_columns(tree, src, 2, d, "f32k", out=out), stream, reps=reps)
    g = torch.rand_like(out)
    grad = torch.zeros((k.numel(), 1), dtype=torch.float64, device=dev)
    ta = timed(lambda: rt.trace_columns_adjoint(tree, src, 2, g, "f32k", grad_dens=grad), stream, reps=reps)
    # recorded paths: the record's cost, and an adjoint replayed from it
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    paths = rt.Paths(tree, src, 2, "f32k")
    torch.cuda.synchronize()
    t_rec = time.perf_counter() - t0
    t_rep = timed(lambda: paths.adjoint(g, grad_dens=grad), stream, reps=reps)
    t_ord = timed(lambda: paths.adjoint(g, grad_dens=grad, ordered=True), stream, reps=reps)
    info = paths.info()
    paths.close()
    tree.close()
    saved = ta - t_rep
    return {"workload": "64^3 base AMR, 1 level above p85 (%d leaves), 1 species, leaf-centre sources, Nside 2"
                        % k.numel(), "forward_ms": tf * 1e3, "adjoint_ms": ta * 1e3,
            "adjoint_over_forward": ta / tf,
            "paths": {"record_ms": t_rec * 1e3, "replayed_adjoint_ms": t_rep * 1e3,
                      "ordered_adjoint_ms": t_ord * 1e3, "record_bytes": info["bytes"],
                      "adjoints_to_repay_the_record": (t_rec / saved) if saved > 0 else None}}


def adjoint_uniform_leg(rt, dev, stream, level, reps=3):
    """The paper-scale adjoint alone: 2^level cubed uniform cloud (sigma 2, 4
    FP32 species), every leaf centre a source, Nside 1: the F32-Kahan forward
    and the adjoint (the leaf gather) seeded with the forward's columns."""
    import torch
    from synth import torchgen
    keys, lev, dens, _ = torchgen.uniform_cloud(level, 2.0, 5, device=dev)
    n = keys.numel()
    src = torchgen.uniform_centres(level, torch.arange(n, device=dev))
    tree = rt.Octree(keys, lev)
    out = torch.empty((n, 12, 4), dtype=torch.float32, device=dev)
    tf = timed(lambda: rt.trace_columns(tree, src, 1, dens, "f32k", out=out), stream, reps=reps)
    grad = torch.zeros((n, 4), dtype=torch.float64, device=dev)
    tree.reset_stats()
    ta = timed(lambda: rt.trace_columns_adjoint(tree, src, 1, out, "f32k", grad_dens=grad), stream, reps=reps)
    st = tree.stats()
    tree.close()
    return {"workload": f"{1 << level}^3 uniform, 4 FP32 species, all leaf centres, Nside 1: forward and adjoint",
            "forward_ms": tf * 1e3, "adjoint_ms": ta * 1e3, "adjoint_over_forward": ta / tf,
            "form": "leaf gather" if st["gathered"] else "scatter",
            "contributions_per_s": st["segments"] / (reps + 1) / ta}


def search_leg(rt, dev, stream, reps=3):
    """Key searches (Sec. 2.2.1, the leaf found by a search of the sorted keys)
    on workloads whose lookups search mixed coarse cells: the 128^3 AMR cloud
    with its coarse table capped at levels 7, 6 and 5 (and uncapped, level 8,
    where no lookup searches), and a 128^3 base refined 5 levels (deepest leaf
    level 12, four levels below its table).  F32-Kahan forward, Nside 2, 1M
    mass-weighted sources each."""
    import torch
    from synth import torchgen
    out = {}
    for name, nref, caps in (("amr128", 2, (-1, 7, 6, 5)), ("deep128", 5, (-1,))):
        keys, lev, dens, ntot, ext = torchgen.amr_cloud(128, nref, 90.0, 1.5, 2 if nref == 2 else 7, device=dev)
        src = torchgen.mass_weighted_sources(keys, lev, ntot, 1_000_000, 102)
        o = torch.empty((src.shape[0], 48, 4), dtype=torch.float32, device=dev)
        rows = []
        for cap in caps:
            rt.set_table_cap(cap)
            tree = rt.Octree(keys, lev, extent=ext)
            rt.set_table_cap(-1)
            row = {"table_cap": cap, "leaves": int(keys.numel()), "max_level": tree.max_level}
            tree.reset_stats()
            t = timed(lambda: rt.trace_columns(tree, src, 2, dens, "f32k", out=o), stream, reps=reps)
            st = tree.stats()
            assert st["status"] == 0, st
            row["value"] = st["segments"] / (reps + 1) / t
            rows.append(row)
            tree.close()
        out[name] = rows
        del keys, lev, dens, ntot, src, o
        torch.cuda.empty_cache()
    return {"workload": "leaf lookups with key searches, per-thread binary search (ray-segments/s)",
            **out}


def dualgrid_leg(rt, dev, stream, level=8, reps=1):
    """The paper's dual grid: a uniform source grid (2^level cells per axis,
    lognormal sigma 2, 4 species); the contribution grid is built from it on
    the GPU (split while n_max >= 1 and (n_max - n_min) / n_max >= 1 %); rays
    leave every source-cell centre (Nside 1) through that AMR grid."""
    import torch
    from synth import torchgen
    keys_u, lev_u, dens_u, ntot = torchgen.uniform_cloud(level, 2.0, 6, device=dev)
    tb0 = torch.cuda.Event(enable_timing=True)
    tb1 = torch.cuda.Event(enable_timing=True)
    tb0.record(stream)
    keys, lev, dens = rt.build_amr(ntot, dens_u, 1.0, 0.01, level)
    tb1.record(stream)
    torch.cuda.synchronize()
    tree = rt.Octree(keys, lev)
    src = torchgen.uniform_centres(level, torch.arange(keys_u.numel(), device=dev))
    out = torch.empty((src.shape[0], 12, 4), dtype=torch.float32, device=dev)
    tree.reset_stats()
    t = timed(lambda: rt.trace_columns(tree, src, 1, dens, "f32k", out=out), stream, reps=reps)
    st = tree.stats()
    assert st["status"] == 0, st
    segs = st["segments"] / (reps + 1)
    res = {"workload": "dual grid: %d^3 source cells, contribution grid of %d leaves built from them "
                       "(n_PDR 1, 1%% variation), Nside 1" % (1 << level, keys.numel()),
           "value": segs / t, "unit": "ray-segments/s", "ms_per_step": t * 1e3, "segments_per_step": int(segs),
           "build_amr_ms": tb0.elapsed_time(tb1)}
    tree.close()
    return res


# ------------------------------------------------ angular convergence (Sec. 3)

def ang2pix_ring(nside: int, v: np.ndarray) -> np.ndarray:
    """HEALPix RING index of the pixel containing each unit vector v [m][3]
    (Gorski et al. 2005 geometry).  In the equatorial belt (|z| <= 2/3) the
    pixel edges are the lines N(1/2 + phi/(pi/2)) -+ (3N/4) z = integer, so two
    floor indices (one per edge family) give the ring and the place in it; in
    a polar cap the edges are tp * N sqrt(3 (1 - |z|)) = integer and
    (1 - tp) * N sqrt(3 (1 - |z|)) = integer, tp the position inside the
    quadrant."""
    v = np.asarray(v, dtype=np.float64)
    z = v[:, 2] / np.linalg.norm(v, axis=1)
    phi = np.mod(np.arctan2(v[:, 1], v[:, 0]), 2.0 * np.pi)
    tt = phi / (0.5 * np.pi)                       # quadrant coordinate in [0, 4)
    n = nside
    npix = 12 * n * n
    out = np.empty(z.shape[0], dtype=np.int64)
    eq = np.abs(z) <= 2.0 / 3.0
    # equatorial belt
    a = n * (0.5 + tt[eq])
    b = 0.75 * n * z[eq]
    jp = np.floor(a - b).astype(np.int64)          # index of the ascending edge below
    jm = np.floor(a + b).astype(np.int64)          # index of the descending edge below
    ring = n + 1 + jp - jm                         # 1 .. 2n+1, counted from z = 2/3
    shift = 1 - (ring & 1)
    k = np.mod((jp + jm - n + shift + 1) // 2, 4 * n)   # place in the ring, 0-based
    out[eq] = 2 * n * (n - 1) + (ring - 1) * 4 * n + k
    # polar caps
    pc = ~eq
    za = np.abs(z[pc])
    tp = tt[pc] - np.floor(tt[pc])
    r = n * np.sqrt(3.0 * (1.0 - za))
    jp = np.floor(tp * r).astype(np.int64)
    jm = np.floor((1.0 - tp) * r).astype(np.int64)
    ring = jp + jm + 1                             # ring counted from the nearer pole
    k = np.mod(np.floor(tt[pc] * ring).astype(np.int64), 4 * ring)
    north = z[pc] > 0
    out[np.flatnonzero(pc)[north]] = (2 * ring * (ring - 1) + k)[north]
    out[np.flatnonzero(pc)[~north]] = (npix - 2 * ring * (ring + 1) + k)[~north]
    return out


def angular_leg(rt, dev, stream, level=7, nsides=(1, 2, 4, 8), nside_ref=64, reps=3):
    """The paper's angular-convergence test on a synthetic 128^3 cloud (one
    species, total hydrogen, lognormal sigma 2, 125 pc box):
    - sky maps of N_H from the leaf centre nearest the domain centre at Nside
      1..8 against Nside 64 (49152 rays): e_NH,q = |N_q - <N^ref>_q| / <N^ref>_q,
      <N^ref>_q the mean of the Nside-64 columns whose directions fall in pixel q;
    - A_V,eff of every cell at Nside 1, 2, 4 against Nside 64, computed inside
      the trace (the fused epilogue), e_AV = |A_V - A_V^ref| / A_V^ref;
    - the many-rays-per-source shape: 1 and 16 sources at Nside 64."""
    import torch
    from synth import torchgen
    keys, lev, dens, ntot = torchgen.uniform_cloud(level, 2.0, 8, fracs=(1.0,), device=dev)
    tree = rt.Octree(keys, lev)
    n_cells = keys.numel()
    box_cm = 125 * 3.0857e18
    a_av = 6.29e-22 * box_cm
    half = 1 << (level - 1)
    c = torch.tensor([[half + 0.5, half + 0.5, half + 0.5]], dtype=torch.float64, device=dev) / (1 << level)
    res = {"workload": "%d^3 uniform lognormal cloud (sigma 2), total H, 125 pc box; sky maps from the cell centre "
                       "nearest the domain centre and A_V,eff of all %d cells, Nside %s against Nside %d"
                       % (1 << level, n_cells, "/".join(str(x) for x in nsides), nside_ref, )}
    # sky maps
    ref = rt.trace_columns(tree, c, nside_ref, dens, "f32k")[0, :, 0].double().cpu().numpy()
    dirs_ref = rt.healpix_dirs(nside_ref)
    maps = {}
    for ns in nsides:
        col = rt.trace_columns(tree, c, ns, dens, "f32k")[0, :, 0].double().cpu().numpy()
        parent = ang2pix_ring(ns, dirs_ref)
        mean_ref = np.bincount(parent, weights=ref, minlength=12 * ns * ns) / np.bincount(parent, minlength=12 * ns * ns)
        e = np.abs(col - mean_ref) / mean_ref
        maps[str(ns)] = {"rays": 12 * ns * ns, "e_NH_mean": float(e.mean()), "e_NH_max": float(e.max())}
    res["sky_map_e_NH"] = maps
    # A_V,eff of every cell
    src = torchgen.uniform_centres(level, torch.arange(n_cells, device=dev))
    tree.reset_stats()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    av_ref = rt.trace_epilogue(tree, src, nside_ref, dens, "av_eff", [1.0], a_av, 3.02)
    e1.record(stream)
    torch.cuda.synchronize()
    st = tree.stats()
    assert st["status"] == 0, st
    t_ref = e0.elapsed_time(e1) / 1e3
    res["av_eff_reference"] = {"nside": nside_ref, "rays": int(st["rays"]), "segments": int(st["segments"]),
                               "seconds": t_ref, "value": st["segments"] / t_ref, "unit": "ray-segments/s",
                               "mean_av_eff": float(av_ref.mean().item())}
    dens_cells = ntot.double()
    dense = dens_cells >= torch.quantile(dens_cells.float(), 0.9).double()
    errs = {}
    for ns in nsides[:3]:
        av = rt.trace_epilogue(tree, src, ns, dens, "av_eff", [1.0], a_av, 3.02)
        e = (av - av_ref).abs() / av_ref
        errs[str(ns)] = {"e_AV_mean": float(e.mean().item()), "e_AV_max": float(e.max().item()),
                         "e_AV_mean_densest_10pct": float(e[dense].mean().item())}
    res["av_eff_e_AV"] = errs
    # many rays per source: 1 and 16 sources near the centre at Nside 64
    rates = {}
    for m in (1, 16):
        s_m = src[n_cells // 2: n_cells // 2 + m]
        out = torch.empty((m, 12 * nside_ref ** 2, 1), dtype=torch.float32, device=dev)
        tree.reset_stats()
        t = timed(lambda: rt.trace_columns(tree, s_m, nside_ref, dens, "f32k", out=out), stream, reps=reps)
        segs = tree.stats()["segments"] / (reps + 1)
        rates[str(m)] = {"rays": m * 12 * nside_ref ** 2, "ms_per_trace": t * 1e3, "value": segs / t,
                         "unit": "ray-segments/s"}
    res["few_sources_nside64"] = rates
    tree.close()
    return res


# -------------------------------------------------------------- reference
# -------------------------------------------------------------- reference

def run_reference(a, rank, world):
    """The reference arm: the plain FP64 oracle on the host cores, on bounded
    samples of the same workload, same metric and unit."""
    if rank != 0:
        return 0
    import torch
    from synth import torchgen
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    keys, lev, dens, _ = torchgen.uniform_cloud(a.level, 2.0, 5, device=dev)
    keys_h = keys.cpu().numpy().view(np.uint64)
    lev_h = lev.cpu().numpy()
    dens_h = dens.cpu().numpy().astype(np.float64)
    del keys, lev, dens
    n = keys_h.shape[0]
    per_step = max(4.0, 60.0 / max(a.steps + a.warmup, 1))
    for _ in range(a.warmup):
        oracle_sample(keys_h, lev_h, dens_h, n, per_step / 4, level=a.level)
    segs, secs, nsrc, th = 0, 0.0, 0, 1
    for k in range(a.steps):
        r = oracle_sample(keys_h, lev_h, dens_h, n, per_step, seed=100 + k, level=a.level)
        segs += r["segments"]
        secs += r["seconds"]
        nsrc += r["n_src"]
        th = r["threads"]
    v = segs / secs
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "ray-segments/s",
            "n_gpus": world, "steps": a.steps, "warmup": a.warmup, "ms_per_step": 1e3 * secs / a.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": f"{1 << a.level}^3 uniform lognormal cloud (sigma 2, 4 species), "
                                   "leaf-centre sources, HEALPix Nside 1", "sampled": True},
            "cpu_baseline": {"value": v, "unit": "ray-segments/s", "cores": th, "kind": "oracle",
                             "sample": f"{nsrc} random leaf-centre sources x 12 rays over {a.steps} steps "
                                       f"({segs} segments), CPU {cpu_model()}"},
            "e2e": {"value": v, "unit": "ray-segments/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------- ours

def main():
    a = parse()
    rank, world, local = dist_env()
    if world > 1 and a.impl == "ours":
        import torch.distributed as dist
        dist.init_process_group("nccl")
    if a.impl == "reference":
        return run_reference(a, rank, world)

    import torch

    import paper_2605_09882_gb300 as rt
    from synth import torchgen

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream()
    if a.workload != "uniform512":
        if a.workload == "amr128":
            r = amr_leg(rt, dev, stream, reps=a.steps, base=a.amr_base)
        elif a.workload == "batched64":
            r = batched_leg(rt, dev, stream, os.path.join(ROOT, "paper_2605_09882_gb300", "autotune_gb300.json"),
                            reps=a.steps)
        elif a.workload == "dualgrid256":
            r = dualgrid_leg(rt, dev, stream, reps=a.steps)
        elif a.workload == "angular128":
            r = angular_leg(rt, dev, stream, reps=a.steps)
        elif a.workload == "search":
            r = search_leg(rt, dev, stream, reps=a.steps)
        elif a.workload == "adjoint_uniform":
            r = adjoint_uniform_leg(rt, dev, stream, a.level, reps=a.steps)
        else:
            r = adjoint_leg(rt, dev, stream, reps=a.steps)
        if rank == 0:
            print(json.dumps({"workload_only": a.workload, "steps": a.steps, **r}), flush=True)
        return 0
    L = a.level
    n_side_cells = 1 << L

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    # ---- inputs, resident in HBM
    keys, lev, dens, _ = torchgen.uniform_cloud(L, 2.0, 5, device=dev)
    n = keys.numel()
    src = torchgen.uniform_centres(L, torch.arange(n, device=dev))
    tree = rt.Octree(keys, lev)
    nd = 12 * NSIDE * NSIDE
    out = torch.empty((n, nd, 4), dtype=torch.float32, device=dev)

    def fwd(mode="f32k", o=None):
        return rt.trace_columns(tree, src, NSIDE, dens, mode, out=o if o is not None else out)

    for _ in range(a.warmup):
        fwd()
    barrier()
    tree.reset_stats()
    clocks = Clocks(local)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * a.steps)]
    barrier()
    for k in range(a.steps):
        ev[2 * k].record(stream)
        fwd()
        ev[2 * k + 1].record(stream)
    barrier()
    clk = clocks.stop()
    launch_ms = [ev[2 * k].elapsed_time(ev[2 * k + 1]) for k in range(a.steps)]
    total_ms = ev[0].elapsed_time(ev[-1])
    st = tree.stats()
    assert st["status"] == 0, st
    seg_per_step = st["segments"] // a.steps
    if world > 1:
        import torch.distributed as dist
        t = torch.tensor([total_ms], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t)
    value = world * seg_per_step * a.steps / (total_ms / 1e3)
    avg_launch_s = float(np.mean(launch_ms)) / 1e3
    peak, peak_kind = peaks()
    roofline = trace_roofline(seg_per_step, avg_launch_s, clk, peak, peak_kind, dev)

    extras = {}
    cpu = None
    e2e = None
    if not a.no_extras:
        # ---- FP64 form (FP64 columns)
        out64 = torch.empty((n, nd, 4), dtype=torch.float64, device=dev)
        fwd("fp64", out64)
        barrier()
        tree.reset_stats()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fwd("fp64", out64)
        e1.record(stream)
        barrier()
        t64 = e0.elapsed_time(e1) / 1e3
        s64 = tree.stats()
        extras["fp64_form"] = {"value": s64["segments"] / t64, "unit": "ray-segments/s",
                               "ms_per_step": t64 * 1e3}
        # the GPU's FP64 rate, the bound of the FP64 form: a cuBLAS DGEMM
        # (8192^3, 2 N^3 flops, best of 3), measured here, not assumed
        A = torch.randn((8192, 8192), dtype=torch.float64, device=dev)
        B = torch.randn((8192, 8192), dtype=torch.float64, device=dev)
        torch.matmul(A, B)
        best = min(timed(lambda: torch.matmul(A, B), stream) for _ in range(3))
        dgemm = 2 * 8192 ** 3 / best
        extras["fp64_peak"] = {"dgemm_tflops": dgemm / 1e12,
                               "what": "cuBLAS FP64 GEMM 8192^3 on this GPU (2 N^3 flops, best of 3)"}
        # its FP64 operations per segment at 4 species: the column update (4 DMUL
        # + 4 DADD; the lengths come from the step tables)
        extras["fp64_form"]["fp64_ops_per_segment"] = 8
        extras["fp64_form"]["fp64_ops_per_s"] = 8 * s64["segments"] / t64
        extras["fp64_form"]["frac_of_dgemm_fma_rate"] = 8 * s64["segments"] / t64 / (dgemm / 2)
        del A, B
        # agreement of the two forms on the full output
        mx = torch.zeros(4, dtype=torch.float64, device=dev)
        sm = torch.zeros(4, dtype=torch.float64, device=dev)
        for c0 in range(0, n, 1 << 22):
            rel = (out[c0:c0 + (1 << 22)].double() - out64[c0:c0 + (1 << 22)]).abs_()
            rel /= out64[c0:c0 + (1 << 22)].abs().clamp_min(1e-300)
            mx = torch.maximum(mx, rel.amax(dim=(0, 1)))
            sm += rel.sum(dim=(0, 1))
        extras["f32k_vs_fp64"] = {"max_rel_per_species": [float(x) for x in mx],
                                  "mean_rel_per_species": [float(x) / (n * nd) for x in sm]}
        del rel, out64
        torch.cuda.empty_cache()
        # ---- adjoint (F32-Kahan walk, FP64 gradient), seed = the forward output:
        # the default (leaf gather, deterministic) and the atomic scatter
        grad = torch.zeros((n, 4), dtype=torch.float64, device=dev)
        rt.trace_columns_adjoint(tree, src, NSIDE, out, "f32k", grad_dens=grad)
        barrier()
        tree.reset_stats()
        e0.record(stream)
        rt.trace_columns_adjoint(tree, src, NSIDE, out, "f32k", grad_dens=grad)
        e1.record(stream)
        barrier()
        tadj = e0.elapsed_time(e1) / 1e3
        sadj = tree.stats()
        grad.zero_()
        rt.trace_columns_adjoint(tree, src, NSIDE, out, "f32k", grad_dens=grad)
        grad2 = torch.zeros_like(grad)
        rt.trace_columns_adjoint(tree, src, NSIDE, out, "f32k", grad_dens=grad2)
        same = bool(torch.equal(grad, grad2))
        del grad2
        grad_sc = torch.zeros_like(grad)
        barrier()
        e0.record(stream)
        rt.trace_columns_adjoint(tree, src, NSIDE, out, "f32k", grad_dens=grad_sc, path_policy=1)
        e1.record(stream)
        barrier()
        tsc = e0.elapsed_time(e1) / 1e3
        dmax = float(((grad - grad_sc).abs() / grad_sc.abs().clamp_min(1e-300)).max())
        extras["adjoint"] = {"ms_per_step": tadj * 1e3, "adjoint_over_forward": tadj / avg_launch_s,
                             "form": "leaf gather" if sadj["gathered"] else "scatter",
                             "segments": int(sadj["segments"]), "bitwise_repeatable": same,
                             "scatter_ms": tsc * 1e3, "scatter_over_forward": tsc / avg_launch_s,
                             "gather_vs_scatter_max_rel": dmax}
        del grad, grad_sc
        torch.cuda.empty_cache()
        # ---- fused A_V,eff epilogue: N_H = n(H) + 2 n(H2), a = A_V0 x 125 pc
        AV0_CM2, BOX_CM = 6.29e-22, 125 * 3.0857e18
        av = torch.empty(n, dtype=torch.float64, device=dev)
        tree.reset_stats()
        tav = timed(lambda: rt.trace_epilogue(tree, src, NSIDE, dens, "av_eff", [1.0, 2.0], AV0_CM2 * BOX_CM,
                                              gamma=3.02, out=av), stream)
        sav = tree.stats()
        extras["av_eff_epilogue"] = {"value": sav["segments"] / 2 / tav, "unit": "ray-segments/s",
                                     "ms_per_step": tav * 1e3, "output_bytes": n * 8,
                                     "what": "A_V,eff per source (N_H = n_H + 2 n_H2, gamma 3.02, 125 pc box) "
                                             "computed inside the trace; no column write"}
        # ---- octree build (validation + coarse table), one-time per tree
        tb = timed(lambda: rt.Octree(keys, lev).close(), stream)
        extras["build_octree_ms"] = tb * 1e3
        # ---- the other workloads
        extras["amr128"] = amr_leg(rt, dev, stream)
        extras["adjoint_amr64"] = adjoint_leg(rt, dev, stream)
        extras["batched64"] = batched_leg(rt, dev, stream,
                                          os.path.join(ROOT, "paper_2605_09882_gb300", "autotune_gb300.json"))
        torch.cuda.empty_cache()
        # ---- CPU oracle on a sample (rank 0, N = 1) + parity of those outputs
        keys_h = keys.cpu().numpy().view(np.uint64)
        lev_h = lev.cpu().numpy()
        if rank == 0 and world == 1:
            dens_h64 = dens.cpu().numpy().astype(np.float64)
            r = oracle_sample(keys_h, lev_h, dens_h64, n, a.cpu_seconds)
            got = out[torch.from_numpy(r["idx"]).to(dev)].double().cpu().numpy()
            err = np.abs(got - r["cols"]) / np.maximum(np.abs(r["cols"]), 1e-300)
            cpu = {"value": r["segments"] / r["seconds"], "unit": "ray-segments/s", "cores": r["threads"],
                   "kind": "oracle",
                   "sample": f"{r['n_src']} random leaf-centre sources x 12 rays ({r['segments']} segments), "
                             f"CPU {cpu_model()}"}
            from oracle import epilogue as oep
            want_av = oep.av_eff(r["cols"], [1.0, 2.0, 0.0, 0.0], AV0_CM2 * BOX_CM, 3.02)
            got_av = av[torch.from_numpy(r["idx"]).to(dev)].cpu().numpy()
            extras["av_eff_epilogue"]["parity_max_rel"] = float(np.max(np.abs(got_av - want_av) / np.abs(want_av)))
            extras["parity_sample"] = {"n_src": r["n_src"], "max_rel": float(err.max()),
                                       "max_rel_per_species": [float(x) for x in err.max(axis=(0, 1))],
                                       "mean_rel_per_species": [float(x) for x in err.mean(axis=(0, 1))]}
            del dens_h64
        # ---- end to end through the public API with host buffers
        host = [torch.from_numpy(keys_h.view(np.int64)), torch.from_numpy(lev_h), dens.cpu(), src.cpu(),
                torch.empty((n, nd, 4), dtype=torch.float32)]
        try:  # page-locked if the host lets this rank pin ~32 GB, else pageable (slower copies)
            host = [t.pin_memory() for t in host]
            kind = "page-locked"
        except RuntimeError:
            kind = "pageable"
        keys_p, lev_p, dens_p, src_p, out_p = host
        del tree, host
        h2d = sum(t.numel() * t.element_size() for t in (keys_p, lev_p, dens_p, src_p))
        d2h = out_p.numel() * out_p.element_size()
        e2e_steps = 2
        # one untimed call sizes the call's persistent device buffers
        rt.trace_columns_host(keys_p, lev_p, src_p, NSIDE, dens_p, "f32k", out=out_p, chunk=E2E_CHUNK)
        barrier()
        t0 = time.perf_counter()
        e0.record(stream)
        for _ in range(e2e_steps):
            # one C-ABI call: host buffers in, octree indexed, columns back,
            # copies pipelined with the traces in source chunks
            _, st_e2e = rt.trace_columns_host(keys_p, lev_p, src_p, NSIDE, dens_p, "f32k", out=out_p,
                                              chunk=E2E_CHUNK)
            assert st_e2e["status"] == 0 and st_e2e["segments"] == seg_per_step, st_e2e
        e1.record(stream)
        barrier()
        wall = time.perf_counter() - t0
        e2e = {"value": world * seg_per_step * e2e_steps / wall, "unit": "ray-segments/s",
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
               "ms_per_step": wall * 1e3 / e2e_steps,
               "call": f"rt_trace_columns_host, {kind} host buffers, {E2E_CHUNK} sources per chunk"}

    line = {
        "metric": METRIC,
        "value": value,
        "unit": "ray-segments/s",
        "n_gpus": world,
        "steps": a.steps,
        "warmup": a.warmup,
        "ms_per_step": total_ms / a.steps,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": f"{n_side_cells}^3 uniform lognormal cloud (P(k)~k^-4, sigma 2), 4 FP32 species, "
                               f"all {n} leaf-centre sources, HEALPix Nside 1 ({n * nd} rays), F32-Kahan columns",
                   "segments_per_step": seg_per_step, "l2": "inputs and output larger than L2 (no flush)",
                   "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
        "roofline": roofline,
        "cpu_baseline": cpu,
        "e2e": e2e,
        "clocks": clk,
        # per step: k_beam_ref, k_beam_setup, k_beam_dens, k_beam and k_trace (for left-out sources: none here)
        "gpu_launches": 5 * a.steps,
    }
    line.update(extras)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
