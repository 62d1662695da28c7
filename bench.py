#!/usr/bin/env python3
"""Throughput of recursive density-matrix purification on one GB300.

One step purifies the dense n = 4096 sweep (F = Q diag(lambda) Q^T, spectrum
[-1, 1], nocc in {n/2, n/4} x gap in {1e-1, 1e-2, 1e-3, 1e-4}: eight
matrices) with both scale-and-fold schemes (Algorithm 2, then Algorithm 1),
i.e. 16 purifications per step, inputs resident in HBM.  Prints one JSON line.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--precision mixed|fp64]
    python bench.py --impl reference     # the CPU oracle on the same metric

With N > 1 (torchrun) every rank purifies its own eight matrices (weak
scaling, no collective on the data path); the time is the max over ranks.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("purified n=4096 matrices/sec + tensor-pipe % at max-err<=1e-6 vs plain FP64; "
          "serve p50/p99")
GAPS = (1e-1, 1e-2, 1e-3, 1e-4)
SCHEMES = ("TC_SF", "FIXED_MU_SF")
SMS = 152                        # GB300 streaming multiprocessors
TENSOR_FLOP_PER_CLK_SM = 8192    # dense bf16 tcgen05 rate per SM and clock (nominal)
FP64_FLOP_PER_CLK_SM = 4         # two float64 FMAs per SM and clock (nominal)
# The tensor pipe's active share of one queue launch of the digit-plane
# product (ncu sm__pipe_tensor_cycles_active of digit_gemm_kernel<32, 5, 2>:
# one TC_SF run at n = 4096, 14 products in one launch).
TENSOR_PIPE_PCT_NCU = 75.3
TENSOR_PIPE_SOURCE = "profiles/digit_gemm_queue_s5_n4096.md (ncu, one queue launch, n=4096, S=5, 14 products)"
# DRAM bytes (read + write) of that launch, from the same ncu capture.
TRAFFIC_DIGIT_GEMM = 17.603e9
TRAFFIC_PRODUCTS = 14
TRAFFIC_SOURCE = ("ncu dram__bytes_read+write of digit_gemm_kernel<32,5,2>, n=4096, one queue launch of 14 "
                  "products (14.272 GB read + 3.331 GB written; 1.257 GB per product)")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    ap.add_argument("--precision", choices=("mixed", "fp64"), default="mixed")
    ap.add_argument("--n", type=int, default=4096)
    ap.add_argument("--tol", type=float, default=1e-9)
    ap.add_argument("--matrices", type=int, default=8,
                    help="use the first K matrices of the sweep (profiling / small runs)")
    ap.add_argument("--schemes", default=",".join(SCHEMES))
    ap.add_argument("--no-fp64-check", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--batch-size", type=int, default=256)
    ap.add_argument("--serve-advance", type=int, default=4,
                    help="products per request per serving call (0: one per round, grouped launches)")
    ap.add_argument("--serve-rates", default="10,30,100,300,1000", help="comma list; empty to skip serving")
    ap.add_argument("--serve-requests", type=int, default=500)
    ap.add_argument("--exact-bounds", action="store_true",
                    help="pass the exact lmin/lmax instead of estimating them inside the step")
    ap.add_argument("--no-variants", action="store_true",
                    help="skip the exact-bounds and refinement variants")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--pipelines", type=int, default=2,
                    help="handles (own stream and host thread each) sharing a step's purifications")
    ap.add_argument("--e2e-pipelines", type=int, default=2,
                    help="the same for the end-to-end run (host copies to overlap as well)")
    ap.add_argument("--no-lattice", action="store_true", help="skip the L^3 block-sparse workload")
    ap.add_argument("--no-autotune", action="store_true",
                    help="launch products with the fixed shape rule instead of measured shapes")
    ap.add_argument("--bits-floor", type=int, default=0,
                    help="per-step digit rule: fewest bits of a step's operands (0: library default)")
    ap.add_argument("--bits-gap", type=int, default=0,
                    help="per-step digit rule: bits beyond log2(1/mapped gap) (0: library default)")
    ap.add_argument("--lattice-size", type=int, default=32, help="L of the L^3 lattice (multiple of 4)")
    ap.add_argument("--lattice-only", action="store_true",
                    help="run only the lattice workload and print its object (profiling)")
    return ap.parse_args()


def workload_specs(n):
    return [(nocc, gap) for nocc in (n // 2, n // 4) for gap in GAPS]


def rank_instance(rank, i):
    """Seed instance of matrix i on rank `rank`: every replica purifies its own
    matrices (distinct seeds), the same workload shape on every rank."""
    return 1000 * rank + i


def replica_rate(ms_local, units_per_rank, world, allreduce_max):
    """Whole-job throughput of independent replicas: all ranks processed
    units_per_rank units each, and the job took the slowest rank's time
    (allreduce_max maps a rank's value to the maximum over ranks)."""
    ms = allreduce_max(ms_local)
    return world * units_per_rank / (ms * 1e-3), ms


def make_inputs(n, rank, count=None):
    from paper_1101_0265_gb300 import inputs as I
    specs = workload_specs(n)[:count]
    return [I.dense_hamiltonian(n, nocc, gap, config=2, instance=rank_instance(rank, i))
            for i, (nocc, gap) in enumerate(specs)]


def make_device_inputs(n, rank, count, dev):
    """The same sweep built on the GPU (torch QR); F and the eigenvectors Q
    (for the closed-form density) stay on the device."""
    from paper_1101_0265_gb300 import inputs as I
    hs, Fs = [], []
    for i, (nocc, gap) in enumerate(workload_specs(n)[:count]):
        spec = I.InstanceSpec(n=n, nocc=nocc, gap=gap, scheme="TC_SF", instance=rank_instance(rank, i),
                              config=2)
        F, h = I.dense_hamiltonian_device(spec, dev, keep_q=True)
        hs.append(h)
        Fs.append(F)
    return hs, Fs


def run_batch(P, dev, stream, count=256, reps=3, tol=1e-9):
    """The batch workload: `count` dense Hamiltonians, n log-uniform in
    [64, 2048], gap log-uniform in [1e-3, 1e-1], nocc = round(U(0.3, 0.7) n),
    TC_SF.  The value is one CUDA-graph replay of the single queue launch in
    which every instance advances on its own; the same batch with one grouped
    launch per round is timed beside it."""
    import numpy as np
    import torch
    from paper_1101_0265_gb300 import inputs as I
    specs = I.batch_specs(count)
    B = P.Batch(device=dev.index, stream=stream.cuda_stream)
    ids, metas = [], []
    for sp in specs:
        F, h = I.dense_hamiltonian_device(sp, dev)
        ids.append(B.add(F, h.nocc, h.lmin, h.lmax, h.homo, h.lumo, scheme="TC_SF", tol=tol, mu=0.0))
        metas.append(h)
        del F
    torch.cuda.synchronize(dev)
    out = {}
    for rounds in (False, True):
        B.run(use_graph=True, rounds=rounds)        # capture + first replay (warm-up)
        times = []
        for _ in range(reps):
            B.run(use_graph=True, rounds=rounds)
            times.append(B.stats(ids[0])["seconds"])
        out[rounds] = statistics.median(times)
        if not rounds:
            D0 = [B.density(i) for i in ids[:4]]
        else:   # the two modes give the same densities, bit for bit
            same = all(np.array_equal(B.density(i), d) for i, d in zip(ids[:4], D0))
    t = out[False]
    st = [B.stats(i) for i in ids]
    B.close()
    tensor = sum(x["tensor_flops"] for x in st)
    return {"workload": f"{count} dense F, n log-uniform [64, 2048], gap log-uniform [1e-3, 1e-1], "
                        f"TC_SF tol {tol:g}, one CUDA-graph replay of one queue launch per batch",
            "value": count / t, "unit": "purifications/s", "ms_per_batch": 1e3 * t,
            "replays": reps, "tensor_tflops": tensor / t / 1e12,
            "multiplications": sum(x["multiplications"] for x in st),
            "max_trace_err": max(x["trace_err"] for x in st),
            "grouped_per_round": {"value": count / out[True], "ms_per_batch": 1e3 * out[True],
                                  "tensor_tflops": tensor / out[True] / 1e12,
                                  "same_densities": bool(same)}}


def run_serve(P, dev, stream, rate, count, budget_gb=64.0, tol=1e-9, advance=4):
    """Continuous batching under Poisson arrivals: requests (n log-uniform in
    [128, 8192], gap log-uniform in [1e-4, 1e-1], half FIXED_MU_SF, half
    TC_SF) are admitted while the HBM budget allows; every call advances all
    admitted requests by up to `advance` products in one queue launch (0: one
    product per round through grouped launches); finished ones are read out
    and freed.  Latency is arrival -> density available."""
    import torch
    from collections import deque
    from paper_1101_0265_gb300 import inputs as I
    specs = I.serve_specs(rate, count)
    reqs = [I.reflected_hamiltonian_device(sp, dev) for sp in specs]   # untimed, O(n^2) each
    torch.cuda.synchronize(dev)
    B = P.Batch(device=dev.index, stream=stream.cuda_stream)
    budget = budget_gb * 2 ** 30
    pending = deque(range(count))
    live, lat, rounds, peak_live = {}, [], 0, 0
    t0 = time.perf_counter()
    while pending or live:
        now = time.perf_counter() - t0
        while pending and specs[pending[0]].arrival <= now:
            k = pending[0]
            if live and B.bytes_in_use() + P.batch_footprint(specs[k].n) > budget:
                break
            F, h = reqs[k]
            live[B.add(F, h.nocc, h.lmin, h.lmax, h.homo, h.lumo, scheme=specs[k].scheme, tol=tol,
                       mu=0.0)] = k
            pending.popleft()
        if not live:
            time.sleep(max(0.0, specs[pending[0]].arrival - (time.perf_counter() - t0)))
            continue
        peak_live = max(peak_live, len(live))
        if advance > 0:
            B.advance(advance)
        else:
            B.step()
        rounds += 1
        t = time.perf_counter() - t0
        for i, k in list(live.items()):
            if B.done(i):
                lat.append(t - specs[k].arrival)
                B.release(i)
                del live[i]
    total = time.perf_counter() - t0
    B.close()
    lat.sort()
    pct = lambda q: 1e3 * lat[min(len(lat) - 1, int(q * len(lat)))]
    return {"rate_per_s": rate, "requests": count, "latencies": len(lat), "p50_ms": pct(0.50),
            "p99_ms": pct(0.99),
            "max_ms": 1e3 * lat[-1], "throughput_per_s": count / total, "rounds": rounds,
            "peak_concurrent": peak_live, "hbm_budget_gb": budget_gb,
            "engine": (f"queue launch per call, up to {advance} products per request" if advance > 0
                       else "one product per request per round, grouped launches")}


def run_lattice(P, dev, stream, L=32, tau=1e-6, tol=1e-9, budget=2e-5, wide_onsite=3.0,
                sweeps=((6.0, (16, 20, 24, 28, 32, 40, 48, 56)), (3.0, (16, 24, 32, 40)))):
    """The block-sparse workload: periodic L^3 cubic tight-binding lattice
    (onsite +-0.5 by sublattice + N(0, 0.05), hopping -1 + U(-0.1, 0.1)),
    n = L^3, nocc = n/2, mu = 0, loaded from COO, 32 x 32 blocks.

    - "C3": tau per step; trace-correcting scale-and-fold (TC_SF) against
      its monotonic baseline (TC_MONO), both block-sparse, and TC_SF dense.
    - "equal_budget": TC_SF against TC_MONO with the same total truncation
      budget (tau = budget / (m + 1)), at the C3 onsite splitting and at a
      wider one (+-wide_onsite), where the density stays sparse.
    - "n_sweep": TC_SF block-sparse at tau per step on L^3 lattices of
      growing L for each (onsite, sizes) of `sweeps`: time per step, the
      kept blocks per block row and the digit-plane pool bytes against n.
    One handle per mode, warmed once; device-event time of one run each."""
    import torch
    from paper_1101_0265_gb300 import inputs as I

    def case(lat, scheme, bs, **opt):
        pur = pool[bs]
        if bs:
            pur.set_options(trunc_tau=opt.get("trunc_tau", tau), trunc_budget=opt.get("trunc_budget", 0.0))
        g = lat.gap_bound
        pur.set_hamiltonian_coo(lat.n, lat.rows, lat.cols, lat.vals, nocc=lat.nocc, mu=0.0,
                                homo=-g, lumo=g)
        pur.run(scheme, tol, 300)
        st = pur.stats()
        r = {"seconds": st["seconds"], "iterations": st["iterations"],
             "tensor_tflops": st["tensor_flops"] / st["seconds"] / 1e12,
             "trace_err": abs(st["trace"] - lat.nocc), "idem_err_fro": st["idem_err_fro"]}
        if bs:
            h = pur.block_history()
            nb = lat.n // 32
            r["nnz_blocks"] = h
            r["final_fill"] = h[-1] / (nb * (nb + 1) / 2)
            r["plane_pool_mib"] = st["plane_pool_mib"]
        return r

    lat = I.lattice_hamiltonian(L)
    pool = {True: P.Purifier(device=dev.index, stream=stream.cuda_stream, precision="mixed",
                             block_sparse=True, trunc_tau=tau),
            False: P.Purifier(device=dev.index, stream=stream.cuda_stream, precision="mixed")}
    case(lat, "TC_SF", True)       # warm-up (allocations, kernel set-up)
    case(lat, "TC_SF", False)
    c3 = {"onsite": 0.5, "gap_bound": lat.gap_bound, "tau": tau,
          "TC_SF": case(lat, "TC_SF", True), "TC_MONO": case(lat, "TC_MONO", True),
          "TC_SF_dense": case(lat, "TC_SF", False)}
    c3["speedup_sf_vs_mono"] = c3["TC_MONO"]["seconds"] / c3["TC_SF"]["seconds"]
    c3["speedup_sparse_vs_dense"] = c3["TC_SF_dense"]["seconds"] / c3["TC_SF"]["seconds"]
    eq = []
    for onsite in (0.5, wide_onsite):
        lt = lat if onsite == 0.5 else I.lattice_hamiltonian(L, onsite=onsite)
        e = {"onsite": onsite, "gap_bound": lt.gap_bound, "budget": budget,
             "TC_SF": case(lt, "TC_SF", True, trunc_budget=budget),
             "TC_MONO": case(lt, "TC_MONO", True, trunc_budget=budget)}
        if onsite != 0.5:
            e["TC_SF_dense"] = case(lt, "TC_SF", False)
            e["speedup_sparse_vs_dense"] = e["TC_SF_dense"]["seconds"] / e["TC_SF"]["seconds"]
        e["speedup_sf_vs_mono"] = e["TC_MONO"]["seconds"] / e["TC_SF"]["seconds"]
        eq.append(e)
    # n-sweeps: the same construction at growing L with wider onsite
    # splittings (shorter decay length of D against the box), tau per step;
    # the dense handle is closed first (the largest lattice needs the room)
    pool[False].close()
    del pool[False]
    torch.cuda.empty_cache()
    sweep = []
    for onsite, sizes in sweeps:
        for Ls in sizes:
            lt = I.lattice_hamiltonian(Ls, onsite=onsite)
            r = case(lt, "TC_SF", True, trunc_tau=tau)
            nb = lt.n // 32
            kept = r["nnz_blocks"][-1]
            n_pad = (lt.n + 127) // 128 * 128
            sweep.append({"onsite": onsite, "L": Ls, "n": lt.n, "seconds": r["seconds"],
                          "iterations": r["iterations"],
                          "seconds_per_step": r["seconds"] / max(1, r["iterations"]),
                          "kept_blocks_per_block_row": 2 * kept / nb, "final_fill": r["final_fill"],
                          "max_fill": max(r["nnz_blocks"]) / (nb * (nb + 1) / 2),
                          "plane_pool_mib": r["plane_pool_mib"],
                          "dense_planes_mib": 2 * 6 * n_pad * n_pad * 2 / 2**20,
                          "dense_fd_mib": 2 * 8 * lt.n * lt.n / 2**20, "trace_err": r["trace_err"]})
    for pur in pool.values():
        pur.close()
    torch.cuda.empty_cache()
    return {"workload": f"{L}^3 periodic cubic tight-binding lattice, n={lat.n}, COO input, "
                        f"32x32 blocks, tol {tol:g}",
            "n": lat.n, "C3": c3, "equal_budget": eq,
            "n_sweep": {"tau": tau, "scheme": "TC_SF block-sparse", "runs": sweep,
                        "note": "plane_pool_mib: peak MiB of the block pools (the iterates' digit planes, "
                                "plane_pairs(s) x 4 KB per 32x32 block, and the last step's float64 density "
                                "blocks, 8 KB each); dense_planes_mib: two dense 6-plane buffers; dense_fd_mib: "
                                "a dense float64 F and D, which a CSR-loaded block-sparse handle does not hold"}}


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


class ClockSampler:
    """nvidia-smi samples during the timed region (started before, stopped after)."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device):
        self.device = device
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.device}", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return float("nan")
        sm = [num(r[1]) for r in rows]
        smax = max(num(r[2]) for r in rows)
        loaded = [r for r in rows if num(r[3]) > 300.0] or rows
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        reasons = sorted({names[i] for r in loaded for i in range(4) if r[5 + i] == "Active"})
        return {"sm_mhz": statistics.median(num(r[1]) for r in loaded), "sm_max_mhz": smax,
                "samples": len(rows), "samples_loaded": len(loaded),
                "power_w_max": max(num(r[3]) for r in rows), "reasons": reasons,
                "sm_mhz_min": min(sm)}


def cpu_baseline(hs, Fs, tol, estimate_bounds=True):
    """The oracle as it stands, on a bounded sample of the step: four
    purifications that cycle through both nocc values, four gaps and both
    schemes (bounds estimated as in the timed step: Gershgorin, then 16
    Lanczos steps)."""
    from oracle import purify_oracle as O
    picks = [(0, "TC_SF"), (6, "FIXED_MU_SF"), (5, "TC_SF"), (3, "FIXED_MU_SF")]
    picks = [(i % len(hs), sc) for i, sc in picks]
    t0 = time.perf_counter()
    for i, sc in picks:
        h, F = hs[i], Fs[i]
        lo, hi = O.lanczos_bounds(F, 16) if estimate_bounds else (h.lmin, h.lmax)
        O.purify(F, sc, min(lo, h.homo), max(hi, h.lumo), mu=0.0, homo=h.homo, lumo=h.lumo, tol=tol)
    dt = time.perf_counter() - t0
    desc = ", ".join(f"{sc} nocc={hs[i].nocc} gap={hs[i].meta['gap']:g}" for i, sc in picks)
    return {"value": len(picks) / dt, "unit": "matrices/s", "cores": _blas_threads(), "kind": "oracle",
            "sample": f"{len(picks)} of the step's 16 purifications at n={hs[0].n} ({desc}; tol {tol:g}, "
                      f"bounds by Gershgorin + 16 Lanczos steps), numpy float64, {dt:.1f} s"}


def _blas_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads") for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(n[0])
    except Exception:
        pass
    env = os.environ.get("OPENBLAS_NUM_THREADS") or os.environ.get("OMP_NUM_THREADS")
    return int(env) if env else os.cpu_count()


def main_config(n, count, schemes, tol, precision, world, exact_bounds=False):
    """The `config` of the dense workload (both arms report the same one)."""
    return {"workload": f"dense F=Q diag(lambda) Q^T n={n}, nocc in {{n/2,n/4}} x gap in "
                        f"{{1e-1,1e-2,1e-3,1e-4}} ({count} matrices) x schemes "
                        f"{', '.join(schemes)}; tol {tol:g}",
            "n": n, "matrices_per_step": count * len(schemes),
            "tol": tol, "parallelism": f"replicas x{world}",
            "bounds": ("lmin/lmax given exactly" if exact_bounds else
                       "lmin/lmax estimated per matrix inside the step (Gershgorin discs, 16 Lanczos "
                       "steps); homo/lumo given"),
            "l2": "inputs larger than L2 (each F is 134 MB, 8 distinct per step)"}


def run_reference(args, rank, world):
    """The reference arm: the CPU oracle (no GPU work), rank 0 only."""
    if rank != 0:
        return
    n = args.n
    schemes = tuple(args.schemes.split(","))
    count = min(args.steps + args.warmup, len(workload_specs(n)))
    hs = make_inputs(n, 0, count)
    from oracle import purify_oracle as O

    def one(i):
        h = hs[i % count]
        lo, hi = O.lanczos_bounds(h.F, 16)
        O.purify(h.F, schemes[i % len(schemes)], min(lo, h.homo), max(hi, h.lumo), mu=0.0, homo=h.homo,
                 lumo=h.lumo, tol=args.tol)
    for i in range(args.warmup):
        one(i)
    t0 = time.perf_counter()
    for i in range(args.steps):
        one(args.warmup + i)
    dt = time.perf_counter() - t0
    value = args.steps / dt
    cores = _blas_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "matrices/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": main_config(n, len(workload_specs(n)), schemes, args.tol, "f64", world),
        "cpu_baseline": {"value": value, "unit": "matrices/s", "cores": cores, "kind": "oracle",
                         "sample": f"a bounded sample of the step: one purification per step "
                                   f"(CPU oracle, numpy float64, bounds by Gershgorin + 16 Lanczos "
                                   f"steps), cycling the first {count} matrices of the sweep and the "
                                   f"schemes {', '.join(schemes)}"},
        "e2e": {"value": value, "unit": "matrices/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def accuracy_pass(P, pur, hs, Fd, Dc, schemes, tol, set_fn, dev, ref=None):
    """Every purification of the step once more, outside the timed region:
    per result the max |D - D_exact| against the closed form Q_occ Q_occ^T,
    |trace D - nocc|, ||D - D^2||_F (both from D itself), the library's own
    reductions, and, with `ref` (a float64 handle), the max |D - D_fp64| of
    the plain float64 recursion on the same schedule."""
    import torch
    n = hs[0].n
    D = torch.empty((n, n), dtype=torch.float64, device=dev)
    D2 = torch.empty((n, n), dtype=torch.float64, device=dev) if ref else None
    out, t64 = [], 0.0
    for i, h in enumerate(hs):
        set_fn(pur, h, Fd[i])
        if ref:
            set_fn(ref, h, Fd[i])
        for sc in schemes:
            if pur.run(sc, tol, 200) != P.OK:
                raise RuntimeError(f"{sc} did not converge")
            st = pur.stats()
            pur.density(D)
            r = {"nocc": h.nocc, "gap": h.meta["gap"], "scheme": sc, "iterations": st["iterations"],
                 "max_err_closed_form": float((D - Dc[i]).abs().max()),
                 "trace_err": abs(float(torch.trace(D)) - h.nocc),
                 "idem_err_fro": float(torch.linalg.matrix_norm(D - D @ D)),
                 "lib_trace_err": st["trace_err"], "lib_idem_err_fro": st["idem_err_fro"]}
            if ref:
                if ref.run(sc, tol, 200) != P.OK:
                    raise RuntimeError(f"float64 {sc} did not converge")
                t64 += ref.stats()["seconds"]
                ref.density(D2)
                r["max_err_vs_fp64"] = float((D - D2).abs().max())
            out.append(r)
    return out, t64


def summarize_accuracy(results, bound=1e-6):
    worst = lambda k: max(r[k] for r in results) if results and k in results[0] else None
    e_cf, e_64 = worst("max_err_closed_form"), worst("max_err_vs_fp64")
    ok = e_cf is not None and e_cf <= bound and e_64 is not None and e_64 <= bound
    return {"bound": bound, "pass": bool(ok), "max_err_closed_form": e_cf, "max_err_vs_fp64": e_64,
            "max_trace_err": worst("trace_err"), "max_idem_err_fro": worst("idem_err_fro")}


def fp64_roofline(acc, pk, pk_kind, sm_mhz):
    """The float64 path's products against the unit they ran on: digit products on the
    tensor cores when the runs issued tensor flops, else the float64 FMA pipe."""
    if acc["tensor_flops"] > 0.0:
        achieved = acc["tensor_flops"] / acc["prod_s"] / 1e12
        peak = pk["bf16_tflops_sustained"]
        return {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak, "traffic": None,
                "kernel": "float64 step: split, f64_digit_product_kernel (digit products on tcgen05), finish",
                "peak_kind": f"{pk_kind} bf16 sustained",
                "useful_tflops_in_products": acc["useful"] / acc["prod_s"] / 1e12}
    achieved = acc["useful"] / acc["prod_s"] / 1e12
    peak = SMS * FP64_FLOP_PER_CLK_SM * sm_mhz * 1e6 / 1e12
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
            "frac": achieved / peak, "traffic": None, "kernel": "step_f64_kernel",
            "peak_kind": f"float64 FMA pipe: {SMS} SMs x {FP64_FLOP_PER_CLK_SM // 2} DFMA per clock x 2 "
                         f"x the median SM clock under load ({sm_mhz:.0f} MHz)"}


def main():
    t_start = time.perf_counter()
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    import torch
    import paper_1101_0265_gb300 as P
    from paper_1101_0265_gb300 import build

    if rank == 0:
        build.build()
    dist = None
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        dist.barrier()
        if rank != 0:
            build.build()
    else:
        torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if args.lattice_only:
        stream = torch.cuda.current_stream(dev)
        print(json.dumps({"lattice": run_lattice(P, dev, stream, L=args.lattice_size)}), flush=True)
        return
    n = args.n
    schemes = tuple(args.schemes.split(","))
    hs, Fd = make_device_inputs(n, rank, args.matrices, dev)
    Fh = [F.cpu().pin_memory() for F in Fd]
    Dh = torch.empty((n, n), dtype=torch.float64).pin_memory()
    stream = torch.cuda.current_stream(dev)
    rule = {"bits_floor": args.bits_floor, "bits_gap": args.bits_gap, "autotune": not args.no_autotune}
    pur = P.Purifier(device=local, stream=stream.cuda_stream, precision=args.precision,
                     time_products=True, **rule)

    def set_h(p, h, F, exact=args.exact_bounds):
        # lmin / lmax NaN: estimated on the device (Gershgorin, then Lanczos)
        if exact:
            p.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        else:
            p.set_hamiltonian(F, nocc=h.nocc, mu=0.0, homo=h.homo, lumo=h.lumo)

    acc = {"launches": 0, "prod_s": 0.0, "prod_n": 0, "tensor_flops": 0.0, "useful": 0.0,
           "mults": 0, "digit_max": 0}

    def one_matrix(p, i, host=False, record=False, exact=args.exact_bounds, Dout=None):
        """Bounds and both schemes for matrix i: one set, one run per scheme."""
        h = hs[i]
        set_h(p, h, Fh[i] if host else Fd[i], exact)
        launches = p.stats()["kernel_launches"]
        for scheme in schemes:
            code = p.run(scheme, args.tol, 200)
            if code != P.OK:
                raise RuntimeError(f"{scheme} did not converge: {P.strerror(code)}")
            s_ = p.stats()
            launches += s_["kernel_launches"]
            if host:
                p.density(Dout)
            if record:
                acc["prod_s"] += s_["product_seconds"]
                acc["prod_n"] += s_["product_launches"]
                acc["tensor_flops"] += s_["tensor_flops"]
                acc["useful"] += s_["useful_flops"]
                acc["mults"] += s_["multiplications"]
                acc["digit_max"] = max(acc["digit_max"], s_["digit_max"])
        if record:
            acc["launches"] += launches
        return launches

    def step(host=False, record=False, exact=args.exact_bounds):
        for i in range(len(hs)):
            one_matrix(pur, i, host=host, record=record, exact=exact, Dout=Dh)

    def timed(k, host=False, record=False, clocks=False, exact=args.exact_bounds):
        if dist:
            dist.barrier()
        torch.cuda.synchronize(dev)
        sampler = ClockSampler(local) if clocks else None
        if sampler:
            sampler.start()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(k):
            step(host=host, record=record, exact=exact)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        ck = sampler.stop() if sampler else None
        if dist:
            dist.barrier()
        return e0.elapsed_time(e1), ck

    def max_over_ranks(ms):
        if not dist:
            return ms
        t = torch.tensor([ms], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        return float(t.item())

    # Pipelines: handles on their own streams and host threads share a step's
    # matrices (one purification's host work and copies overlap another's
    # products).
    npipe = max(1, args.pipelines)
    ne2e = max(1, args.e2e_pipelines)
    per_step = len(hs) * len(schemes)
    pipes = []
    nhandles = max(npipe, ne2e)
    for _ in range(nhandles if nhandles > 1 else 0):
        sp = torch.cuda.Stream(dev)
        pipes.append((sp, P.Purifier(device=local, stream=sp.cuda_stream, precision=args.precision, **rule),
                      torch.empty((n, n), dtype=torch.float64).pin_memory()))

    def pipe_run(p, k, host, errs, launches, use):
        _, pp, Dp = pipes[p]
        try:
            for _ in range(k):
                for i in range(p, len(hs), use):
                    launches[p] += one_matrix(pp, i, host=host, Dout=Dp)
        except Exception as e:  # reported after the join
            errs.append(e)

    def pipelined(k, host, use, clocks=False):
        import threading
        if dist:
            dist.barrier()
        torch.cuda.synchronize(dev)
        sampler = ClockSampler(local) if clocks else None
        if sampler:
            sampler.start()
        e0 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        errs, launches = [], [0] * use
        ths = [threading.Thread(target=pipe_run, args=(p, k, host, errs, launches, use)) for p in range(use)]
        for t in ths:
            t.start()
        for t in ths:
            t.join()
        if errs:
            raise errs[0]
        ends = []
        for sp, _, _ in pipes[:use]:
            e = torch.cuda.Event(enable_timing=True)
            e.record(sp)
            ends.append(e)
        torch.cuda.synchronize(dev)
        ck = sampler.stop() if sampler else None
        if dist:
            dist.barrier()
        return max(e0.elapsed_time(e) for e in ends), ck, sum(launches)

    for _ in range(args.warmup):
        step()
    # one handle in order: the roofline, per-product statistics and launches
    ms1_local, clocks = timed(args.steps, record=True, clocks=npipe == 1)
    value1, ms1 = replica_rate(ms1_local, per_step * args.steps, world, max_over_ranks)
    launches_timed = acc["launches"]
    if npipe > 1:
        for _ in range(max(1, args.warmup // 2)):
            pipelined(1, host=False, use=npipe)
        ms_local, clocks, launches_timed = pipelined(args.steps, host=False, use=npipe, clocks=True)
        value, ms = replica_rate(ms_local, per_step * args.steps, world, max_over_ranks)
    else:
        value, ms = value1, ms1
    # end to end: host F in, host D out, copies inside the timed region
    step(host=True)
    k_e2e = max(1, args.steps // 2)
    ms_e2e_local, _ = timed(k_e2e, host=True)
    value_e2e_serial, _ = replica_rate(ms_e2e_local, per_step * k_e2e, world, max_over_ranks)
    value_e2e = value_e2e_serial
    if ne2e > 1:
        pipelined(1, host=True, use=ne2e)
        ms_pipe_local, _, _ = pipelined(k_e2e, host=True, use=ne2e)
        value_e2e, _ = replica_rate(ms_pipe_local, per_step * k_e2e, world, max_over_ranks)
    for _, pp, _ in pipes:
        pp.close()

    pk, pk_kind = peaks()
    sm_mhz = (clocks or {}).get("sm_mhz") or pk.get("sm_max_mhz", 2070.0)
    if args.precision == "mixed":
        achieved = acc["tensor_flops"] / acc["prod_s"] / 1e12
        peak = pk["bf16_tflops_sustained"]
        at_clock = SMS * TENSOR_FLOP_PER_CLK_SM * sm_mhz * 1e6 / 1e12
        roof = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak, "traffic": TRAFFIC_DIGIT_GEMM,
                "traffic_products_per_launch": TRAFFIC_PRODUCTS,
                "kernel": "digit-plane tcgen05 product (queue launches: a run's products overlapping)",
                "peak_kind": f"{pk_kind} bf16 sustained",
                "traffic_source": TRAFFIC_SOURCE,
                "tensor_pipe_pct_ncu": TENSOR_PIPE_PCT_NCU, "tensor_pipe_source": TENSOR_PIPE_SOURCE,
                "per_clock": {"sm_mhz": sm_mhz, "peak_tflops_at_clock": at_clock,
                              "frac": achieved / at_clock,
                              "rate": f"{TENSOR_FLOP_PER_CLK_SM} dense bf16 flop per clock per SM "
                                      f"x {SMS} SMs (the nominal dense rate)"}}
    else:
        roof = fp64_roofline(acc, pk, pk_kind, sm_mhz)
    line = {
        "metric": METRIC, "value": value, "unit": "matrices/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16" if args.precision == "mixed" else "f64", "data": "synthetic",
        "config": main_config(n, len(hs), schemes, args.tol, args.precision, world, args.exact_bounds),
        "clocks": clocks,
        "e2e": {"value": value_e2e, "unit": "matrices/s",
                "h2d_bytes_per_step": len(hs) * n * n * 8,
                "d2h_bytes_per_step": per_step * n * n * 8,
                "pipelines": ne2e, "serial_value": value_e2e_serial,
                "note": "pinned host F in (once per matrix) and D out (once per purification) through "
                        "purify_set_hamiltonian / purify_get_density; `pipelines` handles, each on its own "
                        "stream and host thread, share the step's matrices"},
        "gpu_launches": launches_timed,
        "pipelines": npipe,
        "single_handle": {"value": value1, "ms_per_step": ms1 / args.steps,
                          "note": "one handle, purifications in order; the roofline, per-product "
                                  "statistics and digit counts come from this run"},
        "roofline": roof,
        "multiplications_per_step": acc["mults"] / args.steps,
        "useful_tflops": acc["useful"] / (ms1 * 1e-3) / 1e12,
    }
    if args.precision == "mixed":
        line["tensor_pipe_pct_of_step_est"] = 100.0 * acc["tensor_flops"] / (ms1 * 1e-3) / (
            SMS * TENSOR_FLOP_PER_CLK_SM * sm_mhz * 1e6)
        line["digit_max"] = acc["digit_max"]
        line["digit_rule"] = {"bits_floor": args.bits_floor or 30, "bits_gap": args.bits_gap or 26}
        shapes = {}
        for s_ in range(1, 7):
            t = P.tuned_shape(local, s_, n)
            if t is not None:
                shapes[str(s_)] = {"kc": t[0], "split_ways": t[1]}
        line["launch_shapes"] = shapes if shapes else "fixed rule"
    # accuracy of every result: closed form, trace, idempotency, float64 path
    Dc = []
    for i, h in enumerate(hs):
        occ = h.Q[:, torch.from_numpy(h.lam < 0.0).to(dev)]
        Dc.append(occ @ occ.T)
    ref = None
    if not args.no_fp64_check and args.precision == "mixed":
        ref = P.Purifier(device=local, stream=stream.cuda_stream, precision="fp64")
    wall = {"headline": time.perf_counter() - t_start}
    t_sec = time.perf_counter()
    results, t64 = accuracy_pass(P, pur, hs, Fd, Dc, schemes, args.tol, set_h, dev, ref=ref)
    wall["accuracy"] = time.perf_counter() - t_sec
    if ref:
        ref.close()
        line["fp64_path"] = {"value": per_step / t64, "unit": "matrices/s",
                             "note": "same schedules through the float64 path, same GPU"}
    elif args.precision == "fp64":
        for r in results:
            r["max_err_vs_fp64"] = 0.0
    accuracy = summarize_accuracy(results)
    line["accuracy"] = accuracy
    line["results"] = results
    line["max_err_vs_fp64"] = accuracy["max_err_vs_fp64"]
    if not accuracy["pass"]:
        # the metric is defined at max-err <= 1e-6: no throughput without it
        line["value_unchecked"] = line["value"]
        line["value"] = None
        line["e2e"]["value"] = None
    # the whole path with other bounds / refinement settings, one pass each
    t_sec = time.perf_counter()
    if world == 1 and args.precision == "mixed" and not args.no_variants:
        variants = {}
        k_var = max(1, args.steps // 4)

        def variant(name, exact, **opt):
            pur.set_options(**opt)
            step(exact=exact)                       # warm-up (allocations)
            ms_v, _ = timed(k_var, exact=exact)
            res, _ = accuracy_pass(P, pur, hs, Fd, Dc, schemes, args.tol,
                                   lambda p, h, F: set_h(p, h, F, exact), dev)
            pur.set_options(**{k: 0 for k in opt})
            a = summarize_accuracy([dict(r, max_err_vs_fp64=0.0) for r in res])
            variants[name] = {"value": per_step * k_var / (ms_v * 1e-3), "unit": "matrices/s",
                              "ms_per_step": ms_v / k_var, "max_err_closed_form": a["max_err_closed_form"],
                              "max_trace_err": a["max_trace_err"], "max_idem_err_fro": a["max_idem_err_fro"]}
        variant("exact_bounds", not args.exact_bounds)
        variant("refine_tc_6digits", args.exact_bounds, refine_squares=1)
        variant("refine_fp64", args.exact_bounds, refine_fp64=1)
        variants["note"] = ("one handle in order, the same 16 purifications: exact_bounds flips how "
                            "lmin/lmax are obtained; refine_tc_6digits appends one McWeeny step at 6 digits "
                            "on the tensor cores; refine_fp64 appends one float64 McWeeny step (two "
                            "products)")
        line["variants"] = variants
    wall["variants"] = time.perf_counter() - t_sec
    t_sec = time.perf_counter()
    if world == 1 and args.precision == "mixed" and not args.no_batch:
        line["batch"] = run_batch(P, dev, stream, count=args.batch_size)
    wall["batch"] = time.perf_counter() - t_sec
    t_sec = time.perf_counter()
    if world == 1 and args.precision == "mixed" and args.serve_rates:
        line["serve"] = [run_serve(P, dev, stream, float(r), args.serve_requests, advance=args.serve_advance)
                         for r in args.serve_rates.split(",")]
    wall["serve"] = time.perf_counter() - t_sec
    t_sec = time.perf_counter()
    if world == 1 and args.precision == "mixed" and not args.no_lattice:
        line["lattice"] = run_lattice(P, dev, stream, L=args.lattice_size)
    wall["lattice"] = time.perf_counter() - t_sec
    t_sec = time.perf_counter()
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(hs, [F.numpy() for F in Fh], args.tol,
                                            estimate_bounds=not args.exact_bounds)
    wall["cpu_baseline"] = time.perf_counter() - t_sec
    line["wall_seconds"] = {k: round(v, 1) for k, v in wall.items()}
    pur.close()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
