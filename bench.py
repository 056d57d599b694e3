#!/usr/bin/env python
"""Benchmark of the state-vector ADAPT-VQE hot path on one GB300 (or N
independent replicas under torchrun).

Workload (one step): one ADAPT-VQE job of the 32-qubit configuration --
16 orbitals, 8 alpha + 8 beta electrons, 165,636,900 determinants, seeded
synthetic integrals shaped like the H16 STO-3G chain, the spin-adapted
singles+doubles pool (3,376 operators) -- run from the Hartree-Fock
determinant for 10 ADAPT iterations (screen, select, append, re-optimise
every parameter by BFGS) in mixed precision with the learned ranker
attached, followed by the double-precision refinement of the final energy.
Each step restarts from Hartree-Fock on the resident Hamiltonian, so every
step does the same work.  `value` = ADAPT iterations per second over all
ranks (10 per step).  While psi has few nonzero amplitudes (the paper's
sparse regime) the sweeps run on the sparse-state path; the record of each
iteration says which screen selected its operator (the ranker is consulted
only once an exact screen would cost more than its feature pass), and the
line reports how often each ran.

Also reported: the same job in plain FP64 with the full exact screen (time,
and the final energies of both legs with their gap); `acceptance_long`, a
longer trajectory from Hartree-Fock (18 iterations by default) in both
precisions, which reaches supports of millions of determinants where float
arithmetic and the ranker pay; `e2e` (the job through the public API from host-resident
integrals: Hamiltonian build, pool, driver, 10 iterations, refinement,
readback, release), matrix-free H|psi> at 32 qubits in FP64 and FP32, and
H|psi> streamed from the explicitly stored Hamiltonian at 28 qubits (the
paper's CSR regime) with its fraction of the measured HBM bandwidth.

Every sweep runs in the library's kernels (libhyperion.so); the FP64 CPU
oracle is timed on a bounded sample for `cpu_baseline` and for the
`--impl reference` arm.  Other modes: --trajectory, --support-eval,
--config2, --batch, --batch-rank, --hmat, --ranker-eval, --sweeps-only,
--oracle-timing.
"""
from __future__ import annotations

import argparse
import csv
import hashlib
import io
import json
import math
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import synth  # noqa: E402

METRIC = ("H|psi> GB/s (% of ~8 TB/s) and ADAPT iters/s at 32 qubits, "
          "plain vs mixed+ranker")
ITERS_PER_JOB = 10     # the workload's ADAPT iterations from Hartree-Fock
REFINE_STEPS = 4       # double-precision BFGS steps of the final refinement
TOP_M = 32
REFRESH = 4            # every 4th ranked iteration selects from the full screen
SCREEN_NAMES = {0: "exact_dense", 1: "exact_sparse", 2: "ranker", 3: "ranker_then_full"}
# DRAM bytes per launch of the kernel classes, from ncu captures committed as
# text under profiles/ (this file names the capture, its command and the
# source files' hashes at capture time; a class whose sources changed since
# reports no traffic)
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "ncu_dram_bytes.json")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="h16_32q")
    ap.add_argument("--iters-per-job", type=int, default=ITERS_PER_JOB)
    ap.add_argument("--no-plain", action="store_true", help="skip the plain FP64 job")
    ap.add_argument("--no-e2e", action="store_true", help="skip the end-to-end leg")
    ap.add_argument("--no-sweeps", action="store_true", help="skip the H|psi> timings")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--accept-iters", type=int, default=18,
                    help="iterations of the long plain-vs-mixed trajectory from Hartree-Fock "
                         "reported as acceptance_long (0 skips it)")
    ap.add_argument("--cpu-budget", type=float, default=12.0,
                    help="seconds of oracle work per CPU sample")
    ap.add_argument("--hmat-workload", default="h14_28q",
                    help="workload of the explicit-H leg of the default run")
    ap.add_argument("--sweeps-only", action="store_true",
                    help="profiling mode: two passes of each sweep (H psi, energy, full screen, "
                         "one exp(theta A)) per dtype on a seeded state, no timing line")
    ap.add_argument("--dtypes", default="f64,f32", help="dtypes of --sweeps-only")
    ap.add_argument("--ranker-eval", action="store_true",
                    help="plain FP64 ADAPT vs mixed+ranker ADAPT with the full screen as judge: "
                         "per-iteration rank of the true argmax and energy gap")
    ap.add_argument("--iters", type=int, default=12,
                    help="iterations of --ranker-eval / --trajectory / --config2")
    ap.add_argument("--sparse-eval", action="store_true",
                    help="--ranker-eval on the sparse-state path (plain reference included)")
    ap.add_argument("--top-m", type=int, default=TOP_M,
                    help="operators the ranker proposes for the exact screen")
    ap.add_argument("--judge-only", action="store_true",
                    help="--ranker-eval without the plain run (ranks of the true argmax only)")
    ap.add_argument("--trajectory", action="store_true",
                    help="plain FP64 and mixed(+ranker) ADAPT from Hartree-Fock over --iters "
                         "iterations: per-iteration energies, selections, errors and times")
    ap.add_argument("--force-ranker", action="store_true",
                    help="--trajectory: consult the ranker on every ranked iteration")
    ap.add_argument("--refine-every", type=int, default=1,
                    help="--trajectory: refine the mixed leg in double every k-th iteration")
    ap.add_argument("--dense", action="store_true", help="--trajectory on the dense sweeps only")
    ap.add_argument("--classes", action="store_true",
                    help="--trajectory: device time per kernel class per iteration")
    ap.add_argument("--support-eval", action="store_true",
                    help="--iters plain iterations, then --reps evaluations of that ansatz "
                         "(large supports: sigma on the support)")
    ap.add_argument("--config2", action="store_true",
                    help="20 qubits: --iters plain FP64 ADAPT iterations, and the full screen as "
                         "one launch against one launch per operator")
    ap.add_argument("--oracle-timing", action="store_true",
                    help="the FP64 CPU oracle on the host cores: full ADAPT at 12 qubits, "
                         "--iters ADAPT iterations at 20 qubits, one H psi at 28 qubits")
    ap.add_argument("--hmat", action="store_true",
                    help="the Hamiltonian stored explicitly: build it for --rows alpha strings of "
                         "--workload and time H psi streamed from it against the matrix-free sweep")
    ap.add_argument("--rows", default="all",
                    help="--hmat row range 'b:e' in alpha strings, or 'all'")
    ap.add_argument("--hmat-dtypes", default="f32,f64", help="dtypes of --hmat")
    ap.add_argument("--reps", type=int, default=5, help="timed repetitions of --hmat")
    ap.add_argument("--batch-rank", action="store_true",
                    help="config 5: the 64-molecule batch with the ranker's top-M screened in "
                         "one persistent launch, the full batched screen as judge")
    ap.add_argument("--batch", action="store_true",
                    help="64 molecules of 8-12 orbitals: H psi + energies of all in one persistent "
                         "graph-captured launch (autotuned tile) vs one launch sequence per molecule")
    return ap.parse_args()


def batch_bench(args, count=64, reps=5):
    """Batched sweeps over the uneven 64-molecule workload."""
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    hams = []
    for n, na, nb, seed in synth.batch_molecules(count):
        h1, h2, ec = synth.integrals(n, seed)
        hams.append(hy.Hamiltonian(h1, h2, ec, n, na, nb))
    b = hy.Batch(hams)
    total = sum(h.n_det for h in hams)
    out = {"batch": f"{count} molecules, n = 8..12 at half filling, seeds 2000+i",
           "determinants": total, "tasks": b.n_tasks}
    st = torch.cuda.current_stream()
    for d, dt in (("f64", torch.float64), ("f32", torch.float32)):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(3)
        states = [torch.randn(h.n_det, dtype=dt, device="cuda", generator=gen) for h in hams]
        states = [x / x.norm() for x in states]
        psi = b.pack(states, dt)
        sig = torch.zeros_like(psi)
        en = torch.empty(count, dtype=torch.float64, device="cuda")
        tile, tune_ms = b.tune(psi, sig)
        b.apply_h(psi, sig, en, graph=True)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        torch.cuda.synchronize()
        l0 = hy.launch_count()
        ev[0].record(st)
        for _ in range(reps):
            b.apply_h(psi, sig, en, graph=True)
        ev[1].record(st)
        l1 = hy.launch_count()
        sigs = [torch.empty_like(x) for x in states]
        eo = [torch.empty((), dtype=torch.float64, device="cuda") for _ in hams]
        for h, x, y, e in zip(hams, states, sigs, eo):     # warm the per-molecule path
            h.apply_h(x, out=y)
            h.energy(x, y, out=e)
        torch.cuda.synchronize()
        l2 = hy.launch_count()
        ev[2].record(st)
        for _ in range(reps):
            for h, x, y, e in zip(hams, states, sigs, eo):
                h.apply_h(x, out=y)
                h.energy(x, y, out=e)
        ev[3].record(st)
        torch.cuda.synchronize()
        l3 = hy.launch_count()
        t_b = ev[0].elapsed_time(ev[1]) / reps
        t_l = ev[2].elapsed_time(ev[3]) / reps
        err = max(abs(float(en[m].item()) - float(eo[m].item())) for m in range(count))
        out[d] = {"tile": tile, "tune_ms": round(tune_ms, 3),
                  "batched_ms": round(t_b, 3), "looped_ms": round(t_l, 3),
                  "speedup": round(t_l / t_b, 2),
                  "batched_launches": (l1 - l0) // reps, "looped_launches": (l3 - l2) // reps,
                  "molecules_per_s": round(count / (t_b / 1e3), 1),
                  "max_energy_diff_vs_looped": err}
    print(json.dumps(out), flush=True)


def batch_rank_bench(args, count=64, train_iters=3, reps=5):
    """Config 5: the uneven 64-molecule batch with the learned ranker.  Each
    molecule runs `train_iters` + 1 plain FP64 ADAPT iterations from
    Hartree-Fock; the exact full screens of the states after iterations
    1 .. train_iters train one MLP ranker (3 x 256) for the whole batch.  On
    the states after the last iteration (held out) the batch then does, on
    packed buffers: sigma = H psi in one persistent launch, the features of
    every molecule's pool, one MLP inference over all operators, the top-32
    per molecule, and the exact screen of those proposals in one persistent
    launch; the full batched screen is the judge (its argmax per molecule
    and its rank among the proposals).  Timings: CUDA events on the stream,
    the ranked batch screen against the full batched screen and against a
    loop of per-molecule full screens."""
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    hams, pools, states, train = [], [], [], []
    for n, na, nb, seed in synth.batch_molecules(count):
        h1, h2, ec = synth.integrals(n, seed)
        ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
        pool = hy.Pool(ham)
        ad = hy.Adapt(ham, pool, "f64", max_iter=train_iters + 2)
        for it in range(train_iters + 1):
            ad.step()
            if it < train_iters:
                train.append((len(hams), ad.state(torch.float64)))
        states.append(ad.state(torch.float64))
        ad.close()
        hams.append(ham)
        pools.append(pool)
    ranker = hy.Ranker(hidden=256, seed=7)
    for m, x in train:
        sig = hams[m].apply_h(x)
        feat = hy.ranker_features(hams[m], pools[m], x, sigma=sig)
        ranker.add_samples(feat, pools[m].gradients(x, sig))
    loss = ranker.fit(epochs=30)
    b = hy.Batch(hams)
    b.set_pools(pools)
    K = np.array([len(p) for p in pools])
    poff = b.pool_offsets
    M = args.top_m
    st = torch.cuda.current_stream()
    psi = b.pack(states, torch.float64)
    sig = torch.zeros_like(psi)
    feat = torch.empty((int(poff[-1]), 16), dtype=torch.float32, device="cuda")
    prop = torch.empty(count * M, dtype=torch.int32, device="cuda")
    poffs = torch.arange(count + 1, dtype=torch.int64, device="cuda") * M
    psis, sigs = b.unpack(psi), b.unpack(sig)

    def ranked():
        b.apply_h(psi, sig, graph=True)
        for m in range(count):
            hy.ranker_features(hams[m], pools[m], psis[m], sigma=sigs[m],
                               out=feat[int(poff[m]):int(poff[m + 1])])
        score = ranker.predict(feat)
        for m in range(count):
            kk = min(M, int(K[m]))
            prop[m * M:m * M + kk] = hy.topk(score[int(poff[m]):int(poff[m + 1])], kk)
            if kk < M:                            # a pool smaller than M: repeat its first
                prop[m * M + kk:(m + 1) * M] = prop[m * M]
        return b.gradients(psi, sig, ops=prop, op_offsets=poffs)

    def full():
        b.apply_h(psi, sig, graph=True)
        return b.gradients(psi, sig)

    def looped():
        out = []
        for m in range(count):
            y = hams[m].apply_h(psis[m])
            out.append(pools[m].gradients(psis[m], y))
        return out

    times = {}
    for name, fn in (("ranked", ranked), ("full", full), ("looped", looped)):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        l0 = hy.launch_count()
        e0.record(st)
        for _ in range(reps):
            r = fn()
        e1.record(st)
        torch.cuda.synchronize()
        times[name] = (e0.elapsed_time(e1) / reps, (hy.launch_count() - l0) // reps)
    gp = ranked().cpu().numpy()
    gf = full().cpu().numpy()
    pr = prop.cpu().numpy()
    hits, ranks, gaps = 0, [], []
    for m in range(count):
        gm = np.abs(gf[poff[m]:poff[m + 1]])
        true = int(np.argmax(gm))
        sub = pr[m * M:m * M + min(M, int(K[m]))]
        pick = int(sub[int(np.argmax(np.abs(gp[m * M:m * M + len(sub)])))])
        hits += pick == true
        where = np.flatnonzero(sub == true)
        ranks.append(int(where[0]) if where.size else -1)
        gaps.append(float(gm[true] - gm[pick]) / max(gm[true], 1e-300))
    out = {"batch_rank": f"{count} molecules, n = 8..12 at half filling, seeds 2000+i",
           "determinants": int(sum(h.n_det for h in hams)), "operators": int(poff[-1]),
           "train": {"states": len(train), "samples": ranker.info()["n_samples"],
                     "final_loss": round(float(loss), 5)},
           "top_m": M,
           "selected_true_argmax": f"{hits} of {count}",
           "true_argmax_rank_in_proposals": ranks,
           "max_relative_gradient_shortfall": round(max(gaps), 4),
           "ms": {k: round(v[0], 3) for k, v in times.items()},
           "launches": {k: v[1] for k, v in times.items()},
           "speedup_ranked_vs_full_batched": round(times["full"][0] / times["ranked"][0], 2),
           "speedup_full_batched_vs_looped": round(times["looped"][0] / times["full"][0], 2)}
    print(json.dumps(out), flush=True)


def hmat_bench(args):
    """H psi streamed from the explicitly stored Hamiltonian (a range of its
    rows) against the matrix-free sweep of the same rows: CUDA events on the
    launching stream, inputs resident, the matrix far larger than L2 so every
    repetition streams it from HBM.  Bytes = the stored matrix (16-bit beta
    columns, values, segment partners) + psi rows read + sigma rows written."""
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    peaks, peak_kind = load_peaks()
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    NA, NB = ham.n_alpha_str, ham.n_beta_str
    b, e = (0, NA) if args.rows == "all" else tuple(int(x) for x in args.rows.split(":"))
    st = torch.cuda.current_stream()
    out = {"hmat": args.workload, "rows": [b, e], "n_det_rows": (e - b) * NB,
           "row_len": None, "peak_gbs": peaks["hbm_gbs"], "peak_kind": peak_kind}
    for d in args.hmat_dtypes.split(","):
        dt = torch.float64 if d == "f64" else torch.float32
        by, nnz = hy.ExplicitH.size(ham, dt, b, e)
        free, _ = torch.cuda.mem_get_info()
        if by + (1 << 30) + 2 * ham.n_det * (8 if d == "f64" else 4) > free:
            out[d] = {"skipped": f"needs {by} bytes, {free} free"}
            continue
        t0 = time.perf_counter()
        m = hy.ExplicitH(ham, dt, b, e)
        t_build = time.perf_counter() - t0
        out["row_len"] = m.row_len
        gen = torch.Generator(device="cuda")
        gen.manual_seed(2)
        psi = torch.randn(ham.n_det, dtype=dt, device="cuda", generator=gen)
        sig = torch.empty((e - b) * NB, dtype=dt, device="cuda")
        m.apply(psi, out=sig)
        ham.apply_h_rows(psi, b, e, out=sig)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * args.reps + 2)]
        torch.cuda.synchronize()
        ms_m = []
        for r in range(args.reps):
            ev[2 * r].record(st)
            m.apply(psi, out=sig)
            ev[2 * r + 1].record(st)
        torch.cuda.synchronize()
        ms_m = [ev[2 * r].elapsed_time(ev[2 * r + 1]) for r in range(args.reps)]
        ref = sig.clone()
        ham.apply_h_rows(psi, b, e, out=sig)
        diff = float(torch.max(torch.abs(sig - ref)).item() / torch.max(torch.abs(ref)).item())
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(args.reps):
            ham.apply_h_rows(psi, b, e, out=sig)
        e1.record(st)
        torch.cuda.synchronize()
        ms_mf = e0.elapsed_time(e1) / args.reps
        es = 8 if d == "f64" else 4
        traffic = by + 2 * (e - b) * NB * es
        ms = statistics.median(ms_m)
        gbs = traffic / (ms / 1e3) / 1e9
        out[d] = {"build_s": round(t_build, 2), "matrix_bytes": by, "nnz": nnz,
                  "ms": round(ms, 4), "ms_all": [round(x, 4) for x in ms_m],
                  "gbs": round(gbs, 1), "frac_of_hbm": round(gbs / peaks["hbm_gbs"], 4),
                  "matrix_free_ms": round(ms_mf, 4),
                  "max_rel_diff_vs_matrix_free": diff}
        del m, psi, sig, ref
        torch.cuda.empty_cache()
    print(json.dumps(out), flush=True)


def ranker_eval(args):
    """The ranker judged against the full screen: plain FP64 ADAPT and the
    mixed+ranker ADAPT (double refinement every iteration so energies compare
    at FP64) run side by side; per iteration the rank of the true argmax
    among the ranker's proposals and the energy gap to the plain run."""
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    it = args.iters
    # the sparse path makes the plain FP64 reference affordable at 32 q; the
    # ranker is asked on every ranked iteration (no exact sparse screen)
    sp = dict(sparse=True, exact_screen_work=-1.0) if args.sparse_eval else {}
    plain = None if args.judge_only else hy.Adapt(ham, pool, "f64", max_iter=it,
                                                  **sp).run(it)
    ranker = hy.Ranker(hidden=256, seed=7)
    ad = hy.Adapt(ham, pool, "mixed", max_iter=it, screen_top_m=args.top_m, judge=True,
                  refine_every=0 if args.judge_only else 1, **sp)
    ad.set_ranker(ranker, warm_iters=args.warmup, epochs=30, refresh_every=REFRESH)
    ranked = ad.run(it)
    rows = []
    for i, r in enumerate(ranked):
        row = {"iter": r["iter"], "e_ranked": r["energy"], "true_rank": r["true_rank"],
               "selected": r["selected"], "true_argmax": r["true_argmax"],
               "t_screen_ranked": round(r["t_screen"], 5), "t_total": round(r["t_total"], 3)}
        if plain is not None:
            p = plain[i]
            row.update({"e_plain": p["energy"], "gap": r["energy"] - p["energy"],
                        "same_op": p["selected"] == r["selected"],
                        "t_screen_plain": round(p["t_screen"], 5)})
        rows.append(row)
    print(json.dumps({"ranker_eval": args.workload, "top_m": args.top_m, "warm": args.warmup,
                      "refresh_every": REFRESH, "pool_ops": len(pool), "rows": rows}), flush=True)


def sweeps_only(args):
    """Two passes of every sweep on a seeded random state, for ncu captures."""
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    for d in args.dtypes.split(","):
        dt = torch.float64 if d == "f64" else torch.float32
        psi = torch.randn(ham.n_det, dtype=dt, device="cuda", generator=gen)
        psi /= psi.norm()
        sig = torch.empty_like(psi)
        for _ in range(2):
            ham.apply_h(psi, out=sig)
            e = ham.energy(psi, sig)
            g = pool.gradients(psi, sig)
            pool.apply_excitation(len(pool) - 1, 0.1, psi)
        torch.cuda.synchronize()
        print(json.dumps({"sweeps": args.workload, "dtype": d, "energy": float(e.item()),
                          "max_grad": float(g.abs().max().item())}), flush=True)


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.idx = device_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        out, _ = self.proc.communicate(timeout=10)
        rows = [r for r in csv.reader(io.StringIO(out)) if len(r) >= 9]
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                sm.append(float(r[1]))
                mx.append(float(r[2]))
            except ValueError:
                continue
            for nm, v in zip(names, r[5:9]):
                if v.strip().lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------
# oracle timing on the host cores (bounded samples of the same workload)
# ---------------------------------------------------------------------------
def oracle_job_estimate(n, na, nb, seed, budget_s, records, state=None):
    """Seconds the FP64 CPU oracle would take for the plain ADAPT job whose
    per-iteration evaluation counts `records` holds ([(ansatz length, evals)]),
    extrapolated from a bounded sample: sigma on sampled rows, the gradient of
    a few pool operators (each O(N_det)), one exp(theta A).  The oracle has no
    sparse path, so each of its evaluations is a full sweep.
    Returns (seconds, threads, seconds actually spent, sample description)."""
    import oracle
    t_start = time.perf_counter()
    h1, h2, ec = synth.integrals(n, seed)
    ref = oracle.System(h1, h2, ec, n, na, nb)
    threads = len(os.sched_getaffinity(0))
    if state is None:
        state = synth.random_state(ref.n_det, 99)
    rng = np.random.default_rng(1)
    rows = rng.integers(0, ref.n_det, 64 * threads)
    t0 = time.perf_counter()
    ref.sigma_rows(state, rows, threads)
    dt = time.perf_counter() - t0
    m = int(min(ref.n_det, max(len(rows), len(rows) * 0.5 * budget_s / max(dt, 1e-6))))
    rows = rng.integers(0, ref.n_det, m)
    t0 = time.perf_counter()
    ref.sigma_rows(state, rows, threads)
    t_rows = time.perf_counter() - t0
    t_sigma = t_rows * ref.n_det / m
    pool = ref.pool()
    nops = max(1, min(threads, 4))
    t0 = time.perf_counter()
    ref.gradients(pool[:nops], state, state, nops)
    t_g = time.perf_counter() - t0
    t_op = t_g / nops            # one operator's gradient, one thread
    t0 = time.perf_counter()
    ref.apply_excitation(pool[len(pool) - 1], 0.1, state)
    t_x = time.perf_counter() - t0
    # per iteration: the screen (all operators, parallel over threads), then
    # per evaluation: prepare (L exps), sigma, energy, adjoint gradient (2L
    # exps and L generator dots)
    t_screen = t_op * len(pool) / threads
    total = 0.0
    for L, ev in records:
        total += t_screen + ev * (t_sigma + 3 * L * t_x + L * t_op)
    spent = time.perf_counter() - t_start
    sample = (f"sigma on {m} sampled rows ({t_rows:.1f} s, {threads} threads), gradients of "
              f"{nops} ops ({t_g:.1f} s), one exp(theta A) ({t_x:.1f} s); extrapolated to the "
              f"plain ADAPT job of {len(records)} iterations ({sum(e for _, e in records)} "
              f"evaluations, screens of {len(pool)} ops) over {ref.n_det} determinants")
    return total, threads, spent, sample


# ---------------------------------------------------------------------------
# the GPU arm
# ---------------------------------------------------------------------------
def max_over_ranks(values, device="cpu"):
    """Element-wise maximum of per-rank timings over the process group (the
    job's time is its slowest replica's)."""
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return t.tolist()


def job_throughput(world, iterations, ms_max):
    """Whole-job iterations per second: every rank ran `iterations` ADAPT
    iterations of its own replica within the slowest rank's `ms_max` ms."""
    return world * iterations / (ms_max / 1e3)


def time_sweeps(ham, pool, dt, reps=3):
    """Mean device time (ms) of H psi and of the full screen in dtype dt, and
    of the alpha-beta coupling alone (events the library records around it)."""
    import torch
    g = torch.Generator(device=ham.device)
    g.manual_seed(5)
    psi = torch.randn(ham.n_det, dtype=dt, device=ham.device, generator=g)
    psi /= psi.norm()
    sig = torch.empty_like(psi)
    gr = torch.empty(len(pool), dtype=torch.float64, device=ham.device)
    st = torch.cuda.current_stream()
    ham.apply_h(psi, out=sig)
    pool.gradients(psi, sig, out=gr)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    torch.cuda.synchronize()
    e[0].record(st)
    for _ in range(reps):
        ham.apply_h(psi, out=sig)
    e[1].record(st)
    for _ in range(reps):
        pool.gradients(psi, sig, out=gr)
    e[2].record(st)
    torch.cuda.synchronize()
    ham.profile_coupling(True)
    cpl = []
    for _ in range(reps):
        ham.apply_h(psi, out=sig)
        cpl.append(ham.coupling_ms())
    ham.profile_coupling(False)
    return e[0].elapsed_time(e[1]) / reps, e[1].elapsed_time(e[2]) / reps, statistics.mean(cpl)


def barrier(world):
    import torch
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
        torch.cuda.synchronize()


def run_job(ad, iters, refine_steps):
    """One ADAPT job from Hartree-Fock: `iters` iterations, then (mixed
    precision) the double-precision refinement.  Returns (records, final
    energy, refinement seconds)."""
    ad.set_ansatz([], [])
    recs = ad.run(iters)
    if ad.precision == "mixed":
        t0 = time.perf_counter()
        e = ad.refine(steps=refine_steps)
        return recs, e, time.perf_counter() - t0
    done = [r for r in recs if not r["converged"]]
    return recs, (done[-1]["energy"] if done else float("nan")), 0.0


def roofline_class(prof):
    """The kernel class the roofline reports: the most device time among the
    classes whose algorithmic work the host knows (None: no such class)."""
    known = [c for c, v in prof.items() if v["launches"] and (v["bytes"] > 0 or v["flops"] > 0)]
    return max(known, key=lambda c: prof[c]["ms"]) if known else None


def profiled_warmup(run, hy):
    """Runs `run` once with CUDA events around every launch of every kernel
    class: the per-class breakdown of an untimed job (and its host wall time
    in ms, synchronised on both sides), from which the class that the timed
    region records is chosen."""
    import torch
    torch.cuda.synchronize()
    hy.profile_enable(hy.PROFILE_CLASSES)
    t0 = time.perf_counter()
    run()
    torch.cuda.synchronize()
    ms = (time.perf_counter() - t0) * 1e3
    prof = {c: hy.profile_read(c) for c in hy.PROFILE_CLASSES}
    hy.profile_enable([])
    return prof, ms


def headline_leg(ham, pool, hy, torch, args, rank, world, clocks):
    """Mixed precision + ranker jobs on the resident Hamiltonian: W warm-up
    jobs (the last one with events around every launch of every kernel
    class), then K timed jobs between CUDA events on the launching stream,
    recording per-launch events for the roofline's kernel class only."""
    J, W, K = args.iters_per_job, args.warmup, args.steps
    stream = torch.cuda.current_stream()
    ranker = hy.Ranker(hidden=256, seed=7 + rank)
    ad = hy.Adapt(ham, pool, "mixed", max_iter=J, screen_top_m=args.top_m, refine_every=1,
                  refine_steps=REFINE_STEPS, sparse=True)
    ad.set_ranker(ranker, warm_iters=3, epochs=30, refresh_every=REFRESH)
    for _ in range(W - 1):
        run_job(ad, J, REFINE_STEPS)
    warm, warm_ms = profiled_warmup(lambda: run_job(ad, J, REFINE_STEPS), hy) if W else ({}, 0.0)
    roof = roofline_class(warm) if W else "hpsi_sparse"
    barrier(world)
    if clocks:
        clocks.start()
    l0 = hy.launch_count()
    hy.profile_enable([roof] if roof else [])
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    jobs = [run_job(ad, J, REFINE_STEPS) for _ in range(K)]
    t1.record(stream)
    barrier(world)
    clk = clocks.stop() if clocks else None
    launches = hy.launch_count() - l0
    ms = t0.elapsed_time(t1)
    prof = {c: hy.profile_read(c) for c in hy.PROFILE_CLASSES}
    hy.profile_enable([])
    del ad
    iters = sum(len(r) for r, _, _ in jobs)
    return dict(ms=ms, launches=launches, clocks=clk, jobs=jobs, prof=prof, ranker=ranker,
                iterations=iters, warm=warm, warm_ms=warm_ms, roof=roof)


def e2e_leg(hy, torch, args, ranker, n, na, nb, seed, world):
    """The job through the public API from host-resident integrals, every
    step: Hamiltonian build (host tables, device upload), pool, driver, the
    iterations and the refinement, readback of the ansatz and energy,
    release.  Bytes: every host->device upload of the build, the pool and
    the driver, and every device->host readback."""
    J, K = args.iters_per_job, args.steps
    h1, h2, ec = synth.integrals(n, seed)
    stream = torch.cuda.current_stream()
    h2d = d2h = 0
    iters = 0
    energies = []
    barrier(world)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    w0 = time.perf_counter()
    t0.record(stream)
    for _ in range(K):
        ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
        pool = hy.Pool(ham)
        ad = hy.Adapt(ham, pool, "mixed", max_iter=J, screen_top_m=args.top_m, refine_every=1,
                      refine_steps=REFINE_STEPS, sparse=True)
        ad.set_ranker(ranker, warm_iters=3, epochs=30, refresh_every=REFRESH)
        recs = ad.run(J)
        e = ad.refine(steps=REFINE_STEPS)
        ops, th = ad.ansatz()
        iters += len(recs)
        energies.append(e)
        i_h2d, i_d2h = ad.io_bytes()
        h2d += ham.upload_bytes(pool) + i_h2d
        d2h += i_d2h + 16 * len(ops) + 8
        ad.close()
        pool.close()
        ham.close()
    t1.record(stream)
    barrier(world)
    wall = time.perf_counter() - w0
    ms = t0.elapsed_time(t1)
    if world > 1:
        ms = max_over_ranks([ms], torch.device("cuda"))[0]
    return dict(ms=ms, wall_s=wall, iterations=iters, h2d=h2d / K, d2h=d2h / K,
                energies=energies)


def plain_leg(ham, pool, hy, torch, args, roof):
    """The same job in plain FP64 (full exact screen of the whole pool every
    iteration): one warm-up job (events around every launch of every class),
    one timed job."""
    J = args.iters_per_job
    stream = torch.cuda.current_stream()
    ad = hy.Adapt(ham, pool, "f64", max_iter=J, sparse=True)
    warm, warm_ms = profiled_warmup(lambda: run_job(ad, J, 0), hy)
    # the same per-launch events as the headline's timed region (the
    # roofline's class), so that both carry the same host cost of recording
    # them
    hy.profile_enable([roof] if roof else [])
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    recs, e, _ = run_job(ad, J, 0)
    t1.record(stream)
    torch.cuda.synchronize()
    ms = t0.elapsed_time(t1)
    prof = {c: hy.profile_read(c) for c in hy.PROFILE_CLASSES}
    hy.profile_enable([])
    del ad
    return dict(ms=ms, records=recs, energy=e, prof=prof, warm=warm, warm_ms=warm_ms)


def explicit_h_leg(hy, torch, args, peaks):
    """H psi streamed from the explicitly stored Hamiltonian of the 28-qubit
    workload (all rows in float when they fit, else a block; half the rows
    in double), against the matrix-free sweep of the same rows."""
    n, na, nb, seed = synth.workload(args.hmat_workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    NA, NB = ham.n_alpha_str, ham.n_beta_str
    st = torch.cuda.current_stream()
    out = {"workload": f"{args.hmat_workload}: {n} orbitals, {ham.n_det} determinants",
           "row_unit": "alpha string (n_beta_str determinants)"}
    for d, dt in (("f32", torch.float32), ("f64", torch.float64)):
        es = 4 if d == "f32" else 8
        free, _ = torch.cuda.mem_get_info()
        room = free - (2 << 30) - 3 * ham.n_det * es
        full_b, _ = hy.ExplicitH.size(ham, dt)
        e_rows = NA if full_b <= room else max(1, int(NA * room / full_b * 0.98))
        b, e = 0, min(NA, e_rows)
        by, nnz = hy.ExplicitH.size(ham, dt, b, e)
        t0 = time.perf_counter()
        m = hy.ExplicitH(ham, dt, b, e)
        t_build = time.perf_counter() - t0
        gen = torch.Generator(device="cuda")
        gen.manual_seed(2)
        psi = torch.randn(ham.n_det, dtype=dt, device="cuda", generator=gen)
        sig = torch.empty((e - b) * NB, dtype=dt, device="cuda")
        m.apply(psi, out=sig)
        torch.cuda.synchronize()
        reps = 5
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * reps)]
        for r in range(reps):
            ev[2 * r].record(st)
            m.apply(psi, out=sig)
            ev[2 * r + 1].record(st)
        torch.cuda.synchronize()
        ms = statistics.median([ev[2 * r].elapsed_time(ev[2 * r + 1]) for r in range(reps)])
        ref = ham.apply_h_rows(psi, b, e)
        rel = float(torch.max(torch.abs(sig - ref)).item() / torch.max(torch.abs(ref)).item())
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(reps):
            ham.apply_h_rows(psi, b, e, out=ref)
        e1.record(st)
        torch.cuda.synchronize()
        traffic = by + 2 * (e - b) * NB * es
        gbs = traffic / (ms / 1e3) / 1e9
        out[d] = {"rows": [b, e], "rows_of": NA, "matrix_bytes": by, "nnz": nnz,
                  "row_len": m.row_len, "build_s": round(t_build, 2), "ms": round(ms, 3),
                  "gbs": round(gbs, 1), "frac_of_hbm": round(gbs / peaks["hbm_gbs"], 4),
                  "matrix_free_rows_ms": round(e0.elapsed_time(e1) / reps, 3),
                  "max_rel_diff_vs_matrix_free": rel}
        del m, psi, sig, ref
        torch.cuda.empty_cache()
    ham.close()
    return out


def run_ours(args, rank, world):
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild

    hybuild.build()
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", 0)))
    torch.cuda.set_device(dev)
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    tb = time.perf_counter()
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    t_build = time.perf_counter() - tb
    out = dict(N=ham.n_det, K=len(pool), n=n, na=na, nb=nb, seed=seed, t_build=t_build,
               conn=ham.connections_per_det(), n_alpha_str=ham.n_alpha_str,
               n_beta_str=ham.n_beta_str)
    out["head"] = headline_leg(ham, pool, hy, torch, args, rank, world, Clocks(dev.index))
    if world > 1:
        out["head"]["ms"] = max_over_ranks([out["head"]["ms"]], torch.device("cuda"))[0]
    if not args.no_plain:
        out["plain"] = plain_leg(ham, pool, hy, torch, args, out["head"]["roof"])
    if args.accept_iters > 0:
        out["accept"] = acceptance_run(ham, pool, hy, args.accept_iters, args.top_m)
    if not args.no_sweeps:
        out["hpsi_ms_f64"], out["screen_ms_f64"], out["cpl_ms_f64"] = time_sweeps(
            ham, pool, torch.float64)
        out["hpsi_ms_f32"], out["screen_ms_f32"], out["cpl_ms_f32"] = time_sweeps(
            ham, pool, torch.float32)
    ranker = out["head"].pop("ranker")
    pool.close()
    ham.close()
    torch.cuda.empty_cache()
    if not args.no_e2e:
        out["e2e"] = e2e_leg(hy, torch, args, ranker, n, na, nb, seed, world)
    del ranker
    torch.cuda.empty_cache()
    if not args.no_sweeps:
        peaks, _ = load_peaks()
        out["explicit_h"] = explicit_h_leg(hy, torch, args, peaks)
    return out


# kernels behind each class of the library's event profiler
CLASS_KERNELS = {
    "hpsi": "k_rows64 (double, up to 1,716 beta strings), k_same or k_spmm with their transposes, "
            "coupling (dense H|psi>)",
    "hpsi_sparse": "sparse H|psi>: k_hpsi_scatter (all of sigma, after a memset), "
                   "k_hss_apply (the stored support Hamiltonian), k_sup_rows (float: k_sup_alpha + k_sup_beta) "
                   "(rows of the support)",
    "excite": "k_excite / k_excite_n (dense pair rotations: 4 s bytes per pair)",
    "sparse_excite": "k_sv_excite, k_sv_prepare, support programs k_prog_prepare[_big] + "
                     "k_prog_grad[_big] and their compilation, H_SS build",
    "screen": "k_screen, k_screen32 or k_grad_partial with their sums (dense pool gradients)",
    "screen_sparse": "k_grad_sparse + k_grad_sparse_final (support-restricted pool "
                     "gradients)",
    "reduce": "dots, norms, renormalisation",
    "features": "k_pair_weights + k_pair_contract + k_pair_reduce + occupations + k_features",
    "hmat": "k_hmat_spmv (H psi streamed from the explicit H)",
}
# the source files whose kernels each class launches (for the traffic record)
CLASS_SOURCES = {
    "hpsi": ["hy_sigma.cu", "hy_cpl_tc.cu", "hy_same.cu", "hy_rows64.cu"],
    "hpsi_sparse": ["hy_sparse.cu", "hy_api.cu", "hy_adapt.cpp"],
    "excite": ["hy_sweeps.cu"], "sparse_excite": ["hy_sparse.cu"],
    "screen": ["hy_sweeps.cu", "hy_screen.cu", "hy_screen32.cu"], "screen_sparse": ["hy_sparse.cu"],
    "reduce": ["hy_sweeps.cu"], "features": ["hy_ranker.cu"], "hmat": ["hy_hmat.cu"],
}


def source_hash(files):
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, "paper_2604_01176_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def traffic_for(cls, launches_per_unit=1.0):
    """DRAM bytes per launch of a kernel class from the committed ncu record,
    or None when there is none or the class's sources changed since."""
    try:
        with open(TRAFFIC_FILE) as f:
            rec = json.load(f).get(cls)
    except (OSError, ValueError):
        return None, None
    if not rec or rec.get("source_sha") != source_hash(CLASS_SOURCES.get(cls, [])):
        return None, rec.get("workload") if rec else None
    return float(rec["dram_bytes_per_launch"]) * launches_per_unit, rec.get("workload")


def breakdown(prof, step_ms):
    """Device time per kernel class in the timed region (CUDA events on the
    launching stream), as a share of the region's wall time."""
    return {c: {"launches": v["launches"], "ms": round(v["ms"], 3),
                "share_of_step": round(v["ms"] / step_ms, 4)}
            for c, v in prof.items() if v["launches"]}


# classes bound by arithmetic rather than HBM
ALU_CLASSES = ("hpsi",)


def step_roofline(prof, peaks, peak_kind, fp32_peak, dominant=None):
    """Roofline of the kernel class with the most device time among those
    whose algorithmic work the host knows: bytes / event time against the
    measured HBM copy rate, or flops / event time against the derived FP32
    rate for the arithmetic-bound classes.  dominant: the class with the most
    device time overall, when prof records only some classes."""
    known = {c: v for c, v in prof.items()
             if v["launches"] and (v["bytes"] > 0 or v["flops"] > 0)}
    estimated = {"sparse_excite": "bytes estimated from the support sizes the host last read back"}
    top_all = dominant or max(prof, key=lambda c: prof[c]["ms"])
    if not known:
        return {"bound": "hbm", "achieved": None, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": None, "traffic": None, "dominant_class": top_all}
    c = max(known, key=lambda k: known[k]["ms"])
    v = known[c]
    traffic, _ = traffic_for(c)
    out = {"kernel_class": c, "kernel": CLASS_KERNELS[c], "launches": v["launches"],
           "ms_per_launch": round(v["ms"] / v["launches"], 4), "dominant_class": top_all,
           "timing": "CUDA events around each launch on its stream, over the timed region",
           "traffic": traffic}
    if c in ALU_CLASSES and v["flops"] > 0:
        tf = v["flops"] / (v["ms"] / 1e3) / 1e12
        out.update(bound="alu", achieved=round(tf, 3), peak=round(fp32_peak, 3), unit="TFLOP/s",
                   frac=round(tf / fp32_peak, 4), flops_per_launch=round(v["flops"] / v["launches"]),
                   peak_kind="derived FP32 FMA rate: 152 SMs x 128 FMA/clk x 2 x max SM clock")
    else:
        gbs = v["bytes"] / (v["ms"] / 1e3) / 1e9
        out.update(bound="hbm", achieved=round(gbs, 1), peak=peaks["hbm_gbs"], unit="GB/s",
                   frac=round(gbs / peaks["hbm_gbs"], 4),
                   bytes_per_launch=round(v["bytes"] / v["launches"]),
                   peak_kind=f"{peak_kind} copy bandwidth (MEASURED_PEAKS.json hbm_gbs)")
        if c in estimated:
            out["bytes_note"] = estimated[c]
    return out


def c_tilde(records):
    """The paper's amortised ADAPT coefficient C~ = j / sqrt(T_j) (Numerical
    performance subsection): j iterations from Hartree-Fock, T_j their summed
    wall time in seconds (each iteration's host-measured total)."""
    t = sum(float(r["t_total"]) for r in records)
    j = len(records)
    return {"iterations": j, "t_s": round(t, 6),
            "value": round(j / math.sqrt(t), 3) if t > 0 else None, "unit": "s^-1/2"}


def screens_used(jobs):
    counts = {}
    for recs, _, _ in jobs:
        for r in recs:
            nm = SCREEN_NAMES.get(int(r["screen"]), str(r["screen"]))
            counts[nm] = counts.get(nm, 0) + 1
    return counts


def run_steps(ad, iters, hy, classes):
    """`iters` ADAPT steps; with `classes`, the device time of every kernel
    class per iteration (CUDA events around each launch) beside each record."""
    recs = []
    for _ in range(iters):
        if classes:
            hy.profile_enable(hy.PROFILE_CLASSES)
        r = ad.step()
        if classes:
            r["classes_ms"] = {c: round(v["ms"], 2) for c in hy.PROFILE_CLASSES
                               for v in [hy.profile_read(c)] if v["launches"]}
            hy.profile_enable([])
        recs.append(r)
        if r["converged"]:
            break
    return recs


def acceptance_run(ham, pool, hy, iters, top_m=TOP_M, refine_every=1, sparse=True,
                   force_ranker=False, classes=False):
    """Plain FP64 (whole pool screened exactly every iteration) and mixed
    precision + ranker ADAPT from Hartree-Fock over `iters` iterations on one
    resident Hamiltonian: per iteration the selected operators, the energies
    (the mixed leg's refined in double every `refine_every` iterations, the
    float error beside it), the screen used and the host wall time; then the
    mixed leg's final double refinement and its gap to the plain energy."""
    t0 = time.perf_counter()
    plain = hy.Adapt(ham, pool, "f64", max_iter=iters, sparse=sparse)
    precs = run_steps(plain, iters, hy, classes)
    plain_s = time.perf_counter() - t0
    plain.close()
    ranker = hy.Ranker(hidden=256, seed=7)
    extra = dict(exact_screen_work=-1.0) if force_ranker else {}
    ad = hy.Adapt(ham, pool, "mixed", max_iter=iters, screen_top_m=top_m,
                  refine_every=refine_every, refine_steps=REFINE_STEPS, sparse=sparse, **extra)
    ad.set_ranker(ranker, warm_iters=3, epochs=30, refresh_every=REFRESH)
    t0 = time.perf_counter()
    mrecs = run_steps(ad, iters, hy, classes)
    t1 = time.perf_counter()
    e_final = ad.refine(steps=REFINE_STEPS)
    mixed_s, refine_s = t1 - t0, time.perf_counter() - t1
    ad.close()
    ranker.close()
    rows = []
    for p, m in zip(precs, mrecs):
        row = {"iter": p["iter"], "op_plain": p["selected"], "op_mixed": m["selected"],
               "same_op": p["selected"] == m["selected"], "e_plain": p["energy"],
               "e_mixed": m["energy"], "e_mixed_minus_plain": m["energy"] - p["energy"],
               "mixed_f32_err": m["energy_bulk_err"],
               "screen_mixed": SCREEN_NAMES.get(int(m["screen"])),
               "support": m["support"], "evals_plain": p["n_evals"],
               "evals_mixed": m["n_evals"], "evals_mixed_f64": m["n_evals_f64"],
               "t_plain_s": round(p["t_total"], 4), "t_mixed_s": round(m["t_total"], 4)}
        if classes:
            row["classes_ms_plain"] = p["classes_ms"]
            row["classes_ms_mixed"] = m["classes_ms"]
        rows.append(row)
    e_plain = precs[-1]["energy"]
    return {"iterations": len(rows), "sparse_path": sparse, "ranker_forced": bool(force_ranker),
            "refine_every": refine_every, "plain_s": round(plain_s, 3),
            "mixed_s": round(mixed_s, 3), "refine_s": round(refine_s, 3),
            "speedup": round(plain_s / (mixed_s + refine_s), 3),
            "e_plain_final": e_plain, "e_mixed_final_refined": e_final,
            "final_gap": e_final - e_plain,
            "equal_final_energy_1e-6": abs(e_final - e_plain) <= 1e-6,
            "same_selections": all(r["same_op"] for r in rows),
            "ranker_consulted_iterations": sum(r["screen_mixed"] == "ranker" for r in rows),
            "rows": rows}


def trajectory(args):
    """--iters iterations of --workload from Hartree-Fock, plain FP64 against
    mixed precision + ranker (acceptance_run), printed as one JSON line."""
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    out = {"trajectory": args.workload}
    out.update(acceptance_run(ham, pool, hy, args.iters, args.top_m, args.refine_every,
                              not args.dense, args.force_ranker, args.classes))
    print(json.dumps(out), flush=True)


def support_eval(args):
    """Large-support evaluations: --iters plain FP64 ADAPT iterations of
    --workload from Hartree-Fock on the sparse path, then --reps evaluations
    of the final ansatz in each precision (the first one lists the support,
    the others form sigma on it only); device time per kernel class."""
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    plain = hy.Adapt(ham, pool, "f64", max_iter=args.iters + 1, sparse=True)
    recs = plain.run(args.iters)
    ops, th = plain.ansatz()
    plain.close()
    import torch
    out = {"support_eval": args.workload, "ansatz_len": len(ops),
           "support": recs[-1]["support"]}
    for prec, dt in (("f64", torch.float64), ("mixed", torch.float32)):
        ad = hy.Adapt(ham, pool, prec, max_iter=len(ops) + 1, sparse=True,
                      sparse_cap=ham.n_det // 8)
        ad.set_ansatz(list(ops), list(th))
        e0, _ = ad.evaluate(th, dt)
        hy.profile_enable(hy.PROFILE_CLASSES)
        t0 = time.perf_counter()
        for _ in range(args.reps):
            e, _ = ad.evaluate(th, dt)
        dt_s = time.perf_counter() - t0
        prof = {c: v for c in hy.PROFILE_CLASSES for v in [hy.profile_read(c)]
                if v["launches"]}
        hy.profile_enable([])
        out[prec] = {"energy": e, "first_minus_rest": e0 - e,
                     "ms_per_eval": round(dt_s / args.reps * 1e3, 3),
                     "classes_ms_per_eval": {c: round(v["ms"] / args.reps, 3)
                                             for c, v in prof.items()}}
        ad.close()
    print(json.dumps(out), flush=True)


def config2(args):
    """20 qubits (63,504 determinants): --iters plain FP64 ADAPT iterations
    from Hartree-Fock on the dense sweeps (iterations/s), then at the final
    state the full screen of the pool as one launch pair against one launch
    pair per operator."""
    import torch
    import paper_2604_01176_gb300 as hy
    from paper_2604_01176_gb300 import build as hybuild
    hybuild.build()
    n, na, nb, seed = synth.workload("h10_20q")
    h1, h2, ec = synth.integrals(n, seed)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    pool = hy.Pool(ham)
    st = torch.cuda.current_stream()
    out = {"config2": "h10_20q", "n_det": ham.n_det, "pool_ops": len(pool)}
    for sparse in (False, True):
        ad = hy.Adapt(ham, pool, "f64", max_iter=args.iters, sparse=sparse)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        recs = ad.run(args.iters)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        key = "adapt_sparse_path" if sparse else "adapt_dense"
        out[key] = {"iterations": len(recs), "s": round(dt, 3),
                    "iters_per_s": round(len(recs) / dt, 3),
                    "final_energy": recs[-1]["energy"],
                    "evals": sum(r["n_evals"] for r in recs),
                    "c_tilde": c_tilde(recs)}
        if not sparse:
            psi = ad.state(torch.float64)
        ad.close()
    sig = ham.apply_h(psi)
    K = len(pool)
    g1 = pool.gradients(psi, sig)
    gk = torch.empty(K, dtype=torch.float64, device="cuda")
    ops = [torch.tensor([k], dtype=torch.int32, device="cuda") for k in range(K)]
    for k in range(K):
        pool.gradients(psi, sig, ops=ops[k], out=gk[k:k + 1])
    reps = 5
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    torch.cuda.synchronize()
    ev[0].record(st)
    for _ in range(reps):
        pool.gradients(psi, sig, out=g1)
    ev[1].record(st)
    for _ in range(reps):
        for k in range(K):
            pool.gradients(psi, sig, ops=ops[k], out=gk[k:k + 1])
    ev[2].record(st)
    torch.cuda.synchronize()
    t_one = ev[0].elapsed_time(ev[1]) / reps
    t_per = ev[1].elapsed_time(ev[2]) / reps
    out["screen"] = {"one_launch_ms": round(t_one, 4), "launch_per_op_ms": round(t_per, 3),
                     "speedup": round(t_per / t_one, 2),
                     "max_abs_diff": float(torch.max(torch.abs(g1 - gk)).item())}
    print(json.dumps(out), flush=True)


def oracle_timing(args):
    """The FP64 CPU oracle as it stands, on the host cores: full ADAPT at 12
    qubits (to convergence, at most 60 iterations), --iters iterations at 20
    qubits, and one H psi at 28 qubits; threads = the affinity set."""
    import oracle
    from oracle import adapt as oadapt
    threads = len(os.sched_getaffinity(0))
    out = {"oracle_timing": True, "threads": threads}
    for name, cap in (("h6_12q", 60), ("h10_20q", args.iters)):
        n, na, nb, seed = synth.workload(name)
        h1, h2, ec = synth.integrals(n, seed)
        ref = oracle.System(h1, h2, ec, n, na, nb)
        pool = ref.pool()
        t0 = time.perf_counter()
        rec = oadapt.run(ref, pool, max_iter=cap)
        dt = time.perf_counter() - t0
        out[name] = {"iterations": len(rec["energy"]), "s": round(dt, 2),
                     "iters_per_s": round(len(rec["energy"]) / dt, 5),
                     "final_energy": rec["energy"][-1] if rec["energy"] else None}
    n, na, nb, seed = synth.workload("h14_28q")
    h1, h2, ec = synth.integrals(n, seed)
    ref = oracle.System(h1, h2, ec, n, na, nb)
    psi = synth.random_state(ref.n_det, 99)
    t0 = time.perf_counter()
    ref.sigma(psi, threads)
    dt = time.perf_counter() - t0
    out["h14_28q_sigma"] = {"s": round(dt, 2), "n_det": ref.n_det,
                            "rows_per_s": round(ref.n_det / dt, 1)}
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if args.impl == "reference":
        return run_reference(args, rank, world)
    if args.sweeps_only:
        return sweeps_only(args)
    if args.ranker_eval:
        return ranker_eval(args)
    if args.batch:
        return batch_bench(args)
    if args.batch_rank:
        return batch_rank_bench(args)
    if args.hmat:
        return hmat_bench(args)
    if args.trajectory:
        return trajectory(args)
    if args.config2:
        return config2(args)
    if args.support_eval:
        return support_eval(args)
    if args.oracle_timing:
        return oracle_timing(args)
    if world > 1:
        import torch
        torch.distributed.init_process_group("nccl")
    r = run_ours(args, rank, world)
    if rank != 0:
        if world > 1:
            import torch
            torch.distributed.destroy_process_group()
        return
    peaks, peak_kind = load_peaks()
    N, K, J = r["N"], args.steps, args.iters_per_job
    mhz = peaks.get("sm_max_mhz", 2070.0)
    fp32_peak = 152 * 128 * 2 * mhz * 1e6 / 1e12
    fp64_peak = 152 * 2 * 2 * mhz * 1e6 / 1e12
    head = r["head"]
    flops = 2.0 * r["conn"] * N
    iters_timed = head["iterations"]
    jobs = head["jobs"]
    e_mixed = [e for _, e, _ in jobs]
    last_recs = jobs[-1][0]
    out = {
        "metric": METRIC,
        "value": round(job_throughput(world, iters_timed, head["ms"]), 4),
        "unit": "ADAPT iters/s",
        "n_gpus": world,
        "steps": K,
        "warmup": args.warmup,
        "ms_per_step": round(head["ms"] / K, 3),
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32 bulk + f64 reductions and refinement",
        "data": "synthetic (seeded integrals shaped like the H16 STO-3G chain; no PySCF)",
        "config": {"workload": f"{args.workload}: {r['n']} orbitals, {r['na']}a+{r['nb']}b, "
                               f"{N} determinants, seed {r['seed']}",
                   "step": (f"one ADAPT job: {J} iterations from Hartree-Fock (screen, select, "
                            "append, BFGS re-optimisation in float, then at most "
                            f"{REFINE_STEPS} double-precision BFGS steps refining every "
                            "iteration; the next screen on the refined double state) + the final "
                            "double-precision refinement; the Hamiltonian resident"),
                   "mode": (f"mixed precision, ranker attached (top-{args.top_m} proposals when "
                            "consulted); psi a sparse vector while its support fits N/16 (float) "
                            "or N/8 (double); float optimisation from 2^20 nonzero amplitudes, "
                            "double below (every iteration of this job); the whole pool screened "
                            "exactly while pool x support <= 5e9"),
                   "pool_ops": r["K"], "replicas": world,
                   "l2": "inputs larger than L2 (state vector 0.66 GB FP32 / 1.33 GB FP64)"},
        "mixed": {"iterations_timed": iters_timed,
                  "screens_used": screens_used(jobs),
                  "ranker_consulted_iterations": sum(
                      1 for recs, _, _ in jobs for x in recs if int(x["screen"]) in (2, 3)),
                  "final_energy_f64_per_job": e_mixed,
                  "selected": [x["selected"] for x in last_recs],
                  "energy_bulk": [x["energy"] for x in last_recs],
                  "support": [x["support"] for x in last_recs],
                  "sigma_support": [x["sigma_support"] for x in last_recs],
                  "n_evals": [x["n_evals"] for x in last_recs],
                  "refine_s_per_job": [round(t, 4) for _, _, t in jobs],
                  "c_tilde": c_tilde(last_recs)},
        "roofline": step_roofline(head["prof"], peaks, peak_kind, fp32_peak,
                                  dominant=max(head["warm"], key=lambda c: head["warm"][c]["ms"])
                                  if head["warm"] else None),
        # the timed region records per-launch events for the roofline's class
        # only; every class is recorded in the last warm-up job
        "kernel_breakdown": breakdown(head["prof"], head["ms"]),
        "kernel_breakdown_warmup_job": breakdown(head["warm"], head["warm_ms"]),
        "gpu_launches": int(head["launches"]),
        "clocks": head["clocks"],
        "build_s": round(r["t_build"], 2),
    }
    if "plain" in r:
        p = r["plain"]
        gap = e_mixed[-1] - p["energy"]
        out["plain_f64"] = {
            "mode": "plain FP64, the whole pool screened exactly every iteration (sparse path)",
            "iters_per_s": round(len(p["records"]) / (p["ms"] / 1e3), 4),
            "ms_per_job": round(p["ms"], 1), "final_energy": p["energy"],
            "selected": [x["selected"] for x in p["records"]],
            "n_evals": [x["n_evals"] for x in p["records"]],
            "kernel_breakdown": breakdown(p["prof"], p["ms"]),
            "kernel_breakdown_warmup_job": breakdown(p["warm"], p["warm_ms"])}
        out["acceptance"] = {
            "test": "mixed+ranker job faster than the plain FP64 full-screen job at equal final "
                    "energy within 1e-6 Ha",
            "final_energy_gap": gap, "equal_final_energy": abs(gap) <= 1e-6,
            "same_selections": out["plain_f64"]["selected"] == out["mixed"]["selected"],
            "speedup": round(p["ms"] / (head["ms"] / K), 3),
            "faster": p["ms"] > head["ms"] / K}
    if "accept" in r:
        a = r["accept"]
        rows = a["rows"]
        out["acceptance_long"] = {
            "test": (f"{a['iterations']} ADAPT iterations from Hartree-Fock on the same resident "
                     "Hamiltonian: mixed precision + ranker (then the final double refinement) "
                     "against plain FP64 screening the whole pool exactly every iteration; host "
                     "wall time of each leg"),
            "plain_s": a["plain_s"], "mixed_s": round(a["mixed_s"] + a["refine_s"], 3),
            "speedup": a["speedup"], "faster": a["speedup"] > 1.0,
            "final_energy_gap": a["final_gap"],
            "equal_final_energy": a["equal_final_energy_1e-6"],
            "same_selections": a["same_selections"],
            "ranker_consulted_iterations": a["ranker_consulted_iterations"],
            "support": [x["support"] for x in rows],
            "screen_mixed": [x["screen_mixed"] for x in rows],
            "mixed_f32_err": [x["mixed_f32_err"] for x in rows],
            "t_plain_s": [x["t_plain_s"] for x in rows],
            "t_mixed_s": [x["t_mixed_s"] for x in rows]}
    if "hpsi_ms_f64" in r:
        def hp(ms, s):
            gbs = 2.0 * N * s / (ms / 1e3) / 1e9
            return {"ms": round(ms, 3), "gbs": round(gbs, 3),
                    "hbm_frac": round(gbs / peaks["hbm_gbs"], 6),
                    "tflops": round(flops / (ms / 1e3) / 1e12, 4)}
        cpl_units = (r["na"] * (r["n"] - r["na"]) + 1) * (r["nb"] * (r["n"] - r["nb"]) + 1)
        cflops = 2.0 * cpl_units * N
        out["hpsi_matrix_free"] = {
            "f64": hp(r["hpsi_ms_f64"], 8), "f32": hp(r["hpsi_ms_f32"], 4),
            "algorithmic_bytes": "2 * N_det * sizeof(amplitude)",
            "connections_per_det": r["conn"], "state": "dense seeded random state",
            "fp64_frac_of_derived_fp64_peak": round(flops / (r["hpsi_ms_f64"] / 1e3) / 1e12 /
                                                    fp64_peak, 4),
            "fp32_frac_of_derived_fp32_peak": round(flops / (r["hpsi_ms_f32"] / 1e3) / 1e12 /
                                                    fp32_peak, 4),
            "coupling_ms": {"f64": round(r["cpl_ms_f64"], 3), "f32": round(r["cpl_ms_f32"], 3)},
            "coupling_useful_tflops_f32": round(cflops / (r["cpl_ms_f32"] / 1e3) / 1e12, 3),
            "screen_ms": {"f64": round(r["screen_ms_f64"], 3), "f32": round(r["screen_ms_f32"], 3)}}
    if "explicit_h" in r:
        xh = r["explicit_h"]
        out["hpsi_explicit"] = xh
        tr, tw = traffic_for("hmat")
        out["hpsi_explicit"]["roofline_f32"] = {
            "bound": "hbm", "kernel": "k_hmat_spmv<float>",
            "achieved": xh["f32"]["gbs"], "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": xh["f32"]["frac_of_hbm"],
            "traffic": tr, "traffic_workload": tw,
            "peak_kind": f"{peak_kind} copy bandwidth (MEASURED_PEAKS.json hbm_gbs)"}
    if "e2e" in r:
        e = r["e2e"]
        out["e2e"] = {"value": round(job_throughput(world, e["iterations"], e["ms"]), 4),
                      "unit": "ADAPT iters/s", "h2d_bytes_per_step": int(e["h2d"]),
                      "d2h_bytes_per_step": int(e["d2h"]),
                      "path": "public API from host integrals: hy_build_hamiltonian, "
                              "hy_pool_create, hy_adapt_create, 10 x hy_adapt_step, "
                              "hy_adapt_refine, hy_adapt_ansatz readback, destroy",
                      "final_energy_f64_per_step": e["energies"]}
    if not args.no_cpu_baseline and world == 1 and "plain" in r:
        recs = [(x["iter"] + 1, x["n_evals"]) for x in r["plain"]["records"]]
        n, na, nb, seed = r["n"], r["na"], r["nb"], r["seed"]
        del r, head
        tot, thr, spent, sample = oracle_job_estimate(n, na, nb, seed, args.cpu_budget, recs)
        out["cpu_baseline"] = {"value": len(recs) / tot, "unit": "ADAPT iters/s", "cores": thr,
                               "kind": "oracle", "sample": sample}
    print(json.dumps(out), flush=True)
    if world > 1:
        import torch
        torch.distributed.destroy_process_group()


def run_reference(args, rank, world):
    """The oracle as it stands, timed on the host cores.  Each step is a
    bounded sample (--cpu-budget seconds) of the plain FP64 job's work --
    sigma on sampled rows, a few operators' gradients, one exp(theta A) --
    and the line's value is the job's iterations over the oracle time the
    samples extrapolate to (10 iterations, 10 evaluations each at the
    ansatz lengths of a job: the oracle has no sparse path, every
    evaluation is a full sweep).  ms_per_step is the sample's own time."""
    if rank != 0:
        return
    import oracle
    n, na, nb, seed = synth.workload(args.workload)
    h1, h2, ec = synth.integrals(n, seed)
    n_det = oracle.System(h1, h2, ec, n, na, nb).n_det
    state = synth.random_state(n_det, 99)
    J = args.iters_per_job
    recs = [(l + 1, 10) for l in range(J)]
    per = max(2.0, min(args.cpu_budget, 150.0 / max(1, args.steps + args.warmup)))
    for _ in range(args.warmup):
        oracle_job_estimate(n, na, nb, seed, per, recs, state)
    tots, spent = [], []
    for _ in range(args.steps):
        tot, thr, sp, sample = oracle_job_estimate(n, na, nb, seed, per, recs, state)
        tots.append(tot)
        spent.append(sp)
    v = J / statistics.mean(tots)
    out = {"metric": METRIC, "value": v, "unit": "ADAPT iters/s", "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": 1e3 * statistics.mean(spent),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "f64", "data": "synthetic", "impl": "reference",
           "config": {"workload": f"{args.workload}: {n} orbitals, {na}a+{nb}b, "
                                  f"{n_det} determinants, seed {seed}",
                      "mode": "FP64 CPU oracle, plain full screen",
                      "step": f"a bounded sample ({per:.1f} s budget) of the oracle's work for "
                              f"one {J}-iteration job, extrapolated to the whole job"},
           "cpu_baseline": {"value": v, "unit": "ADAPT iters/s", "cores": thr,
                            "kind": "oracle", "sample": sample},
           "e2e": {"value": v, "unit": "ADAPT iters/s", "h2d_bytes_per_step": 0,
                   "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    main()
