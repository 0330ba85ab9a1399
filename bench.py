#!/usr/bin/env python
"""Benchmark: AD-PRD operator applies/s on the Mg II h&k-like workload
(70 heights x 64 directions x 200 wavelengths, N = 3.58e6 unknowns, FP32),
plus one preconditioned GMRES solve, as one JSON line on stdout.

A step is one operator apply y = (Id - Lambda Sigma) x (all stages S1-S8 of
the hot path) on inputs resident in HBM.  N > 1 GPUs (torchrun, one rank per
GPU) run independent instances (weak scaling, no data-path collective).

--impl reference times the FP64 CPU oracle on all host cores on bounded
samples of the same workload (one whole scattering-angle class at one height
plus formal-solution rays per step), scaled to one full apply.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)
# the CPU oracle runs one process per host core: keep numpy's BLAS single-threaded
for _v in ("OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import numpy as np   # noqa: E402

METRIC = "AD-PRD operator applies/s, GMRES solve s at 1e-5 rel err; % of roofline"
UNIT = "applies/s"
PEAKS_FALLBACK = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}
# layout tag of the contraction whose DRAM traffic profiles/traffic.json records;
# the traffic figure is reported only while it matches the kernel that runs
KERNEL_LAYOUT = "f32-v7"
# what each value of --contraction multiplies on the tensor cores
PRODUCTS = {"tf32x3": "bf16 planes x6, FP32 level", "bf16x3": "bf16 planes x3", "bf16x2": "bf16 hi plane x2"}
N_PRODUCTS = {"tf32x3": 6.0, "bf16x3": 3.0, "bf16x2": 2.0}


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return PEAKS_FALLBACK, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu):
        self.gpu = gpu
        self.rows = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([s.strip() for s in line.split(",")])

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        sm = [float(r[1]) for r in self.rows if len(r) > 8 and r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if len(r) > 8 and r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows if len(r) > 8 for i in range(4)
                          if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(sm)}


# ---------------------------------------------------------------- CPU baseline (oracle)
# A real partial apply of the FP64 oracle, spread over the host cores: one
# whole scattering-angle class at one height (its R_II tiles computed once, as
# the oracle's full apply shares them per (height, class), then the blocks of
# every direction pair of the class against all frequencies and Stokes
# parameters), plus formal solutions along sampled rays.  The per-apply time is
# scaled from the two phases: tiles x (heights x classes), blocks x (heights x
# direction pairs), rays x (directions x frequencies).
_W = {}


def _w_init(cfg, seed):
    for v in ("OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS", "OMP_NUM_THREADS"):
        os.environ[v] = "1"
    from oracle.problem import Problem
    P = Problem(cfg, normalise=False)
    _W["P"] = P
    _W["x"] = np.random.default_rng(seed).uniform(0.1, 1.0, P.shape())


def _w_meta():
    P = _W["P"]
    return dict(nz=P.nz, nO=P.nO, nN=P.nN, cls=P.cls, thetas=P.thetas, nu=P.nu_states, nl=P.nl_states)


def _w_tiles(iz, c, combos):
    """R_II tiles of class c at height iz for the (k_u', k_l, k_l') combinations."""
    P = _W["P"]
    P._tiles.clear()
    s = P.shift[iz]
    for kv, kl, klp in combos:
        P.tile(iz, P.thetas[c], s[kv, kl], s[kv, klp])
    return dict(P._tiles)


def _w_blocks(iz, pairs, tiles):
    """Comoving emissivity contributions of the direction pairs (o, o')."""
    P = _W["P"]
    P._tiles.clear()
    P._tiles.update(tiles)
    P._r3.clear()
    x = _W["x"]
    sb = np.zeros((P.nO, P.nN, 4))
    for o, op in pairs:
        blk = P.block(iz, o, op).reshape(P.nN * 4, P.nN * 4)
        sb[o] += (blk @ (P.interp_in(iz, op) @ x[iz, op]).ravel()).reshape(P.nN, 4)
    return sb


def _w_rays(rays):
    P = _W["P"]
    return sum(float(P.lambda_ray(_W["x"], o, n)[-1, 0]) for o, n in rays)


class OraclePool:
    """The oracle set up once in `cores` spawned worker processes (set-up not
    timed); `sample` times one partial apply and scales it to a full apply."""

    def __init__(self, cfg, cores=None, seed=5):
        from concurrent.futures import ProcessPoolExecutor
        from multiprocessing import get_context
        self.cores = cores or len(os.sched_getaffinity(0))
        self.ex = ProcessPoolExecutor(max_workers=self.cores, mp_context=get_context("spawn"),
                                      initializer=_w_init, initargs=(cfg, seed))
        metas = list(self.ex.map(_w_meta_wait, range(self.cores)))   # every worker set up
        self.m = metas[0]

    def sample(self, step, warm=False):
        """Warm-up samples take a class with the fewest direction pairs; timed
        samples a class with the most."""
        m = self.m
        nz, nO, nN, cls = m["nz"], m["nO"], m["nN"], m["cls"]
        counts = np.bincount(cls.ravel(), minlength=len(m["thetas"]))
        inner = [c for c in range(len(counts)) if counts[c] > 0 and 0.0 < m["thetas"][c] < np.pi]
        want = min(counts[c] for c in inner) if warm else max(counts[c] for c in inner)
        pick = [c for c in inner if counts[c] == want]
        c = pick[(5 * step) % len(pick)]
        iz = (7 * step + nz // 2) % nz
        combos = [(kv, kl, klp) for kv in range(m["nu"]) for kl in range(m["nl"]) for klp in range(m["nl"])]
        pairs = [tuple(p) for p in np.argwhere(cls == c)]
        n_rays = self.cores if warm else 4 * self.cores
        rays = [((3 * r + step) % nO, (7 * r + step) % nN) for r in range(n_rays)]
        k = self.cores
        t0 = time.perf_counter()
        parts = list(self.ex.map(_w_tiles, [iz] * k, [c] * k, [combos[i::k] for i in range(k)]))
        tiles = {}
        for d in parts:
            tiles.update(d)
        t1 = time.perf_counter()
        sb = sum(self.ex.map(_w_blocks, [iz] * k, [pairs[i::k] for i in range(k)], [tiles] * k))
        t2 = time.perf_counter()
        list(self.ex.map(_w_rays, [rays[i::k] for i in range(k)]))
        t3 = time.perf_counter()
        n_cls = int(np.count_nonzero(counts))
        per_apply = nz * (n_cls * (t1 - t0) + nO * nO * (t2 - t1) / len(pairs)) + nO * nN * (t3 - t2) / n_rays
        desc = (f"FP64 oracle on {self.cores} host processes: one scattering-angle class at one height "
                f"({len(pairs)} direction pairs x {nN} frequencies x 4 Stokes, its {len(combos)} R_II tiles "
                f"computed once) and {n_rays} formal-solution rays, scaled by heights x classes (tiles), "
                f"heights x direction pairs (blocks: {nz}x{nO * nO}) and rays ({nO * nN}); "
                f"sample {t3 - t0:.1f} s")
        return per_apply, desc, float(np.abs(sb).sum())

    def close(self):
        self.ex.shutdown()


def _w_meta_wait(_):
    return _w_meta()


def useful_contraction_flops(P, n_t):
    """Useful work of one R_II contraction: F3 = 16 N_r n_t N_nu^2 C, C the
    number of distinct (scattering angle, incident direction) combinations
    with Theta != 0 (the product integration of every incident node against
    every output node once per angle class, complex kernel x 4 real Stokes
    parameters), n_t the transition triples (k_u, k_l, k_l')."""
    nv = np.stack([np.sqrt(1 - P.mu ** 2) * np.cos(P.chi), np.sqrt(1 - P.mu ** 2) * np.sin(P.chi), P.mu], -1)
    th = 2.0 * np.arctan2(np.linalg.norm(nv[:, None] - nv[None], axis=-1),
                          np.linalg.norm(nv[:, None] + nv[None], axis=-1))
    order = np.argsort(th, axis=None)
    vals = th.ravel()[order]
    cls = np.empty(vals.size, dtype=np.int64)
    cls[order] = np.concatenate([[0], np.cumsum(np.diff(vals) > 1e-10)])
    cls = cls.reshape(th.shape)
    inc = np.broadcast_to(np.arange(P.nO)[None, :], th.shape)
    C = len({(int(c), int(o)) for c, o, t in zip(cls.ravel(), inc.ravel(), th.ravel()) if t > 1e-10})
    return 16.0 * P.nz * n_t * P.nN ** 2 * C, C


def batch_throughput(local, n=32):
    """S12 beside the headline: n ragged Mg II-like instances (6-10 heights,
    varied frequency grids and fields, FP32), solved to tol 1e-8 once as one
    prd_solve_batch (lockstep rounds, one parent-graph launch per iteration)
    and once one after another with prd_solve; solves/s of each (after one
    untimed batch that captures every instance's Arnoldi step)."""
    import torch
    from paper_2505_20968_gb300 import inputs
    from paper_2505_20968_gb300.binding import PRD, solve_batch
    cfgs = [inputs.mgii(n_z=6 + (i % 5), n_core_each=5 + (i % 3), n_wing=4 + (i % 2), n_mu_half=2, n_chi=4,
                        seed=500 + i) for i in range(n)]
    Ps = [PRD(c, device=local) for c in cfgs]
    unknowns = sum(P.n for P in Ps)
    solve_batch(Ps, tol=1e-8, max_iter=600, restart=60)
    launches0 = [P.graph_launches() for P in Ps]
    torch.cuda.synchronize()
    t0 = time.time()
    _, infos = solve_batch(Ps, tol=1e-8, max_iter=600, restart=60)
    torch.cuda.synchronize()
    tb = time.time() - t0
    rounds = sum(P.graph_launches() - k for P, k in zip(Ps, launches0))
    t0 = time.time()
    for P in Ps:
        P.solve(tol=1e-8, max_iter=600, restart=60)
    torch.cuda.synchronize()
    ts = time.time() - t0
    for P in Ps:
        P.close()
    return {"instances": n, "unknowns": unknowns, "tol": 1e-8, "precision": "fp32",
            "batch_solves_per_s": n / tb, "sequential_solves_per_s": n / ts, "batch_seconds": tb,
            "sequential_seconds": ts, "applies": sum(i["iters"] for i in infos),
            "instance_steps_in_graph_rounds": rounds, "all_converged": all(i["rc"] == 0 for i in infos)}


def max_over_ranks(ms, dist, device):
    """The job's time: the largest per-rank time over the ranks (any backend)."""
    if dist is None:
        return ms
    import torch
    t = torch.tensor([ms], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(world, ms):
    """Whole-job applies/s: every rank applies its own instance once per step."""
    return world * 1e3 / ms


def run_reference(args, cfg, workload):
    pool = OraclePool(cfg)
    per = []
    desc = ""
    for step in range(args.warmup + args.steps):
        t, desc, _ = pool.sample(step, warm=step < args.warmup)
        if step >= args.warmup:
            per.append(t)
    pool.close()
    value = 1.0 / statistics.median(per)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 / value,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": workload,
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": pool.cores, "kind": "oracle", "sample": desc},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-solve", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--solve-tol", type=float, default=1e-10,
                    help="GMRES tol; 1e-10 is the largest meeting 1e-5 on emergent I in the Mg II parity case")
    ap.add_argument("--contraction", default="tf32x3", choices=["tf32x3", "bf16x3", "bf16x2"],
                    help="split products of the timed R_II contraction (tf32x3: FP32-level accuracy)")
    ap.add_argument("--workload", default="mgii", choices=["mgii", "mgii_small", "lambda_wide"],
                    help="mgii_small (8 heights) is only for ncu captures of single kernels; lambda_wide "
                         "(two-level, angle-averaged, 300 heights x 128 directions x 200 frequencies) sizes "
                         "the formal-solution sweep beyond L2 for its HBM capture")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)

    from paper_2505_20968_gb300 import inputs
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.workload == "lambda_wide":
        cfg = inputs.twolevel_slab(n_z=300, n_x=200, n_mu_half=8, n_chi=8, seed=2 + rank)
        cfg["quad"]["mode"] = inputs.MODE_AA
        cfg["precision"] = "fp32"
    else:
        cfg = inputs.mgii(seed=2 + rank) if args.workload == "mgii" else inputs.mgii(n_z=8, seed=2 + rank)
    nz, nnu = len(cfg["atm"]["z_km"]), len(cfg["quad"]["grid"])
    nmu, nchi = cfg["quad"]["n_mu_half"], cfg["quad"]["n_chi"]
    atom = "two-term Mg II h&k" if args.workload != "lambda_wide" else "two-level J 0->1 angle-averaged"
    workload = {"workload": f"{'mgii_hk_like' if args.workload != 'lambda_wide' else 'lambda_wide'}: {atom}, "
                            f"{nz} heights, {nnu} {'wavelengths' if args.workload != 'lambda_wide' else 'frequencies'}, "
                            f"{nmu}+{nmu} GL mu x {nchi} chi ({2 * nmu * nchi} directions)"
                            f"{', B<=100 G, |v|<=5 km/s' if args.workload != 'lambda_wide' else ''}, "
                            f"N={4 * nz * nnu * 2 * nmu * nchi:,}",
                "precision": "fp32 tiles/vectors, fp64 reductions", "parallelism": f"{world} independent instances",
                "l2": "inputs larger than L2 (R_II tiles ~40 GB streamed per apply)"}
    if args.impl == "reference":
        if rank == 0:
            run_reference(args, cfg, workload)
        return

    import torch
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2505_20968_gb300.binding import PRD

    t0 = time.time()
    # bf16x3: a PRD_FP32_BF16X3 context, whose tiles are stored as bf16 hi/lo planes
    P = PRD(cfg, device=local, precision={"bf16x3": "fp32_bf16x3", "bf16x2": "fp32_bf16x2"}.get(args.contraction))
    torch.cuda.synchronize()
    setup_s = time.time() - t0
    g = torch.Generator(device="cuda").manual_seed(1234 + rank)
    x = torch.rand(P.shape, device="cuda", dtype=P.dtype, generator=g)
    x[..., 1:] *= 0.05
    y = P.empty()
    autotune = None
    if P.prec == 1:
        # the contraction's tile-ring depth, measured (tune.py)
        from paper_2505_20968_gb300.tune import tune_tile_stages
        best, res = tune_tile_stages(P)
        autotune = {"tile_stages": best, "ms_per_apply": res}
    for _ in range(args.warmup):
        P.apply_operator(x, y)
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        P.apply_operator(x, y)
    e1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    clk = clocks.stop()
    ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, dist, "cuda")
    value = job_value(world, ms)

    # end to end through the public API with host buffers (pinned), copies timed
    xh = x.cpu().pin_memory()
    yh = torch.empty_like(xh).pin_memory()
    xd = torch.empty_like(x)
    for _ in range(2):
        xd.copy_(xh, non_blocking=True)
        P.apply_operator(xd, y)
        yh.copy_(y, non_blocking=True)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(args.steps):
        xd.copy_(xh, non_blocking=True)
        P.apply_operator(xd, y)
        yh.copy_(y, non_blocking=True)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_e2e = max_over_ranks(e0.elapsed_time(e1) / args.steps, dist, "cuda")
    nbytes = x.numel() * x.element_size()

    # per-stage durations (CUDA events on the library stream) for the roofline
    P.set_profiling(True)
    for _ in range(3):
        P.apply_operator(x, y)
    st = P.stage_times()
    P.set_profiling(False)
    r2_ms = st["S3_R2_contraction"][0] / max(st["S3_R2_contraction"][1], 1)
    flops, tile_bytes = P.contraction_work()
    # transition triples (k_u, k_l, k_l'): 18 for the two-term S_1/2 -> P_1/2,3/2 atom, 3 for J 0 -> 1
    n_t = 18 if cfg["atom"]["twoS"] == 1 else 3
    useful, n_theta_omega = useful_contraction_flops(P, n_t=n_t)
    peaks, src = _peaks()
    # The contraction runs six products of bf16 planes per FP32-level product (three or two for
    # the bf16 precisions) and streams the tiles once; the longer of the two at the measured bf16 and
    # HBM rates bounds it (FP32: the products).  `issued` counts the products over the stored tiles
    # (J-level means plus per-triple deviations, 20 per angle class), `useful_tflops` the useful
    # work F3 and `hbm` the tile bytes.
    achieved_tf = useful / (r2_ms * 1e-3) / 1e12
    issued_tf = N_PRODUCTS[args.contraction] * flops / (r2_ms * 1e-3) / 1e12
    achieved_gbs = tile_bytes / (r2_ms * 1e-3) / 1e9
    kernel = "r2_f32_kernel" if args.contraction == "tf32x3" else "r2_tc_kernel"
    tensor_bound = issued_tf / peaks["bf16_tflops"] > achieved_gbs / peaks["hbm_gbs"]
    traffic = None
    try:
        with open(os.path.join(ROOT, "profiles", "traffic.json")) as f:
            tr = json.load(f)
        if tr.get("kernel") == kernel and tr.get("workload") == "mgii" and tr.get("layout") == KERNEL_LAYOUT:
            traffic = tr.get("dram_bytes_per_launch")
    except (OSError, ValueError):
        pass
    bound = ({"bound": "tensor", "achieved": issued_tf, "peak": peaks["bf16_tflops"], "unit": "TFLOP/s issued",
              "frac": issued_tf / peaks["bf16_tflops"]} if tensor_bound else
             {"bound": "hbm", "achieved": achieved_gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
              "frac": achieved_gbs / peaks["hbm_gbs"]})
    roofline = {**bound, "kernel": f"{kernel} (S3+S4 R_II contraction, tcgen05, {PRODUCTS[args.contraction]})",
                "useful_tflops": achieved_tf, "useful_frac": achieved_tf / peaks["bf16_tflops"],
                "issued": issued_tf, "issued_frac": issued_tf / peaks["bf16_tflops"],
                "peak_source": src, "traffic": traffic,
                "algorithmic_flops_per_launch": useful, "issued_flops_per_launch": N_PRODUCTS[args.contraction] * flops,
                "useful_flops_formula": f"16 N_r n_t N_nu^2 C = 16 x {P.nz} x {n_t} x {P.nN}^2 x {n_theta_omega}",
                "algorithmic_bytes_per_launch": tile_bytes,
                "hbm": {"achieved": achieved_gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                        "frac": achieved_gbs / peaks["hbm_gbs"]},
                "launch_ms": r2_ms, "stage_ms": {k: v[0] / max(v[1], 1) for k, v in st.items()}}
    # S7+S8 formal solution: 64 algorithmic bytes per (z, Omega, nu) per sweep in FP32
    # (eps 16 B, the I read of y = x - Lambda eps 16 B, K'/eta_1 and DELO weights 28 B,
    # dtau 4 B); the Mg II sweep (57 MB) stays in L2, lambda_wide's (629 MB) does not
    delo_ms = st["S7_delo"][0] / max(st["S7_delo"][1], 1)
    delo_bytes = 64.0 * P.nz * P.nO * P.nN
    roofline["formal_solver"] = {"kernel": "delo_kernel (S7+S8)", "bytes_per_launch": delo_bytes,
                                 "launch_ms": delo_ms, "achieved_gbs": delo_bytes / (delo_ms * 1e-3) / 1e9,
                                 "peak_gbs": peaks["hbm_gbs"],
                                 "frac": delo_bytes / (delo_ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
                                 "l2_resident": delo_bytes < 129e6}

    solve = None
    if not args.no_solve:
        torch.cuda.synchronize()
        t0 = time.time()
        sol, info = P.solve(tol=args.solve_tol, max_iter=600, restart=200, check=False)
        torch.cuda.synchronize()
        solve = {"seconds": time.time() - t0, "tol": args.solve_tol, "applies": info["iters"],
                 "true_rel_res": info["true_rel_res"], "rc": info["rc"], "setup_seconds": setup_s}

    # the split-BF16 contraction (BF16x3): a PRD_FP32_BF16X3 context on the same
    # atmosphere (set up after this one is released: both would not fit beside
    # their FP64 residual copies), its contraction time and its refined solve at
    # the same tolerance (the FP64 residuals fix the accuracy)
    modes = {}
    if cfg.get("precision", "fp32") == "fp32" and not args.no_solve and args.contraction == "tf32x3":
        modes["tf32x3"] = {"contraction_ms": r2_ms, "useful_tflops": achieved_tf,
                           "solve_seconds": solve["seconds"], "solve_applies": solve["applies"]}
        P.close()
        del P
        torch.cuda.synchronize()
        t0 = time.time()
        Pb = PRD(cfg, device=local, precision="fp32_bf16x3")
        torch.cuda.synchronize()
        setup_b = time.time() - t0
        for _ in range(2):
            Pb.apply_operator(x, y)
        Pb.set_profiling(True)
        for _ in range(3):
            Pb.apply_operator(x, y)
        st16 = Pb.stage_times()
        Pb.set_profiling(False)
        b16_ms = st16["S3_R2_contraction"][0] / max(st16["S3_R2_contraction"][1], 1)
        torch.cuda.synchronize()
        t0 = time.time()
        sol16, info16 = Pb.solve(tol=args.solve_tol, max_iter=900, restart=200, check=False)
        torch.cuda.synchronize()
        modes["bf16x3"] = {"contraction_ms": b16_ms, "useful_tflops": useful / (b16_ms * 1e-3) / 1e12,
                           "issued_frac_of_bf16_peak": N_PRODUCTS["bf16x3"] * flops / (b16_ms * 1e-3) / 1e12 / peaks["bf16_tflops"],
                           "hbm_frac": tile_bytes / (b16_ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
                           "solve_seconds": time.time() - t0, "solve_applies": info16["iters"],
                           "solve_true_rel_res": info16["true_rel_res"], "rc": info16["rc"],
                           "setup_seconds": setup_b, "tiles": "bf16 hi/lo planes (PRD_FP32_BF16X3)"}
        Pb.close()
        del Pb
        # BF16x2: the hi plane alone (half the tile bytes), two products
        torch.cuda.synchronize()
        t0 = time.time()
        Pc = PRD(cfg, device=local, precision="fp32_bf16x2")
        torch.cuda.synchronize()
        setup_c = time.time() - t0
        for _ in range(2):
            Pc.apply_operator(x, y)
        Pc.set_profiling(True)
        for _ in range(3):
            Pc.apply_operator(x, y)
        stc = Pc.stage_times()
        Pc.set_profiling(False)
        c2_ms = stc["S3_R2_contraction"][0] / max(stc["S3_R2_contraction"][1], 1)
        # no solve: with Sigma good to ~1e-3 the refinement stalls on this problem (PRD_E_NOCONV)
        modes["bf16x2"] = {"contraction_ms": c2_ms, "useful_tflops": useful / (c2_ms * 1e-3) / 1e12,
                           "hbm_frac": tile_bytes / 2 / (c2_ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
                           "setup_seconds": setup_c, "tiles": "bf16 hi plane (PRD_FP32_BF16X2)",
                           "solve": "not run: Sigma to ~1e-3 stalls the refinement (tests/test_gpu_parity.py)"}
        Pc.close()

    batch = None
    if rank == 0 and not args.no_solve and args.workload == "mgii":
        batch = batch_throughput(local)

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        pool = OraclePool(cfg)
        per, desc, _ = pool.sample(0)
        pool.close()
        cpu = {"value": 1.0 / per, "unit": UNIT, "cores": pool.cores, "kind": "oracle", "sample": desc}

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": workload,
                "clocks": clk,
                "e2e": {"value": job_value(world, ms_e2e), "unit": UNIT, "h2d_bytes_per_step": nbytes,
                        "d2h_bytes_per_step": nbytes},
                "gpu_launches": 6 * args.steps, "roofline": roofline, "cpu_baseline": cpu, "solve": solve,
                "contraction_modes": modes, "autotune": autotune, "batch": batch}
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
