"""A fixed small case of the streaming kernels to run under ncu, and the summary
of what ncu measured on it.

    python -m paper_1410_3464_gb300.profile_case run [--warm 2] [--steps 3] [--fp64]
        porous discs 1024x512 (seed 1), FP32 (or FP64), three transported species:
        --warm then --steps single steps.  The working set (about 160 MB) is larger
        than the 129 MB L2, so DRAM counters mean something, and small enough for
        a multi-pass ncu capture.
    python -m paper_1410_3464_gb300.profile_case run --batch 32 [--warm 2] [--steps 3]
        the same for a batch of 32 members of the 256-member benchmark trace
        (every 8th request: sides 128-1024, about 6 M nodes, 2 GB of device
        state).  Its DRAM bytes scale to the 256-member batch by the ratio of the
        algorithmic bytes.
    python -m paper_1410_3464_gb300.profile_case summarize LAUNCHES.csv OUT.json [--batch 32] [--fp64]
        reads the ncu --csv --print-units base launch list of the run above
        (kernels matching k_pot|k_move, metrics dram__bytes_read.sum,
        dram__bytes_write.sum, gpu__time_duration.sum; FP64 also the DFMA, DADD
        and DMUL thread counts and the FP64 pipe's active share) and writes the
        means per kernel and step of the launches after the warm-up, keyed by the
        hash of the device sources they were built from.
"""
from __future__ import annotations

import argparse
import csv
import hashlib
import json
import os
import statistics
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNELS = ("k_pot", "k_move")
WORKLOAD = "porous discs 1024x512 (seed 1), FP32, 3 species"


def kernel_source_hash(precision="fp32"):
    """Hash of the device sources the streaming kernels of a precision are compiled from."""
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_1410_3464_gb300", "csrc")
    unit = {"fp32": "kernels_f32.cu", "fp64": "kernels_f64.cu"}[precision]
    for f in ("device.cuh", "step.cuh", "kernels_impl.cuh", unit):
        h.update(f.encode())
        h.update(open(os.path.join(d, f), "rb").read())
    return h.hexdigest()[:16]


def batch_members(count):
    """Every (256 / count)-th request of the 256-member benchmark trace (seed 4)."""
    from . import inputs
    reqs = inputs.request_stream(256, seed=4, size_range=(128, 1024), budget_range=(1000, 10000),
                                 rate_range=(1e-6, 1e-1), porosity_range=(0.4, 0.8), stop_fraction=0.0)
    return reqs[::max(1, 256 // count)][:count], reqs


def algorithmic_bytes(types, ns):
    """FP32 bytes of one step of the streaming kernels (fluid x 144 + liquid x 40 ns + 2 per node)."""
    return int((types <= 1).sum()) * 144 + int((types == 0).sum()) * 40 * ns + 2 * types.size


def run_batch(args):
    from . import inputs, pslbm
    members, _ = batch_members(args.batch)
    scenes = [inputs.request_scene(r) for r in members]
    sims = [pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"],
                             precision=pslbm.FP32) for sc in scenes]
    b = pslbm.Batch(sims)
    for _ in range(args.warm + args.steps):
        b.step(1)
    b.sync()
    b.close()
    alg = sum(algorithmic_bytes(s.read(pslbm.F_TYPE)["type"], s.ns) for s in sims)
    print(json.dumps({"algorithmic_bytes_per_launch": alg, "members": len(sims),
                      "nodes": sum(s.nx * s.ny for s in sims)}), flush=True)
    for s in sims:
        s.close()
    return 0


def run(args):
    if args.batch:
        return run_batch(args)
    from . import inputs, pslbm
    sc = inputs.porous_discs(nx=1024, ny=512, seed=1)
    prec = pslbm.FP64 if args.fp64 else pslbm.FP32
    with pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"],
                          precision=prec) as sim:
        for _ in range(args.warm + args.steps):
            sim.step(1)
        sim.sync()
        print(json.dumps({"algorithmic_bytes_per_launch": algorithmic_bytes(sim.read(pslbm.F_TYPE)["type"], sim.ns)}),
              flush=True)
    return 0


_SCALE = {"byte": 1.0, "kbyte": 1e3, "mbyte": 1e6, "gbyte": 1e9,
          "nsecond": 1e-9, "usecond": 1e-6, "msecond": 1e-3, "second": 1.0,
          "ns": 1e-9, "us": 1e-6, "ms": 1e-3, "s": 1.0}


def read_launches(path):
    """{launch id: (kernel name, {metric: value in bytes or seconds})} of an ncu csv."""
    rows = {}
    with open(path, newline="") as fh:
        lines = [ln for ln in fh if ln.startswith('"')]
    for r in csv.DictReader(lines):
        if "Metric Name" not in r or r.get("ID") in (None, ""):
            continue
        lid = int(r["ID"])
        name, metrics = rows.setdefault(lid, (r["Kernel Name"], {}))
        v = float(r["Metric Value"].replace(",", ""))
        metrics[r["Metric Name"]] = v * _SCALE.get(r.get("Metric Unit", "").strip().lower(), 1.0)
    return rows


def summarize(args):
    rows = read_launches(args.csv)
    prec = "fp64" if args.fp64 else "fp32"
    per = {k: [rows[i][1] for i in sorted(rows) if k in rows[i][0]][args.warm:] for k in KERNELS}
    if any(len(v) != args.steps for v in per.values()):
        raise SystemExit(f"expected {args.warm} + {args.steps} launches of each of {KERNELS}")

    def mean(k, m):
        return statistics.mean(x[m] for x in per[k])

    out = {"kernel": "k_pot + k_move, 3 species, " + ("batch" if args.batch else "single simulation"),
           "workload": (f"{args.batch} members of the 256-member benchmark batch (every {256 // args.batch}th "
                        "request), FP32, 3 species" if args.batch else WORKLOAD.replace("FP32", prec.upper())),
           "source_hash": kernel_source_hash(prec),
           "dram_bytes_read": {k: int(mean(k, "dram__bytes_read.sum")) for k in KERNELS},
           "dram_bytes_write": {k: int(mean(k, "dram__bytes_write.sum")) for k in KERNELS},
           "ncu_duration_us": {k: round(mean(k, "gpu__time_duration.sum") * 1e6, 2) for k in KERNELS},
           "note": ("ncu replays each launch with caches flushed; means over the "
                    f"{args.steps} steps after {args.warm} warm-up steps; writes still "
                    "resident in L2 at kernel end are not counted"),
           "command": args.command}
    out["traffic_per_step"] = sum(out["dram_bytes_read"].values()) + sum(out["dram_bytes_write"].values())
    if args.fp64:
        # 2 per DFMA, 1 per DADD and DMUL, over the executed thread instructions
        op = "sm__sass_thread_inst_executed_op_{}_pred_on.sum"
        out["fp64_flops_per_step"] = int(sum(2 * mean(k, op.format("dfma")) + mean(k, op.format("dadd")) +
                                             mean(k, op.format("dmul")) for k in KERNELS))
        out["fp64_pipe_active_pct"] = {
            k: round(mean(k, "sm__pipe_fp64_cycles_active.avg.pct_of_peak_sustained_active"), 2) for k in KERNELS}
    if args.batch:
        # the traffic per node does not depend on which members are in the batch
        out["algorithmic_bytes_small"], out["algorithmic_bytes_full"] = args.alg_small, args.alg_full
        out["traffic_measured_small"] = out["traffic_per_step"]
        out["traffic_per_step"] = int(out["traffic_per_step"] * args.alg_full / args.alg_small)
    with open(args.out, "w") as fh:
        json.dump(out, fh, indent=1)
        fh.write("\n")
    print(out["traffic_per_step"])
    return 0


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    sub = ap.add_subparsers(dest="cmd", required=True)
    for name in ("run", "summarize"):
        p = sub.add_parser(name)
        p.add_argument("--warm", type=int, default=2)
        p.add_argument("--steps", type=int, default=3)
        p.add_argument("--batch", type=int, default=0, help="members of the benchmark batch (0: one lattice)")
        p.add_argument("--fp64", action="store_true", help="the FP64 path")
        if name == "summarize":
            p.add_argument("--alg-small", type=int, default=0, help="algorithmic bytes per launch of the run")
            p.add_argument("--alg-full", type=int, default=0, help="algorithmic bytes per launch of the full batch")
            p.add_argument("csv")
            p.add_argument("out")
            p.add_argument("--command", default="", help="the ncu command line that made the csv")
    args = ap.parse_args(argv)
    return run(args) if args.cmd == "run" else summarize(args)


if __name__ == "__main__":
    sys.exit(main())
