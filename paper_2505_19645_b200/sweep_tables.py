"""Turns the "sweeps" of a bench.py record into one table per shape / variant.

    python -m paper_2505_19645_b200.sweep_tables RESULT.json [OUT_DIR]

RESULT.json is the file `bench.py --record` wrote (its last line is read).  Writes
OUT_DIR/sweep_<key>.md (default OUT_DIR: profiles/ beside the package) with, per (B, gamma)
point, the layer time, tokens/s, the roofline fraction, the verify-cost ratio
T(B,gamma)/T(B,0) of Sec. 3.1 and the activation statistics of Sec. 3.2 / 3.3.
"""
from __future__ import annotations

import json
import os
import sys


def table(key: str, sw: dict, meta: dict) -> str:
    shape = sw["shape"]
    rows = sw["rows"]
    at70 = sum(1 for r in rows if r["roof_frac"] >= 0.70)
    out = ["# Sweep of the %s layer%s" % (key, "" if not sw.get("zipf") else
                                           " (Zipf-like expert popularity, s = %g)" % sw["zipf"]),
           "",
           "Generated by `python -m paper_2505_19645_b200.sweep_tables` from the record of",
           "`%s` (B200, %s peaks: %.1f GB/s, %.1f TFLOP/s bf16; clocks during the run: median %s MHz,"
           % (meta["command"], meta["peak_source"], meta["hbm_gbs"], meta["bf16_tflops"],
              meta["clocks"].get("sm_mhz")),
           "reasons %s).  Cold L2, CUDA events, %d samples per point in three passes over the grid."
           % (meta["clocks"].get("reasons"), rows[0]["samples"] if rows else 0),
           "",
           "H=%d, E=%d, K=%d, I=%d, I_s=%d; T_thres(0.95) = %d tokens.  %d of %d points at or above 0.70 of the"
           % (shape["hidden"], shape["n_experts"], shape["top_k"], shape["inter"],
              shape["shared_inter"], sw.get("t_thres", 0), at70, len(rows)),
           "roofline (median of all samples; `best` = lowest of the three pass medians).",
           "",
           "| B | gamma | T | us (median) | us (best) | tokens/s | bound | roof us | frac | frac (best) | "
           "T(B,g)/T(B,0) | N_act | Eq. N(t) | T_exp | Eq. T_exp | T > T_thres | launches |",
           "|---|---|---|---|---|---|---|---|---|---|---|---|---|---|---|---|---|"]
    for r in rows:
        out.append("| %d | %d | %d%s | %.1f | %.1f | %.0f | %s | %.1f | %.3f | %.3f | %s | %d | %.2f | %.2f | %.2f | %s | %d |" % (
            r["B"], r["gamma"], r["T"], " (extra)" if r.get("extra") else "", r["us"],
            r["us_best_pass"], r["tokens_per_s"], r["bound"], r["roof_us"], r["roof_frac"],
            r["roof_frac_best_pass"],
            "-" if r["ratio_vs_gamma0"] is None else "%.3f" % r["ratio_vs_gamma0"],
            r["n_active"], r["n_active_expected"], r["t_exp"], r["t_exp_expected"],
            "yes" if r["beyond_t_thres"] else "no", r.get("launches", 0)))
    return "\n".join(out) + "\n"


def main(argv):
    if not argv:
        print(__doc__)
        return 2
    line = [l for l in open(argv[0]).read().splitlines() if l.startswith("{")][-1]
    d = json.loads(line)
    out_dir = argv[1] if len(argv) > 1 else os.path.join(
        os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "profiles")
    peaks = d["layer_roofline"]["peaks"]
    meta = {"command": "python bench.py --steps %d --warmup %d" % (d["steps"], d["warmup"]),
            "peak_source": peaks["source"], "hbm_gbs": peaks["hbm_gbs"],
            "bf16_tflops": peaks["bf16_tflops"], "clocks": d.get("clocks") or {}}
    for key, sw in d["sweeps"].items():
        path = os.path.join(out_dir, "sweep_%s.md" % key.replace(":", "_"))
        with open(path, "w") as f:
            f.write(table(key, sw, meta))
        print("wrote", path)
    return 0


if __name__ == "__main__":
    sys.exit(main(sys.argv[1:]))
