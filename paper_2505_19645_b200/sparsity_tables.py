"""Tables of the sparsity sweep (Sec. 4.3) and of the analytical-model fit (Sec. 3.4) from
bench.py records.

    python -m paper_2505_19645_b200.sparsity_tables OUT.md RESULT.json [RESULT.json ...]

Each RESULT.json is the record of one run
    python bench.py --config qwen2-57b-a14b --top-k K --grid sparsity --no-cpu-baseline --record RESULT.json
(or --dense-contrast instead of --top-k).  Writes OUT.md: target efficiency T(B,0)/T(B,gamma)
per variant and batch size, roofline fractions, and the fit of
time(t) = bias + k1 G(t) + k2 N(t) + k3 G(T_exp(t)) to the K variants' layer times with the
mean squared error over all points for strided subsets of the measurements.
"""
from __future__ import annotations

import json
import os
import statistics
import sys

from . import model_fit


def _line(path):
    return json.loads([l for l in open(path).read().splitlines() if l.startswith("{")][-1])


def main(argv):
    if len(argv) < 2:
        print(__doc__)
        return 2
    out_path, paths = argv[0], argv[1:]
    variants = []
    for p in paths:
        d = _line(p)
        for key, sw in d["sweeps"].items():
            variants.append((sw["shape"], sw["rows"], p, d))
    variants.sort(key=lambda v: (v[0]["n_experts"] == 1, v[0]["top_k"]))
    batches = sorted({r["B"] for _, rows, _, _ in variants for r in rows})
    gammas = sorted({r["gamma"] for _, rows, _, _ in variants for r in rows if r["gamma"] > 0})
    peaks = variants[0][3]["layer_roofline"]["peaks"]
    out = ["# Sparsity sweep and dense contrast on the Qwen2-57B-A14B shape; fit of the analytical model",
           "",
           "Generated by `python -m paper_2505_19645_b200.sparsity_tables` from the records of",
           "`python bench.py --config qwen2-57b-a14b --top-k K --grid sparsity --no-cpu-baseline` for",
           "K = %s and `--dense-contrast` (B200, %s peaks %.1f GB/s / %.1f TFLOP/s; cold L2, CUDA events,"
           % (", ".join(str(v[0]["top_k"]) for v in variants if v[0]["n_experts"] > 1),
              peaks["source"], peaks["hbm_gbs"], peaks["bf16_tflops"]),
           "30 samples per point in three passes, median).", ""]
    for g in gammas:
        out += ["## Target efficiency T(B,0)/T(B,gamma) of the layer at gamma = %d (Sec. 3.1)" % g, "",
                "| variant | " + " | ".join("B=%d" % b for b in batches) + " |",
                "|---|" + "---|" * len(batches)]
        for shape, rows, _, _ in variants:
            name = "dense" if shape["n_experts"] == 1 else "K=%d" % shape["top_k"]
            by = {(r["B"], r["gamma"]): r for r in rows}
            cells = []
            for b in batches:
                r = by.get((b, g))
                cells.append("-" if r is None or r["target_efficiency"] is None
                             else "%.2f" % r["target_efficiency"])
            out.append("| %s | %s |" % (name, " | ".join(cells)))
        out.append("")
    out += ["## Roofline fraction of the layer over each variant's points", "",
            "| variant | points | median | min | max |", "|---|---|---|---|---|"]
    for shape, rows, _, _ in variants:
        name = "dense" if shape["n_experts"] == 1 else "K=%d" % shape["top_k"]
        fr = [r["roof_frac"] for r in rows]
        out.append("| %s | %d | %.2f | %.2f | %.2f |" % (name, len(fr), statistics.median(fr), min(fr), max(fr)))
    out.append("")

    # fit on the K variants (the dense contrast has another expert width)
    k_paths = [p for shape, _, p, _ in variants if shape["n_experts"] > 1]
    if k_paths:
        data, shape = model_fit.load_sweeps(k_paths)
        bw = peaks["hbm_gbs"] * 1e9
        ridge = peaks["bf16_tflops"] * 1e12 / bw
        H, I, Is, E = shape["hidden"], shape["inter"], shape["shared_inter"], shape["n_experts"]
        lo, hi = model_fit.default_bounds(6.0 * H * Is + 4.0 * E * H, 6.0 * H * I, bw)
        cols = {k: data[k] for k in ("t", "K", "E", "us")}
        n = len(cols["t"])
        out += ["## Fit of time(t) = bias + k1 G(t) + k2 N(t) + k3 G(T_exp(t)) (Sec. 3.4, Algorithm 1)", "",
                "%d measured layer times (us), sorted by K, gamma, batch size; ridge point %.0f rows;" % (n, ridge),
                "parameters fitted on every stride-th point, mean squared error over all points:", "",
                "| fit points m | stride | MSE us^2 | bias | k1 | k2 | k3 | lambda | s |",
                "|---|---|---|---|---|---|---|---|---|"]
        for stride in (25, 16, 11, 8, 4, 2, 1):
            sel = {k: v[::stride] for k, v in cols.items()}
            x, _ = model_fit.fit(sel, ridge, lo, hi)
            out.append("| %d | %d | %.1f | %s |" % (len(sel["t"]), stride, model_fit.mse(x, cols, ridge),
                                                   " | ".join("%.4g" % v for v in x)))
        med = statistics.median(cols["us"].tolist())
        out += ["", "Median layer time of the fitted points: %.0f us." % med, ""]
    with open(out_path, "w") as f:
        f.write("\n".join(out))
    print("wrote", out_path)
    return 0


if __name__ == "__main__":
    sys.exit(main(sys.argv[1:]))
