"""Autotuner of the contraction schedule per virtual-space size bucket.

For each bucket it builds one synthetic domain of that virtual size (few
occupied orbitals, so a trial takes milliseconds), times lno_ot_energy with
every candidate row (cap on the contraction tile's width x cap on the triplets
of a group) written to a one-row table, and keeps the library's own schedule
unless another row is faster by more than the trials differ.  The result is the
text table the library reads through lno_ot_options.tune_cache ("vmax bn
group_cap").

    python -m paper_2311_10048_gb300.tune out.txt [--precision bf16x6]
"""
from __future__ import annotations

import argparse
import os
import tempfile
import time

BUCKETS = (96, 160, 224, 320, 448)          # vmax of each bucket
# What the library does without a table: no cap on the width, 1024 triplets a group.
DEFAULT = (0, 1024)
# Caps on the tile width (columns, multiples of 16; 0 = none: 512 / S columns for S
# slices, 256 at most).  The last of each row is the widest tile with two accumulator
# sets (2 S w <= 512 TMEM columns), whose epilogue overlaps the next tile entirely.
TILE_WIDTHS = {"bf16x3": (0, 192, 128), "tf32": (0, 192, 128), "bf16x6": (0, 112, 80),
               "bf16x10": (0, 96, 80, 64), "bf16x15": (0, 64, 48)}
# Every cap is a row's upper bound: below the default, launch gaps and part-filled last
# rounds of tiles cost up to a fifth of a mid-size domain's call.
GROUP_CAPS = (1024, 256, 64)
MARGIN = 0.98   # repeated trials differ by about 1 %


def candidates(precision):
    return [(bn, g) for bn in TILE_WIDTHS.get(precision, (0,)) for g in GROUP_CAPS]


def pick(times):
    """Fastest row of {row: ms}; the default unless beaten by more than the margin."""
    best = min(times, key=times.get)
    return best if times[best] < MARGIN * times[DEFAULT] else DEFAULT


def _time_row(lno_ot, dd, precision, row, reps=3):
    fd, path = tempfile.mkstemp(suffix=".tune")
    with os.fdopen(fd, "w") as f:
        f.write(f"{100000} {row[0]} {row[1]}\n")
    try:
        ctx = lno_ot.Context(0, precision, tune_cache=path)
        ctx.energy(dd)                                   # warm-up
        best = float("inf")
        for _ in range(reps):
            ctx.energy(dd)
            best = min(best, ctx.stats()["ms_total"])   # launch gaps included
        ctx.close()
    finally:
        os.unlink(path)
    return best


def autotune(path, precision="bf16x6", buckets=BUCKETS, nocc=(10, 8), log=print):
    """Write the tuning table to ``path``; returns the rows."""
    from . import lno_ot
    from .synth import make_domain
    rows = []
    for vmax in buckets:
        v = vmax - 16
        d = make_domain(v + nocc[0], nocc, naux=3 * (v + nocc[0]), L=0.75 * (v + nocc[0]),
                        seed=vmax)
        dd = lno_ot.to_device(d)
        times = {row: _time_row(lno_ot, dd, precision, row) for row in candidates(precision)}
        best = pick(times)
        rows.append((vmax,) + best)
        log(f"bucket v<={vmax}: " + ", ".join(f"bn={c} cap={g}: {t:.2f} ms"
                                            for (c, g), t in times.items()) + f" -> {best}")
        del dd
    with open(path, "w") as f:
        f.write(f"# lno_ot tuning table ({precision}); vmax bn group_cap\n")
        for r in rows:
            f.write(f"{r[0]} {r[1]} {r[2]}\n")
    return rows


if __name__ == "__main__":
    ap = argparse.ArgumentParser()
    ap.add_argument("out")
    ap.add_argument("--precision", default="bf16x6")
    a = ap.parse_args()
    t = time.time()
    autotune(a.out, a.precision)
    print(f"tuned in {time.time() - t:.1f} s -> {a.out}")
