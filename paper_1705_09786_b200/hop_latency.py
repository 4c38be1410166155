"""Where the time of one instance goes when a single key is in flight: `python -m paper_1705_09786_b200.hop_latency`.

With max_active_keys = 1 no two instances overlap: in every round the cells that have a row of the instance work on it and the cells
that read them wait.  The kernel's own cycle counters (ampnet_get_phase_cycles: the first CTA of every cell) say how long each cell
worked.  A dense row is in one cell at a time, so what is left of its latency is the hand-over from one cell to the next: fence,
counter and poll, and the block barriers around them (the "output" phase holds a cell's own fence).  The tokens of a list and the
nodes of a tree work side by side, so there the cells' times add up to more than the latency.  Accumulators are beside the way.
Asynchronous epochs of the MLP, list and tree workloads are measured; sizes are kept small (seconds).
"""
import argparse

import numpy as np

from workloads import data, ir, params as wp

from . import Engine

CASES = {"mlp": (lambda: ir.mlp((784, 256, 256, 10)), lambda n: data.mlp_instances(n=n), 2048, 32),
         "rnn": (ir.rnn, lambda n: data.list_instances(n=n), 3000, 50),
         "tree": (ir.tree, lambda n: data.tree_instances(n=n), 600, 100)}
PHASES = ("gather", "product", "output", "loss")       # marks 2..5 of a forward cell, 10..13 of an input-gradient cell


def measure(family, sm_mhz):
    build, make, n, muf = CASES[family]
    g, inst = build(), make(n)
    e = Engine(g)
    e.load_instances(inst)
    e.set_params(wp.init_params(g))
    for _ in range(3):
        st, _ = e.run_epoch(mak=1, muf=muf, lr=0.01, deterministic=False, timeout_s=60)
    per_inst = st.seconds * 1e6 / inst.n
    lines = [f"{family}: {per_inst:.1f} us per instance with one key in flight ({inst.n / st.seconds:.0f} instances/s), "
             f"{st.node_messages / inst.n:.1f} node messages per instance"]
    busy_total = 0.0
    for node in g.ppt_nodes():
        a, _ = e.phase_cycles(node)
        us = a.astype(np.float64) / sm_mhz / inst.n                    # microseconds per instance
        parts = lambda v: ", ".join(f"{k} {x:.2f}" for k, x in zip(PHASES, v) if x >= 0.005)
        f_busy, b_busy, acc = us[2:6].sum(), us[10:14].sum(), us[7] + us[14] + us[15]
        busy_total += f_busy + b_busy
        lines.append(f"  {g.names[node]:<12} forward cell works {f_busy:6.2f} us per instance ({parts(us[2:6])})" +
                     (f"; gradient cell {b_busy:6.2f} us ({parts(us[10:14])})" if b_busy > 0 else "") +
                     (f"; accumulator {acc:6.2f} us" if acc > 0 else ""))
    lines.append(f"  these cells together {busy_total:.1f} us per instance" +
                 (f", hand-overs {per_inst - busy_total:.1f} us" if family == "mlp" else " (messages of one instance work in several at a time)"))
    e.close()
    return lines


def main():
    ap = argparse.ArgumentParser(description=__doc__)
    ap.add_argument("--families", default="mlp,rnn,tree")
    ap.add_argument("--sm-mhz", type=float, default=None, help="SM clock the cycle counters ran at (default: the device's maximum)")
    args = ap.parse_args()
    import torch
    mhz = args.sm_mhz or getattr(torch.cuda.get_device_properties(0), "clock_rate", 1965000) / 1e3
    for fam in args.families.split(","):
        print("\n".join(measure(fam, mhz)))


if __name__ == "__main__":
    main()
