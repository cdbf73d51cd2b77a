"""The persistent level loop under register pressure: a variant library whose loop takes its parent
tiles by the fixed stride with loads ahead (NP_LOOP_AHEAD=1, more spilled registers), in a process of
its own. Its grid barrier once let warps run ahead of thread 0 there (wrong distances with child
blocks that are not staged, a coarsening factor of 8 or 16). Exact against the oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_loop_with_loads_ahead():
    from paper_2201_02789_gb300 import build
    lib = build.build(defines=("NP_LOOP_AHEAD=1",), out_dir=os.path.join(build.BUILD, "opt_loop_ahead"))
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=dict(os.environ, NESTPAR_LIB=lib),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "120 solves, wrong: []" in r.stdout, (r.stdout[-3000:], r.stderr[-3000:])


def main():
    sys.path[:0] = [os.path.dirname(HERE), HERE]
    import numpy as np
    import oracle
    from gpu_util import DevGraph, bfs, sssp
    from paper_2201_02789_gb300 import gen
    from paper_2201_02789_gb300 import nestpar as npb
    ctx, g, wrong, solves = npb.Context(0), gen.bfs4k(), [], 0
    dg = DevGraph(g)
    level, dist = oracle.bfs(g.row_ptr, g.col, 0), oracle.sssp(g.row_ptr, g.col, g.w, 0)
    for cf in (1, 2, 4, 8, 16):
        for threshold in (0, 1, 2, 32):
            for grid in (0, 1, 4):
                cfg = npb.config("tca", driver=npb.NP_DRIVER_PERSISTENT, threshold=threshold, cfactor=cf,
                                 parent_grid=grid)
                for name, solve, ref in (("bfs", bfs, level), ("sssp", sssp, dist)):
                    solves += 1
                    if not np.array_equal(solve(ctx, dg, 0, cfg), ref):
                        wrong.append((name, cf, threshold, grid))
    ctx.close()
    print(f"{solves} solves, wrong: {wrong}")


if __name__ == "__main__":
    main()
