"""Compiles small programs over the library's kernel headers (no GPU needed): the host-side plans a layer would get, and
the registers and spills the assembler reports for kernel instances."""
import re
import subprocess
import tempfile
from pathlib import Path

from paper_2504_06881_b200 import inputs
from paper_2504_06881_b200 import build

NVCC = build._nvcc_base(verbose=True)      # as the library is compiled, with the assembler's report

PLAN_MAIN = """
#include <cstdio>
#include "tconv_bwd_sum.cuh"
using namespace tconv;
int main() {
    Geo g;
    memset(&g, 0, sizeof(g));
    while (scanf("%d %d %d %d %d %d %d", &g.N, &g.C, &g.K, &g.OH, &g.OW, &g.RS, &g.mode) == 7) {
        g.OWP = g.OW;
        g.wide = g.RS > 16;
        g.chan = CH_SUM;
        SumGwPlan p;
        const bool ok = plan_sum_gw(g, &p);
        printf("%d %d %d %d %d %zu\\n", (int)ok, p.flat, p.blocks, p.per, p.splits, p.smem);
    }
}
"""
MODES = ["max_plus", "min_plus", "compound", "parallel"]


def sum_gw_plans(layers):
    """The grad_w plan of each Sum-form layer: dicts of ok, flat, blocks, per, splits, smem."""
    with tempfile.TemporaryDirectory() as tmp:
        src, exe = Path(tmp) / "plan.cu", Path(tmp) / "plan"
        src.write_text(PLAN_MAIN)
        subprocess.run(NVCC + ["-o", str(exe), str(src)], check=True, capture_output=True)
        lines = []
        for d in layers:
            oh, ow = inputs.output_hw(d)
            lines.append(f"{d['N']} {d['C']} {d['K']} {oh} {(ow + 3) // 4 * 4} {d['R'] * d['S']} {MODES.index(d['mode'])}")
        out = subprocess.run([str(exe)], input="\n".join(lines), check=True, capture_output=True, text=True).stdout
    return [dict(zip(("ok", "flat", "blocks", "per", "splits", "smem"), map(int, line.split()))) for line in out.splitlines()]


def resources(header, kernels):
    """{instance: (registers, bytes of spill stores)} of kernel instances like "bwd_sum_finish_kernel<16>"."""
    with tempfile.TemporaryDirectory() as tmp:
        src = Path(tmp) / "probe.cu"
        src.write_text(f'#include "{header}"\nusing namespace tconv;\nvoid* const table[] = {{' +
                       ", ".join(f"(void*){k}" for k in kernels) + "};\nvoid* const* all_of_them() { return table; }\n")
        r = subprocess.run(NVCC + ["-c", "-o", str(Path(tmp) / "probe.o"), str(src)], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
    log = subprocess.run(["c++filt"], input=r.stderr, capture_output=True, text=True, check=True).stdout
    found = {}
    for m in re.finditer(r"entry function '(?:void )?tconv::(.*?)\(tconv::.*?(\d+) bytes spill stores.*?Used (\d+) registers", log, re.S):
        found[m.group(1)] = (int(m.group(3)), int(m.group(2)))
    return {k: found[k] for k in kernels}
