"""Register budget of the sweeps and of the many-step kernel (host-side
compilation, no GPU), as test_kernel_resources has for the single-step kernels:
the blocks per SM that their comments justify by registers hold only while the
row loops compile without spills.  The many-step kernel accepts small ones where
it was measured faster with them (20 warps per SM at 96 registers, FP64 storage
at 128): their limits are the measured sizes, rounded up."""
import re
import subprocess

import pytest

from paper_2301_00228_gb300 import build as B

FLOAT, HALF, BF16, BFP, DOUBLE = ("PopDirectIfE", "PopNeq16I6__halfE", "PopNeq16I13__nv_bfloat16E", "PopBfp13",
                                  "PopDirectIdE")
# (unit, kernel, policy, rest of the template arguments, registers, bytes of spill loads at most)
SHAPES = [("lbps_sweep", "sweep_kernel", FLOAT, "Li4ELi3ELb0", 168, 0)]
for p, minb in ((FLOAT, 5), (BFP, 5), (HALF, 4), (BF16, 4)):
    SHAPES += [("lbps_sweep", "sweep_kernel", p, f"Li2ELi{minb}ELb{x}", 65536 // (128 * minb) // 8 * 8, 0) for x in (0, 1)]
    SHAPES += [("lbps_sweep", "sweep_periodic_kernel", p, "Li4", 128, 0), ("lbps_sweep", "sweep_batch_kernel", p, "", 128, 0)]
    SHAPES += [("lbps_fused", "fused_kernel", p, f"Li512ELi1ELb{x}", 128, 0) for x in (0, 1)]
    SHAPES += [("lbps_fused", "fused_kernel", p, f"Li640ELi1ELb{x}", 96, 96 if p == BFP else 40) for x in (0, 1)]
SHAPES += [("lbps_fused", "fused_kernel", DOUBLE, f"Li512ELi1ELb{x}", 128, 112) for x in (0, 1)]


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("ptxas")
    info = {}
    for unit in ("lbps_sweep", "lbps_fused"):
        r = subprocess.run([nvcc] + B.flags() + ["-Xptxas", "-v", "-c", str(B.CSRC / f"{unit}.cu"), "-o",
                                                 str(out / f"{unit}.o")], capture_output=True, text=True, timeout=900)
        assert r.returncode == 0, r.stderr[-3000:]
        cur = None
        for line in r.stderr.splitlines():
            m = re.search(r"(?:Compiling entry function|Function properties for) '?(_Z\w+)", line)
            if m:
                cur = (unit, m.group(1))
                info.setdefault(cur, [None, None])
            m = re.search(r"(\d+) bytes spill loads", line)
            if m and cur:
                info[cur][1] = int(m.group(1))
            m = re.search(r"Used (\d+) registers", line)
            if m and cur:
                info[cur][0] = int(m.group(1))
    return info


@pytest.mark.parametrize("unit,kernel,policy,rest,regs,spill", SHAPES)
def test_shapes_fit(report, unit, kernel, policy, rest, regs, spill):
    pat = re.compile(rf"\d{kernel}INS_\d+{policy}E?{rest}")
    hits = [v for (u, k), v in report.items() if u == unit and pat.search(k)]
    assert len(hits) == 1, (kernel, policy, rest, len(hits))
    assert hits[0][0] <= regs and hits[0][1] <= spill, (kernel, policy, rest, hits[0])
