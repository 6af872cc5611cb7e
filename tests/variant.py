"""A copy of the package whose library has one translation unit compiled with
other macros (a wait that runs out at once, a driver without a feature)."""
import os
import shutil
import subprocess
import sys

from paper_2301_00228_gb300 import build as B


def package(where, unit, *macros):
    """The package with csrc/<unit>.cu compiled with -D<macro> for each, under
    the directory `where` (to be first in a child's sys.path)."""
    B.build()
    pkg = where / B.PKG.name
    pkg.mkdir()
    for py in B.PKG.glob("*.py"):
        shutil.copy(py, pkg)
    obj = where / f"{unit}.o"
    subprocess.run([B.nvcc()] + B.flags() + [f"-D{m}" for m in macros] + ["-c", str(B.CSRC / f"{unit}.cu"), "-o",
                                                                       str(obj)], check=True)
    objs = [obj if s.stem == unit else B.BUILD / f"{s.stem}.o" for s in B.sources()]
    subprocess.run([B.nvcc()] + B.ARCH + ["-shared", "-o", str(pkg / B.LIB.name)] + [str(o) for o in objs], check=True)
    return where


def run(where, code, timeout=600):
    """Runs `code` in a child process that imports that package; its output."""
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([str(where), str(B.ROOT / "tests")]))
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=timeout, env=env,
                         cwd=str(where))
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-3000:]
    return out.stdout
