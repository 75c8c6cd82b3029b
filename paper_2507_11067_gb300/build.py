"""Build the sm_103a CUDA library libmms.so in-tree (paper_2507_11067_gb300/_build).

Each translation unit is compiled by nvcc in parallel with one -gencode
(compute_103a -> sm_103a) and linked into a shared library with the CUDA
runtime linked statically, so the library depends only on the driver.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libmms.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

SOURCES = ["abi.cu", "sweep_cc.cu", "sweep_star.cu", "sweep_box_high.cu", "sweep_2d.cu", "sweep_any.cu", "wave.cu",
           "band_tc.cu", "noalloc.cu", "aniso.cu", "sweep_f64.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2",
                     "--expt-relaxed-constexpr", "-I" + INCLUDE, "-I" + CSRC, "-I" + os.path.join(BUILD, "gen")]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the CUDA toolkit is required to build libmms.so")


TABLE = os.path.join(HERE, "tuned.json")
GEN = os.path.join(BUILD, "gen")
SHAPE_IDS = {"star": 0, "box": 1, "star2d": 2, "box2d": 3}
PATH_IDS = {"cuda_core": 1, "tf32": 2, "3xtf32": 3, "bf16x3": 4, "naive": 5}


def tuned_rows(table: str = TABLE):
    """The autotuner's table as the library builds it in: for every GPU model
    and (shape, radius, path), the variant tuned on its largest grid (the row
    tune.load_table() registers).  Returns sorted (gpu, shape id, r, path id,
    variant) tuples."""
    import json
    best = {}
    if os.path.exists(table):
        for k, v in json.load(open(table)).items():
            gpu, shape, rr, path, size = k.split("|")
            dims = [int(x) for x in size.split("x")]
            vol = dims[0] * dims[1] * dims[2]
            key = (gpu, SHAPE_IDS[shape], int(rr[1:]), PATH_IDS[path])
            if key not in best or vol > best[key][0]:
                best[key] = (vol, int(v["variant"]))
    return sorted(k + (v,) for k, (_, v) in best.items())


def write_tuned_defaults(table: str = TABLE, out_dir: str = GEN) -> str:
    """Writes tuned_defaults.inc (C++ rows of the tuned table, included by
    abi.cu); rewrites it only when its content changes."""
    os.makedirs(out_dir, exist_ok=True)
    path = os.path.join(out_dir, "tuned_defaults.inc")
    lines = ["// Generated by build.py from tuned.json: the tuned variant of each (GPU model,",
             "// shape, radius, path), tuned on its largest grid.  Do not edit.",
             "static const TunedRow kTunedRows[] = {"]
    rows = tuned_rows(table)
    for gpu, shape, r, pth, var in rows:
        lines.append(f'    {{"{gpu}", {shape}, {r}, {pth}, {var}}},')
    if not rows:
        lines.append('    {"", -1, 0, 0, -1},')
    lines.append("};")
    text = "\n".join(lines) + "\n"
    if not os.path.exists(path) or open(path).read() != text:
        with open(path, "w") as f:
            f.write(text)
    return path


def _deps():
    return (glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
            + glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__), TABLE])


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _deps())


def _compile(src: str, extra) -> str:
    obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
    cmd = [nvcc()] + NVCC_FLAGS + list(extra) + ["-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
    if r.stderr.strip():
        sys.stderr.write(r.stderr)
    return obj


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    """Compile every CUDA source and link libmms.so; returns its path."""
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    write_tuned_defaults()
    extra = ["-Xptxas", "-v"] if verbose_ptxas else []
    with cf.ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 4)) as ex:
        objs = list(ex.map(lambda s: _compile(s, extra), SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc()] + ARCH + ["-shared", "-cudart", "static", "-o", tmp] + objs + ["-ldl", "-lpthread", "-lrt"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv)
    print(LIB)
