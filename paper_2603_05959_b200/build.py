"""Build the CUDA library in-tree: paper_2603_05959_b200/libovggt.so (sm_100a only)."""
import os
import re
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libovggt.so")
OUT_CHECKED = os.path.join(HERE, "libovggt_checked.so")     # the same library built with -DOVGGT_BOUNDS_CHECK
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def needs_build(out: str = OUT) -> bool:
    if not os.path.exists(out):
        return True
    deps = sources() + [os.path.join(os.path.dirname(HERE), "include", "ovggt.h")]
    return any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def check_register_pool(ptxas_log: str, kernel: str = "k_attn_tcgen05") -> None:
    """The attention kernels move registers between their warpgroups with setmaxnreg, inside the pool they were
    launched with; an increase the pool cannot serve would wait for ever.  The source states the launch count they were
    budgeted for (kRegsLaunch); refuse a build whose ptxas report says otherwise."""
    src = open(os.path.join(CSRC, "attn_tcgen05.cuh")).read()
    want = int(re.search(r"constexpr int kRegsLaunch = (\d+);", src).group(1))
    used = re.findall(rf"Compiling entry function '[^']*{kernel}[^']*'.*?Used (\d+) registers", ptxas_log, re.S)
    if not used:
        raise RuntimeError(f"ptxas report for {kernel} not found")
    for regs in used:                                   # (every instantiation)
        if int(regs) != want:
            raise RuntimeError(f"{kernel} is launched with {regs} registers, budgeted for {want}")


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    """checked: the variant in which every index a kernel reads from device memory is range-checked (a bad one is
    skipped and reported through the status word); written to libovggt_checked.so, loaded by the binding when the
    environment says OVGGT_LIBRARY=checked."""
    OUT = OUT_CHECKED if checked else globals()["OUT"]
    if not force and not needs_build(OUT):
        return OUT
    tmp = OUT + ".tmp"
    cmd = [NVCC, "-Xptxas", "-v", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "--cudart", "static"] + (["-DOVGGT_BOUNDS_CHECK"] if checked else []) + [
           "-o", tmp, os.path.join(CSRC, "ovggt_api.cu"), "-ldl"]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or r.returncode != 0:
        print(r.stdout, file=sys.stderr)
    if r.returncode != 0:
        raise subprocess.CalledProcessError(r.returncode, cmd)
    try:
        for kernel in ("k_attn_tcgen05", "k_attn_f32"):
            check_register_pool(r.stdout, kernel)
    except Exception:
        os.remove(tmp)
        raise
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, checked="--checked" in sys.argv))
