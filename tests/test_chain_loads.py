"""Kernels launched programmatically (launch_chain) run beside the kernel that
writes their input until chain_wait returns, so nothing of that input may be
read through the read-only path (ld.global.nc wants data that no one writes
while the kernel lives) or by a load that the compiler may move above the
wait.  Checked on the source: a kernel with a chain_wait takes const
__restrict__ pointers to, and uses __ldg on, only what no kernel of a chain
writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1312_4587_gb300", "csrc")

# fixed at creation, or the caller's (a call's first kernel is launched plainly)
FIXED = {"x", "y", "w", "h", "M", "rank", "slabs", "cell_pin_ptr", "scale", "scale_dev", "done"}


def sources():
    out = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(p).read())
        out[os.path.basename(p)] = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return out


def kernels():
    """(file, name, parameter list, body) of every __global__ function."""
    for f, s in sources().items():
        for m in re.finditer(r"__global__\s+void(?:\s*__launch_bounds__\((?:[^()]|\([^()]*\))*\))?"
                             r"\s*(\w+)\s*\(([^)]*)\)\s*\{", s):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(s[i], 0)
                i += 1
            yield f, m.group(1), m.group(2), s[m.end():i]


def chained():
    return [k for k in kernels() if "chain_wait()" in k[3]]


def test_the_kernels_are_found():
    names = {k[1] for k in chained()}
    for n in ("k_rows_fwd", "k_cols", "k_rows_inv", "k_gather", "k_wa", "k_pin_sum", "k_split",
              "k_loop_g", "k_loop_update", "k_report", "k_energy_out"):
        assert n in names


def test_no_read_only_path_to_what_a_chain_writes():
    bad = []
    for f, name, params, body in chained():
        for p in re.findall(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", params):
            if p not in FIXED:
                bad.append(f"{f}: {name}: const __restrict__ {p}")
        # restricted aliases of what the loop's kernels hand on within an iteration
        for src in re.findall(r"const\s+\w+\*\s*__restrict__\s+\w+\s*=\s*([\w.]+)", body):
            if src in ("b.gN", "b.gW", "b.g"):
                bad.append(f"{f}: {name}: restricted {src}")
        for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?\s*(\w+)", body):
            if arg not in FIXED:
                bad.append(f"{f}: {name}: __ldg({arg})")
    assert not bad, "\n".join(bad)


def test_field_loads_stay_behind_the_wait():
    src = sources()["fftpl_internal.cuh"]
    found = re.findall(r"__device__ __forceinline__ \w+ (load_field4|ld_dep)\([^)]*\)\s*\{(.*?)\n\}",
                       src, flags=re.S)
    assert {name for name, _ in found} == {"load_field4", "ld_dep"}
    for name, body in found:
        assert "asm volatile" in body and '"memory"' in body and ".nc" not in body, name
