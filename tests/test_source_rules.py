"""Rules of the step kernels that no safe run can show broken, checked on the
source.

A chained step kernel (launched with programmatic serialization) starts
while the kernel before it still writes the chained kernel's input.  A const
__restrict__ parameter would promise that the input never changes while the
kernel runs, and would allow its loads to move above the wait or to go through
the non-coherent cache.  A stale cell cannot be provoked safely, so the rule is
checked on the source: no kernel named in a launch_chained call has such a
parameter, and launch_chained itself refuses a bare pointer to const."""
import glob
import os
import re
import subprocess

from paper_2006_15932_gb300 import build as B

KERNEL = re.compile(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^{;]*)\)\s*\{", re.S)
INPUT = re.compile(r"\bconst\s+\w+\s*\*\s*(?:__restrict__\s*)?\w+|__ldg\(")


def test_no_chained_kernel_promises_a_read_only_input():
    text = {f: open(f).read() for f in glob.glob(os.path.join(B.CSRC, "*.cu*"))}
    every = "\n".join(text.values())
    chained = set(re.findall(r"launch_chained\(\s*(k_\w+)", every))
    assert {"k_step_f64", "k_step_f64_small", "k_step_tma", "k_step_half", "k_step_staged", "k_step_bf16"} <= chained
    seen = set()
    for m in KERNEL.finditer(every):
        if m.group(1) in chained:
            seen.add(m.group(1))
            assert not INPUT.search(m.group(2)), m.group(1)
    assert seen == chained


def test_chained_launch_refuses_a_bare_pointer_to_const(tmp_path):
    src = tmp_path / "bare.cu"
    src.write_text("""#include "dbm_device.cuh"
__global__ void k_bare(const float *in, float *out) { out[0] = in[0]; }
cudaError_t go(const float *in, float *out) { return dbm::launch_chained(k_bare, dim3(1), dim3(1), 0, 0, in, out); }
""")
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-c", str(src), "-o", str(tmp_path / "bare.o")],
                       capture_output=True, text=True)
    assert r.returncode != 0 and "ChainedIn" in r.stdout + r.stderr, r.stderr


def test_later_waits_have_the_limit_of_the_first_wait_and_its_second():
    """A wait that gives up must not let the CTA leave with a copy in flight: a
    step's first wait and the species-staged buffers have a second wait behind
    them; the wait for a later species of a tile has both limits at once."""
    every = "\n".join(open(f).read() for f in glob.glob(os.path.join(B.CSRC, "*.cu*")))
    reported = re.findall(r"!\s*mbar_wait\(([^;]*?)\)\)\s*raise_flag", every)
    assert reported and all(r.endswith("2 * TMA_WAIT_LIMIT") for r in reported), reported
