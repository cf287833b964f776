"""k_hop's shared memory (csrc/dwf_kernels.cuh) without a GPU: how many CTAs of the default shape
fit on an SM, from the kernels' own size arithmetic compiled with nvcc into a host program."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_0423_gb300", "csrc")
SM_BYTES, PER_CTA = 228 * 1024, 1024  # shared memory of an SM, and what it takes per CTA beside its own

PROG = r'''
#include <cstdio>
#include "dwf_launch.cuh"
using namespace dwf;
int main() {
  for (int Ns = 1; Ns <= 64; ++Ns) {
    const int spb = hop_sites_per_block(P_F64, Ns);
    printf("%d %d %zu %zu\n", Ns, spb, hop_smem_bytes<P_F64, E_PLAIN>(spb, Ns), hop_smem_bytes<P_F64, E_M>(spb, Ns));
  }
}
'''


@pytest.mark.skipif(not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")), reason="needs nvcc")
def test_fp64_hops_fit_the_ctas_their_registers_are_capped_for(tmp_path):
    """Four 128-thread CTAs per SM (the launch bounds' register cap); three where Ns = 1 or 2
    makes a CTA's sites, not its threads, the limit."""
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROG)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-DDWF_KERNEL_TU", "-I", CSRC,
                           "-c", str(src), "-o", str(exe) + ".o"])
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", str(exe) + ".o", "-o", str(exe)])
    rows = [list(map(int, ln.split())) for ln in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert len(rows) == 64
    for ns, spb, plain, m5 in rows:
        assert 1 <= spb * ns <= 128
        for size in (plain, m5):
            assert (size + PER_CTA) * (3 if ns < 3 else 4) <= SM_BYTES, (ns, spb, size)
