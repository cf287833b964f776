"""Launch shapes and shared memory (csrc/dwf_launch.cuh, dwf_kernels.cuh) without a GPU: how many of
k_hop's CTAs of the default shape fit on an SM, and k_smix's CTA sizes, from the launchers' own
arithmetic compiled with nvcc into a host program."""
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
    printf("%d %d %zu %zu", Ns, spb, hop_smem_bytes<P_F64, E_PLAIN>(spb, Ns), hop_smem_bytes<P_F64, E_M>(spb, Ns));
    for (int mode : {S_PLAIN, S_CGP, S_DUAL}) {
      const int s32 = smix_sites_per_block(P_F32, mode, Ns), s64 = smix_sites_per_block(P_F64, mode, Ns);
      printf(" %d %zu %d", s32, smix_smem_bytes<P_F32>(s32, Ns, mode == S_DUAL), s64);
    }
    printf("\n");
  }
}
'''


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("needs nvcc")
    tmp_path = tmp_path_factory.mktemp("shapes")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROG)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-DDWF_KERNEL_TU", "-I", CSRC,
                           "-c", str(src), "-o", str(exe) + ".o"])
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", str(exe) + ".o", "-o", str(exe)])
    rows = [list(map(int, ln.split())) for ln in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert [r[0] for r in rows] == list(range(1, 65))
    return rows


def test_fp64_hops_fit_the_ctas_their_registers_are_capped_for(rows):
    """Four 128-thread CTAs per SM (the launch bounds' register cap); three where Ns = 1 or 2
    makes a CTA's sites, not its threads, the limit."""
    for ns, spb, plain, m5, *_ in rows:
        assert 1 <= spb * ns <= 128
        for size in (plain, m5):
            assert (size + PER_CTA) * (3 if ns < 3 else 4) <= SM_BYTES, (ns, spb, size)


def test_smix_ctas_are_wide_where_their_matrices_are_large(rows):
    """256 threads from Ns = 33 (plain), 48 (p-update) and 32 (two matrices) on, 128 below and for the
    dense FP64 form; never more than the kernel's 256 threads or an SM's shared memory."""
    for ns, _, _, _, *smix in rows:
        for i, wide_from in enumerate((33, 48, 32)):
            s32, smem, s64 = smix[3 * i:3 * i + 3]
            assert s32 == (256 // ns if ns >= wide_from else max(1, min(64, 128 // ns)))
            assert s64 == max(1, min(64, 128 // ns))
            assert s32 * ns <= 256 and smem + PER_CTA <= SM_BYTES
