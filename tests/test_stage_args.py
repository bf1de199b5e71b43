"""A stage whose local term and hop disagree about the dagger is refused before any launch, in
every precision (the FP32 and 16-bit kernels have one switch for both).  Runs in a child process
that sees no device."""
import os
import subprocess

PROGRAM = r"""
#include <cstdio>
#include "stage.cuh"
namespace dwf {
cudaError_t launch_stage_prec(int, const StageArgs&, int, bool, bool, cudaStream_t);
}
int main() {
  int devices = 0;
  if (cudaGetDeviceCount(&devices) == cudaSuccess && devices) return 2;
  for (int prec = 0; prec < 4; prec++)
    for (int dag = 0; dag < 2; dag++)
      for (int local : {dwf::LOC_NONE, dwf::LOC_M5, dwf::LOC_M5DAG}) {
        dwf::StageArgs a{};
        a.hop_scale = 1.0;
        a.l_alpha = 1.0;
        a.Vp = a.Vhb = a.Vhb_pad = 32;
        a.seg_cps = 1;
        a.local_mode = local;
        const bool refused = dwf::launch_stage_prec(prec, a, 8, dag, false, 0) ==
                             cudaErrorInvalidValue;
        const bool agree = local == dwf::LOC_NONE || (local == dwf::LOC_M5DAG) == (dag == 1);
        if (refused == agree) printf("prec %d dag %d local %d\n", prec, dag, local);
      }
  return 0;
}
"""


def test_mismatched_local_term_is_refused(tmp_path):
    from paper_1804_08593_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "args.cu", tmp_path / "args"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe), lib, "-lcudart",
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe)], env=dict(os.environ, CUDA_VISIBLE_DEVICES=""),
                       capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    assert r.stdout == ""
