"""Host-side rules of the launchers that no GPU is needed for: a small program linked against the library calls
them with no device visible.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1307_6101_gb300")

PRELUDE = r"""
#include <cstdio>
#include <cstdlib>
#include <exception>
#include "kernels.h"
using namespace dd;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
// a lattice of two SAP blocks per direction
static Geom geom(int b0, int b1, int b2, int b3) {
  Geom g{};
  const int B[4] = {b0, b1, b2, b3};
  g.V = g.vB = 1;
  for (int d = 0; d < 4; ++d) {
    g.B[d] = B[d];
    g.L[d] = 2 * B[d];
    g.fB[d] = fdiv_make(B[d]);
    g.vB *= B[d];
    g.V *= g.L[d];
  }
  return g;
}
"""


def run(tmp_path, body):
    """Compile and run main() { PRELUDE; body } with no GPU visible."""
    import __graft_entry__
    __graft_entry__.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PRELUDE + "int main() {\n  int nd = 0;\n  if (cudaGetDeviceCount(&nd) == cudaSuccess && nd > 0) "
                   "return 2;\n" + body + "\n  return 0;\n}\n")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr", "-O0", "-I",
           os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"), str(src), os.path.join(PKG, "libddamg.so"),
           "-Xlinker", "-rpath=" + PKG, "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)


def test_persistent_sap_stages_the_blocks_of_its_own_plan(tmp_path):
    """Levels that only the plan of the FP16 kernels takes (sap_nsl stays 0 there): the persistent launch has room for
    every block inside its SAP blocks, and refuses a plan that stages fewer."""
    run(tmp_path, r"""
  const int shapes[][5] = {{3, 2, 2, 2, 32}, {3, 3, 2, 2, 16}, {2, 3, 3, 3, 8}, {5, 2, 2, 2, 24}};
  const int cls[] = {8, 4, 2, 8}, slots[] = {6, 7, 8, 6};
  for (int t = 0; t < 4; ++t) {
    CoarseOp<float> op{};
    op.g = geom(shapes[t][0], shapes[t][1], shapes[t][2], shapes[t][3]);
    op.n = shapes[t][4];
    CHECK(coarse_sap_slots(op.g) == slots[t]);
    op.saph_cls = cls[t];
    op.saph_nst = slots[t];
    const size_t nn = (size_t)op.n * op.n, spc = op.g.vB / cls[t];
    for (int nbpc = 1; nbpc <= 2; ++nbpc)
      CHECK(coarse_sap_persist_smem(op, nbpc) > 2 * nbpc * spc * slots[t] * nn * sizeof(__half2));
    op.saph_nst = slots[t] - 1;
    op.sap_nsl = slots[t];
    CHECK(coarse_sap_persist_smem(op, 1) == 0);
    op.saph_nst = 0;
    CHECK(coarse_sap_persist_smem(op, 1) == 0);
    CHECK(!coarse_sap_persist_fits(op, 4, 4));
  }
""")


def test_fine_sap_sweep_reports_a_refused_launch(tmp_path):
    """A block that six threads per site cannot hold, and a launch that the runtime refuses: the caller learns of both."""
    run(tmp_path, r"""
  FineOp<double> op{};
  op.g = geom(8, 8, 8, 4);
  CHECK(fine_sap_sweep<double>(nullptr, nullptr, op, nullptr, 4, 1, 0, 3, nullptr) == cudaErrorInvalidConfiguration);
  op.g = geom(2, 2, 2, 2);
  CHECK(fine_sap_sweep<double>(nullptr, nullptr, op, nullptr, 4, 1, 0, 3, nullptr) != cudaSuccess);
  CHECK(fine_sap_sweep<double>(nullptr, nullptr, op, nullptr, 0, 1, 0, 3, nullptr) == cudaSuccess);
  FineOp<float> f{};
  f.g = geom(2, 2, 2, 2);
  CHECK(fine_sap_sweep<float>(nullptr, nullptr, f, nullptr, 4, 1, 0, 3, nullptr) != cudaSuccess);
""")


def test_attributes_are_set_once_per_device(tmp_path):
    """A kernel's shared-memory limit belongs to a device: each device of the process gets it once, a failure is tried
    again, and without a device nothing is marked as done."""
    run(tmp_path, r"""
  DeviceOnce once;
  int calls = 0;
  auto count = [&] { ++calls; return cudaSuccess; };
  for (int round = 0; round < 2; ++round)
    for (int device : {0, 1, 63}) CHECK(once.run(device, count) == cudaSuccess);
  CHECK(calls == 3);
  CHECK(once.run(2, [&] { ++calls; return cudaErrorInvalidValue; }) == cudaErrorInvalidValue);
  CHECK(once.run(2, count) == cudaSuccess && calls == 5);
  CHECK(once.run(64, count) == cudaSuccess && once.run(64, count) == cudaSuccess && calls == 7);
  DeviceOnce limit;
  CHECK(raise_smem_limit(limit, nullptr) != cudaSuccess);
""")


def test_setup_kernels_report_a_refused_launch(tmp_path):
    """Restriction and orthonormalisation return the status of their launch (refused here: there is no device)."""
    run(tmp_path, r"""
  Geom g = geom(2, 2, 2, 2);
  g.vA = 16;
  g.nAgg = g.V / 16;
  CHECK(restrict_op<double>(nullptr, nullptr, nullptr, g, g, true, 12, 4, 1, 0, 0, 0, nullptr, nullptr) != cudaSuccess);
  CHECK(restrict_op<float>(nullptr, nullptr, nullptr, g, g, true, 12, 4, 1, 0, 0, 0, nullptr, nullptr) != cudaSuccess);
  CHECK(orthonormalise(nullptr, g, true, 12, 4, nullptr, nullptr) != cudaSuccess);
""")


def test_residual_of_a_term_is_refused(tmp_path):
    """b - (term of D) in FP64 has no kernel: it is refused, not computed without b."""
    run(tmp_path, r"""
  FineOp<double> op{};
  op.g = geom(2, 2, 2, 2);
  const cplx<double>* b = reinterpret_cast<const cplx<double>*>(&op);
  for (int sel : {SEL_AGG_SELF, SEL_AGG_FWD, SEL_AGG_BWD, SEL_FULL}) {
    bool refused = false;
    try {
      fine_dslash<double>(nullptr, nullptr, b, op, 1, 0, sel, 0, 0, nullptr);
    } catch (const std::exception&) {
      refused = true;
    }
    CHECK(refused);
  }
""")


def test_fp64_sap_kernel_per_batch(tmp_path):
    """The FP64 SAP kernel by block, blocks per colour and batch: the faster of the two in each measured case."""
    run(tmp_path, r"""
  const Geom b4 = geom(4, 4, 4, 4), b442 = geom(4, 4, 2, 2), b43 = geom(4, 4, 4, 2), b3 = geom(3, 3, 3, 3);
  for (int blocks : {8, 16, 32, 64, 96}) CHECK(fine_sap_takes_split(b4, blocks, 1));
  CHECK(fine_sap_takes_split(b4, 8, 12) && fine_sap_takes_split(b4, 16, 12) && fine_sap_takes_split(b4, 16, 4));
  CHECK(!fine_sap_takes_split(b4, 16, 8) && !fine_sap_takes_split(b4, 32, 4) && !fine_sap_takes_split(b4, 64, 2));
  CHECK(!fine_sap_takes_split(b4, 64, 12) && !fine_sap_takes_split(b4, 128, 1) && !fine_sap_takes_split(b4, 512, 12));
  CHECK(fine_sap_takes_split(b43, 64, 2) && fine_sap_takes_split(b43, 32, 12) && !fine_sap_takes_split(b43, 32, 8));
  CHECK(fine_sap_takes_split(b442, 128, 4) && fine_sap_takes_split(b442, 512, 2) && !fine_sap_takes_split(b442, 512, 1));
  CHECK(fine_sap_takes_split(b3, 32, 8) && fine_sap_takes_split(b3, 128, 1) && !fine_sap_takes_split(b3, 128, 2));
  CHECK(fine_sap_takes_split(b3, 128, 4) && fine_sap_takes_split(b3, 128, 12) && !fine_sap_takes_split(b442, 512, 8));
  CHECK(fine_sap_takes_split(geom(4, 4, 4, 3), 192, 1) && !fine_sap_takes_split(geom(4, 4, 4, 3), 192, 8));
  CHECK(!fine_sap_takes_split(geom(3, 3, 3, 2), 192, 12) && fine_sap_takes_split(geom(3, 3, 3, 2), 192, 4));
  CHECK(fine_sap_takes_split(geom(3, 3, 3, 2), 8, 1) && !fine_sap_takes_split(geom(3, 3, 3, 2), 8, 64));
  for (int batch : {1, 2, 8, 12}) CHECK(fine_sap_takes_split(geom(2, 2, 2, 2), 2048, batch));
  CHECK(fine_sap_takes_split(geom(8, 8, 4, 4), 512, 12));
""")
