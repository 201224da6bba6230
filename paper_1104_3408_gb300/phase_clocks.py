"""Per-CTA phase clocks of the tensor-core operator kernel (a diagnostic).

Builds a copy of the library whose persistent kernel k_op_ws sums, for every CTA of the
d_theta + d_phi launch, SM clock64 intervals of each role: the MMA thread's
waits (operator copies, slices, accumulators) and its issue, a producer warp's
wait for a free stage, slicing and load issue, an epilogue warp's wait for
products, its reading of the accumulators and the rest of its stores.  Runs
RK4 steps of a shell with it and prints the means over the CTAs of the last
such launch, per work item.  The copy lives under the package's build folder;
the library itself is unchanged.

    python -m paper_1104_3408_gb300.phase_clocks [--mhz F] [--shape NR,NTHETA]

(F: the SM clock used to turn cycles into microseconds, default 2070.)
"""

import argparse
import ctypes
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
OUT = os.path.join(PKG, "_lib", "phase_clocks")

NAMES = ["mma: wait for operator copies", "mma: wait for slices", "mma: wait for accumulators",
         "mma: issue of the products", "mma: whole loop", "producer: wait for a free stage", "producer: slicing",
         "producer: next k-step's loads issued", "epilogue: wait for products", "epilogue: accumulators read",
         "epilogue: last rows folded and stored", "set-up"]


# (text of the kernel, text with the clocks) pairs applied to a copy of csrc/ops.cu
_PATCHES = [
    ("// STAGE: the launch is d_r (one operator class, all rows in one group), whose",
     "__device__ unsigned long long g_instr[1024][16];\n#define CK clock64()\n"
     "// STAGE: the launch is d_r (one operator class, all rows in one group), whose"),
    ("  const int total = B.first[B.nclass];\n",
     "  const int total = B.first[B.nclass];\n  const long long c_entry = CK;\n  long long ins[12] = {0};\n"),
    ("  const uint32_t tm = tmem_base;\n", "  const uint32_t tm = tmem_base;\n  const long long c_setup = CK;\n"),
    ("      if (use > 0 && !(ok = __all_sync", "      const long long p0_ = CK;\n      if (use > 0 && !(ok = __all_sync"),
    ("      unsigned char* xs = smtc + s * C::kStage + xoff;\n",
     "      unsigned char* xs = smtc + s * C::kStage + xoff;\n      const long long p1_ = CK;\n"),
    ("      bar_arrive(&xfull[s]);\n", "      bar_arrive(&xfull[s]);\n      const long long p2_ = CK;\n"),
    ("      if (STAGE != 2 && have) gather16<FI>(B.a[x.cls], col, ks * 16, w);\n    }\n",
     "      if (STAGE != 2 && have) gather16<FI>(B.a[x.cls], col, ks * 16, w);\n      ins[5] += p1_ - p0_;\n      ins[6] += p2_ - p1_;\n"
     "      ins[7] += CK - p2_;\n    }\n"),
    ("        const int ai = n % A, ause = n / A;\n        if (ause > 0",
     "        const int ai = n % A, ause = n / A;\n        const long long a0_ = CK;\n        if (ause > 0"),
    ("        const uint32_t ta = tm + ai * 256;\n        for (int ks",
     "        const uint32_t ta = tm + ai * 256;\n        ins[2] += CK - a0_;\n        for (int ks"),
    ("          ok = pipe_wait(&wfull[s], ph, B.wait_ns) && pipe_wait(&xfull[s], ph, B.wait_ns);\n",
     "          const long long m0_ = CK;\n          ok = pipe_wait(&wfull[s], ph, B.wait_ns);\n          const long long m1_ = CK;\n"
     "          ok = ok && pipe_wait(&xfull[s], ph, B.wait_ns);\n          const long long m2_ = CK;\n"
     "          ins[0] += m1_ - m0_;\n          ins[1] += m2_ - m1_;\n"),
    ("          tc::commit(&empty[s]);\n", "          tc::commit(&empty[s]);\n          ins[3] += CK - m2_;\n"),
    ("      tc::bar_wait(&drained, 0, kTcWaitNs);\n", "      tc::bar_wait(&drained, 0, kTcWaitNs);\n      ins[4] = CK - c_setup;\n"),
    ("      ok = __all_sync(0xffffffffu, pipe_wait(&accfull[ai], ause & 1, B.wait_ns));\n",
     "      const long long e0_ = CK;\n      ok = __all_sync(0xffffffffu, pipe_wait(&accfull[ai], ause & 1, B.wait_ns));\n"
     "      long long e1_ = CK, e2_ = 0;\n"),
    ("          // the accumulators are read: the next item may overwrite them\n",
     "          e2_ = CK;\n          // the accumulators are read: the next item may overwrite them\n"),
    ("      if constexpr (STAGE != 0) {\n        // d_r: a quarter",
     "      ins[8] += e1_ - e0_;\n      if (e2_) ins[9] += e2_ - e1_, ins[10] += CK - e2_;\n"
     "      if constexpr (STAGE != 0) {\n        // d_r: a quarter"),
    ("  ok = __syncthreads_and(ok);\n",
     "  if (!STAGE && B.sum6 && B.nclass == 2 && lane == 0) {\n    const int lo = warp == kMmaWarp ? 0 : warp == kProdWarp0 ? 5 : warp == 0 ? 8 : 12;\n"
     "    const int hi = warp == kMmaWarp ? 5 : warp == kProdWarp0 ? 8 : warp == 0 ? 11 : 12;\n"
     "    for (int q = 0; q < 11; ++q)\n      if (q >= lo && q < hi) g_instr[blockIdx.x][q] = (unsigned long long)ins[q];\n"
     "    if (warp == 0) {\n      g_instr[blockIdx.x][11] = (unsigned long long)(c_setup - c_entry);\n"
     "      g_instr[blockIdx.x][12] = (total - blockIdx.x + gridDim.x - 1) / gridDim.x;\n    }\n  }\n"
     "  ok = __syncthreads_and(ok);\n"),
    ("// ---------------------------------------------------------------------------\n// Host side\n",
     "extern \"C\" __attribute__((visibility(\"default\"))) int cffyn_instr_read(unsigned long long* host) {\n"
     "  return (int)cudaMemcpyFromSymbol(host, g_instr, sizeof(g_instr));\n}\n"
     "// ---------------------------------------------------------------------------\n// Host side\n"),
]


def _patched_ops(src):
    s = src
    for a, b in _PATCHES:
        if a not in s:
            raise RuntimeError("the operator kernel changed: the phase-clock patch no longer applies")
        s = s.replace(a, b, 1)
    return s


def build():
    """Builds the instrumented copy (libcffyn_phase_clocks.so) and returns its path."""
    from . import _build
    if os.path.isdir(OUT):
        shutil.rmtree(OUT)
    csrc = os.path.join(OUT, "pkg", "csrc")
    shutil.copytree(_build.CSRC, csrc)
    shutil.copytree(os.path.join(ROOT, "include"), os.path.join(OUT, "include"))
    p = os.path.join(csrc, "ops.cu")
    with open(p) as fh:
        s = _patched_ops(fh.read())
    with open(p, "w") as fh:
        fh.write(s)
    nvcc = _build._nvcc()
    objs = []
    procs = []
    for src in _build.SOURCES:
        obj = os.path.join(OUT, src.replace(".cu", ".o"))
        objs.append(obj)
        procs.append(subprocess.Popen([nvcc] + _build.ARCH + _build.FLAGS +
                                      ["-I", os.path.join(OUT, "include"), "-c", os.path.join(csrc, src),
                                       "-o", obj]))
    if any(q.wait() != 0 for q in procs):
        raise RuntimeError("nvcc failed on the instrumented copy")
    lib = os.path.join(OUT, "libcffyn_phase_clocks.so")
    cuda_lib = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    subprocess.check_call([nvcc] + _build.ARCH + ["-shared", "-o", lib] + objs +
                          ["-L", cuda_lib, "-lcufft", "-Xlinker", "-rpath", "-Xlinker", cuda_lib,
                           "-lcudart_static", "-lrt", "-lpthread", "-ldl"])
    return lib


def report(buf, shape, mhz):
    """The table of the clocks read back (a row per CTA: cycles of NAMES, then its
    items; zero rows: CTAs that recorded nothing)."""
    import numpy as np
    rec = buf[buf[:, 12] > 0].astype(np.float64)
    name = "x".join(str(n) for n in shape)
    if not len(rec):
        raise RuntimeError(f"no clocks recorded: the d_theta + d_phi launch of the {name} shell has too few items "
                           "for the persistent kernel (runs_persistent in csrc/ops.cu)")
    items = rec[:, 12]
    lines = [f"d_theta + d_phi launch of the {name} shell: {len(rec)} CTAs, {items.mean():.2f} items each; "
             f"microseconds at {mhz:.0f} MHz per item (mean, p10, p90)"]
    for q, nm in enumerate(NAMES):
        us = rec[:, q] / mhz / (items if q < 11 else 1.0)
        lines.append(f"{nm:45s} {us.mean():7.2f} {np.percentile(us, 10):7.2f} {np.percentile(us, 90):7.2f}")
    return "\n".join(lines)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--mhz", type=float, default=2070.0)
    ap.add_argument("--shape", default="33,48", help="n_r,n_theta")
    args = ap.parse_args()
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    import numpy as np
    import torch

    from . import cffyn, inputs
    lib = cffyn.load(build())
    lib.cffyn_instr_read.argtypes = [ctypes.c_void_p]
    n_r, N = (int(v) for v in args.shape.split(","))
    J, L = 2 * N, N - 2
    sh = cffyn.Shell(n_r, N, J, 1.8, 11.0, L)
    u = torch.from_numpy(inputs.kerr_schild_state(n_r, N, J, 1.8, 11.0, amp=1e-4, ell=4, seed=0)).cuda()
    sh.init_gauge_from_state(u)
    for _ in range(3):
        sh.rk4_step(u, 0.0, 1)
    torch.cuda.synchronize()
    buf = np.zeros((1024, 16), dtype=np.uint64)
    if lib.cffyn_instr_read(buf.ctypes.data) != 0:
        raise RuntimeError("reading the phase clocks failed")
    sh.destroy()
    print(report(buf, (n_r, N, J), args.mhz))


if __name__ == "__main__":
    main()
