"""Rules of csrc/rules.h, compiled with the host compiler: no GPU, no CUDA."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_10523_gb300", "csrc")


def run(tmp_path, body, extra=()):
    src = tmp_path / "t.cpp"
    src.write_text('#include <cstdio>\n#include "rules.h"\nusing namespace tnq;\nint main() {\n%s\nreturn 0;\n}\n' % body)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, *extra, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_ranges_overlap(tmp_path):
    cases = [(0, 8, 8, 8, 0), (8, 8, 0, 8, 0), (0, 9, 8, 8, 1), (8, 8, 0, 9, 1), (0, 64, 16, 8, 1), (16, 8, 0, 64, 1),
             (0, 8, 0, 8, 1), (0, 8, 64, 8, 0)]
    body = "\n".join(f'printf("%d\\n", ranges_overlap((void*){0x1000 + p}, {n}, (void*){0x1000 + q}, {m}));'
                     for p, n, q, m, _ in cases)
    assert run(tmp_path, body) == [str(c[4]) for c in cases]


def test_kernels_reach_own_device_and_managed_memory_only(tmp_path):
    """Device memory of another GPU is not addressed from kernels, host memory neither."""
    cases = [(1, 0, 0, 0, 1), (1, 0, 1, 1, 1), (1, 0, 1, 0, 0), (1, 0, 0, 1, 0), (0, 1, 0, 1, 1), (0, 0, 0, 0, 0)]
    body = "\n".join(f'printf("%d\\n", kernels_reach({d}, {m}, {at}, {ctx}));' for d, m, at, ctx, _ in cases)
    assert run(tmp_path, body) == [str(c[4]) for c in cases]


def test_buffers_are_asked_for_the_context_device():
    """Every caller buffer that kernels may address is classified by its device
    against the context's, not by being device memory alone."""
    src = open(os.path.join(CSRC, "executor.cu")).read()
    assert "kernels_reach(dev, managed, a.device, ctx->device)" in src
    assert src.count("cudaPointerGetAttributes") == 1 and "is_device_ptr" not in src


def test_aligned(tmp_path):
    cases = [(16, (0x1000, 0x2000, 0), 1), (16, (0x1008, 0x2000, 0), 0), (16, (0x1000, 0x2008, 0), 0),
             (16, (0x1000, 0x2000, 0x3008), 0), (8, (0x1008, 0x2000, 0x3010), 1), (8, (0x1004, 0x2000, 0), 0)]
    body = "\n".join('printf("%%d\\n", aligned(%d, (void*)%d, (void*)%d, (void*)%d));' % (n, *p) for n, p, _ in cases)
    assert run(tmp_path, body) == [str(c[2]) for c in cases]


def test_sixteen_byte_accesses_to_caller_tensors_ask_first():
    """The vectorised permute and the tensor map over an operand read in place are
    the two places a caller's A, B or C meets accesses wider than 8 bytes beside
    the pair loads of the gather and tall-skinny kernels."""
    def src(name):
        return open(os.path.join(CSRC, name)).read()

    assert "if (!aligned(16, src, dst0, dst1)) return false;" in src("kernels.cu")
    assert "!perm_b && aligned(16, b_src)" in src("executor.cu")
    for name in ("skinny.cu", "gemm_tc_rows.cu"):
        assert "(reinterpret_cast<uintptr_t>(Gsrc) & 15) == 0" in src(name)


def test_workspace_base(tmp_path):
    """The first multiple of 256, within the bytes the sizes asked for add."""
    at = [0x1000, 0x1001, 0x1008, 0x10ff, 0x1100]
    body = "\n".join(f'printf("%zu\\n", (size_t)workspace_base((void*){p}));' for p in at)
    assert run(tmp_path, body) == [str((p + 255) // 256 * 256) for p in at]
    body = 'printf("%zu\\n", kWorkspaceAlign);'
    assert run(tmp_path, body) == ["256"]


def test_shared_memory_limits_are_fixed_and_per_device():
    """Dynamic shared-memory limits go through once_per_device (a process-wide flag
    would leave a second device at the default limit) with a size that does not
    depend on the call (two threads could lower each other's limit)."""
    import glob
    import re
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = open(f).read()
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize", src):
            at = src.rfind("once_per_device(", 0, m.start())
            end = src.find("\n}", at)
            assert at >= 0 and m.start() < end, (f, src.count("\n", 0, m.start()) + 1)
    prep = open(os.path.join(CSRC, "gemm_tc.cu")).read()
    assert prep.count("call_once") == 1  # the driver entry point: one per process


def test_long_k_steps_with_many_rows_take_the_rows_kernel(tmp_path):
    """The lines of splitk.h at the sizes they were measured at: (permuted, log2 M, N,
    H, K) of steps the long-K and the one-launch kernel ran up to 3 and 17 times
    slower than the rows kernel, and of steps that stay where they are."""
    faster = [(0, 3, 20, 0, 6, 1), (1, 3, 20, 0, 6, 1), (0, 3, 14, 0, 6, 0), (1, 3, 15, 0, 6, 0), (0, 1, 10, 9, 6, 1),
              (0, 5, 17, 0, 8, 1), (1, 5, 19, 0, 8, 0), (0, 3, 5, 14, 6, 0), (0, 0, 20, 0, 7, 0), (0, 3, 20, 0, 11, 0),
              (0, 6, 20, 0, 6, 0), (0, 3, 20, 0, 5, 0)]
    ordered = [(0, 4, 14, 0, 10, 1), (1, 4, 12, 0, 12, 1), (0, 3, 6, 0, 17, 1), (1, 3, 10, 0, 12, 0), (0, 1, 8, 0, 18, 1),
               (1, 1, 8, 0, 18, 0), (0, 0, 14, 0, 12, 0), (0, 2, 4, 6, 14, 0)]
    src = "\n".join(f'printf("%d\\n", rows_faster({p}, {m}, {n}, {h}, {k}));' for p, m, n, h, k, _ in faster)
    src += "\n" + "\n".join(f'printf("%d\\n", rows_ordered({p}, {m}, {n}, {h}, {k}));' for p, m, n, h, k, _ in ordered)
    got = run(tmp_path, src, extra=("-include", os.path.join(CSRC, "splitk.h")))
    assert got == [str(x[-1]) for x in faster + ordered]
