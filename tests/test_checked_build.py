"""Checked builds (SSD_CHECKED=1) of the stand-alone projection: the alignment and
the bounds of its accesses are checked on the device, an access that fails is
skipped, and ssd_linear_noalloc reports it.

On the CPU: what the checks accept and refuse, at both ends of every operand, by a
small program around the kernel's own predicates.  On the GPU: a checked build of
the source beside the library passes its checks over the kernel's edges and gives
the same bits.
"""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_08168_gb300", "csrc")
NVCC = ["nvcc", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-DSSD_CHECKED", "-I", CSRC,
        "-I", os.path.join(ROOT, "include")]
STUB = 'namespace ssd { int set_last_error(int code, const char*) { return code; } }\n'
SOURCE = '#include "gemm.cu"\n#include <cstdio>\n' + STUB + r"""
using namespace ssd;
int main() {
    int bad = 0, id = 0;
    auto expect = [&](bool got, bool want) { ++id; if (got != want) { printf("check %d: %d\n", id, got); ++bad; } };
    const int sizes[][3] = {{1, 16, 1}, {100, 528, 3}, {129, 80, 16}, {32000, 4096, 4}};
    for (auto& z : sizes) {
        LinearArgs a{};
        a.N = z[0]; a.K = z[1]; a.M = z[2];
        a.w = (const bf16*)0x10000000; a.x = (const float*)0x40000000; a.y = (float*)0x50000000;
        const size_t W = (size_t)a.N * a.K, X = (size_t)a.M * a.K, Y = (size_t)a.M * a.N;
        expect(a.weights_in(a.w, 8), true);
        expect(a.weights_in(a.w + W - 8, 8), true);
        expect(a.weights_in(a.w + W - 16, 16), true);
        expect(a.weights_in(a.w + W, 8), false);
        expect(a.weights_in(a.w + W - 8, 16), false);
        expect(a.weights_in(a.w - 8, 8), false);
        expect(a.weights_in(a.w + 1, 8), false);
        expect(a.inputs_in(a.x, 8), true);
        expect(a.inputs_in(a.x + X - 8, 8), true);
        expect(a.inputs_in(a.x + X - 4, 8), false);
        expect(a.inputs_in(a.x - 4, 8), false);
        expect(a.inputs_in(a.x + 2, 8), false);
        expect(a.output_in(a.y), true);
        expect(a.output_in(a.y + Y - 1), true);
        expect(a.output_in(a.y + Y), false);
        expect(a.output_in(a.y - 1), false);
    }
    if (!bad) printf("ok\n");
    return bad;
}
"""


def test_what_the_checks_accept(tmp_path):
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(SOURCE)
    subprocess.check_call([*NVCC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_every_global_access_of_the_kernel_is_checked():
    src = open(os.path.join(CSRC, "gemm.cu")).read()
    kernel = src[src.index("ld_weights("):src.index("size_t linear_smem_bytes")]
    for access in ('asm volatile("ld.global.L1', 'asm volatile("cp.async.bulk', "split8(__ldcg", "a.y[(size_t)m"):
        at = kernel.index(access)
        assert "SSD_GUARD(" in kernel[:at].rstrip().rsplit("\n", 1)[-1], access


@pytest.mark.gpu
def test_checked_projection_passes_and_gives_the_same_bits(tmp_path):
    torch = pytest.importorskip("torch")
    import paper_2309_08168_gb300 as ssd
    src, so = tmp_path / "checked.cu", tmp_path / "libchecked.so"
    src.write_text('#include "gemm.cu"\n' + STUB)
    subprocess.check_call([*NVCC, "-O3", "-shared", "-Xcompiler", "-fPIC", str(src), "-o", str(so)])
    checked = ctypes.CDLL(str(so)).ssd_linear_noalloc
    checked.argtypes = ssd.lib.ssd_linear_noalloc.argtypes
    checked.restype = ctypes.c_int
    for M, K, N in [(1, 16, 1), (3, 48, 127), (9, 272, 128), (16, 528, 300), (2, 1040, 257), (5, 4112, 640), (1, 2064, 39000)]:
        g = torch.Generator(device="cuda").manual_seed(M * K + N)
        w = torch.empty(N, K, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=g)
        x = torch.randn(M, K, device="cuda", generator=g)
        y, z = torch.empty(M, N, device="cuda"), torch.empty(M, N, device="cuda")
        stream = torch.cuda.current_stream().cuda_stream
        ssd.ssd_linear_noalloc(w, x, y, N, K, M, stream)
        assert checked(w.data_ptr(), x.data_ptr(), z.data_ptr(), N, K, M, stream) == ssd.SSD_OK
        assert torch.equal(y, z)
