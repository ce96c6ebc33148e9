"""Which products the tensor-core GEMMs and their epilogues take: the host-side rules (dm_internal.h), compiled and run without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"

PROGRAM = r"""
#include <cstdio>
#include "dm_internal.h"
using namespace dm;
int main() {
    GemmArgs g{};
    char *base = reinterpret_cast<char *>(0x100000);          // (addresses only: nothing is read)
    float *f = reinterpret_cast<float *>(0x200000);
    g.A = base; g.lda = 64; g.B = base; g.ldb = 64; g.C = base; g.ldc = 32; g.in_dtype = DM_BF16; g.c_dtype = DM_F32; g.M = 300; g.N = 32; g.K = 64;
    auto row = [&](const char *name, GemmArgs a) { std::printf("%s %d %d %d %d\n", name, gemm_tensor_ok(a), gemm_tma_io(a), gemm_sum_ok(a, g), gemm_sum_ok(g, a)); };
    GemmArgs a = g;
    row("plain", a);
    a = g; a.c_dtype = DM_BF16; row("bf16_out", a);
    a = g; a.addend = f; a.ld_add = 32; row("addend", a);
    a = g; a.addend = f; a.ld_add = 30; row("addend_ragged", a);
    a = g; a.c_dtype = DM_BF16; a.addend = f; a.ld_add = 32; row("bf16_out_addend", a);
    a = g; a.ldc = 33; row("ragged_out", a);
    a = g; a.rs_ssq = f; a.rs_n = 8; row("ssq", a);
    a = g; a.rs_ssq = f + 1; a.rs_n = 8; row("ssq_off_vectors", a);
    a = g; a.rs_ssq = f + 1; a.rs_n = 6; row("ssq_off_scalars", a);
    a = g; a.addend = f + 1; a.ld_add = 32; row("addend_off", a);
    a = g; a.lda = 60; row("operand_ragged", a);
    a = g; a.col_bias = f; row("bias", a);
    a = g; a.gelu = 1; row("gelu", a);
    a = g; a.silu_cols = 8; row("silu", a);
    a = g; int n; a.m_dev = &n; row("device_rows", a);
    a = g; a.K = 128; row("other_k", a);
}
"""

# name: operands and epilogue pointers, output through TMA, as first and as second (the one with the output) product of a sum
WANT = {
    "plain": (1, 1, 1, 1), "bf16_out": (1, 1, 1, 1), "addend": (1, 1, 1, 1), "addend_ragged": (1, 0, 1, 0),
    "bf16_out_addend": (1, 1, 1, 0),        # a single product stores it in halves; the sum's epilogues do not
    "ragged_out": (1, 0, 1, 0), "ssq": (1, 1, 1, 1),
    "ssq_off_vectors": (0, 1, 0, 0), "ssq_off_scalars": (1, 1, 1, 1),      # 16-byte alignment where rows are read as float4, none where they are not
    "addend_off": (0, 1, 0, 0), "operand_ragged": (0, 1, 0, 0),
    "bias": (1, 1, 0, 0), "gelu": (1, 1, 0, 0), "silu": (1, 1, 0, 0),      # the sum's epilogues have no bias and no activation
    "device_rows": (1, 1, 0, 0), "other_k": (1, 1, 0, 0),
}


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA_INCLUDE), reason="needs g++ and the CUDA headers")
def test_gemm_rules(tmp_path):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2511_15927_b200", "csrc"), "-I", CUDA_INCLUDE,
                    str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    got = {line.split()[0]: tuple(int(v) for v in line.split()[1:]) for line in out.splitlines()}
    assert got == WANT
