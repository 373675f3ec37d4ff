"""The width in which the solvers sum (no GPU): the text of a kernel is compiled as C++, its threads run
one after another, and the partial sums are compared with the exact sum of what the kernel rounds --
FP32 products, whose sums are FP64 wherever a thread per element would sum them so."""
import ctypes
import math
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_07392_gb300", "csrc")

SHIM = r"""
#include <cstdint>
#include <cstring>
#include <cstddef>
#define __global__
#define __device__
#define __restrict__
#define __launch_bounds__(...)
struct Dim { int x, y, z; };
static Dim blockIdx, blockDim, gridDim, threadIdx;
struct float4 { float x, y, z, w; };
template <class T> struct V3 { T *p[3]; };
static const size_t kPartComp = (1 << 20) / 3;
static unsigned __float_as_uint(float x) { unsigned u; memcpy(&u, &x, 4); return u; }
static double __hiloint2double(int hi, int lo)
{
    uint64_t u = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
    double d;
    memcpy(&d, &u, 8);
    return d;
}
static double g_sum;   // of the block's threads, which run one after another
static double block_sum_flat(double v) { g_sum = threadIdx.x ? g_sum + v : v; return g_sum; }
"""


def _source(name):
    return open(os.path.join(CSRC, name)).read()


def _function(text, head):
    """The function whose declaration matches head, to its closing brace in the first column."""
    m = re.search(head, text)
    assert m, head
    return text[m.start():text.index("\n}\n", m.start()) + 3]


@pytest.fixture(scope="module")
def kernels(tmp_path_factory):
    d = tmp_path_factory.mktemp("kernels")
    solvers, bits, head = _source("solvers.cu"), _source("fpbits.cuh"), _source("ebv_internal.cuh")
    dot = re.sub(r"if \(threadIdx\.x == 0\) (part\[)", r"if (threadIdx.x == blockDim.x - 1) \1",
                 _function(solvers, r"__global__ void __launch_bounds__\(256\) k_dot32\("))
    src = SHIM
    src += re.search(r"constexpr int kReduceBlocks = \d+;", head).group(0) + "\n"
    src += "\n".join(re.findall(r"^constexpr int kWideDot = [^;]*;", solvers, flags=re.M)) + "\n"
    src += _function(bits, r"__device__ inline double f32_to_f64\(")
    src += "\n".join(re.findall(r"^__device__ inline double dot_term\(.*$", solvers, flags=re.M)) + "\n" + dot + r"""
extern "C" int blocks() { return kReduceBlocks; }
extern "C" void dot(const float *a, const float *b, int n, int nb, double *part)
{
    V3<const float> av = {{a, a, a}}, bv = {{b, b, b}};
    blockDim = {256, 1, 1};
    gridDim = {nb, 1, 1};
    for (int q = 0; q < nb; q++)
        for (int t = 0; t < 256; t++) {
            blockIdx = {q, 0, 0};
            threadIdx = {t, 0, 0};
            k_dot32(av, bv, n, part);
        }
}
"""
    cpp, lib = d / "k.cpp", d / "k.so"
    cpp.write_text(src)
    # (no contraction: a product that is added in FP64 is rounded to FP32 first)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fno-strict-aliasing", "-shared", "-fPIC", "-o", str(lib), str(cpp)], check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1024, 1025, 4913, 35937, 274625, 1245183])
def test_small_dot_sums_in_fp64(kernels, n):
    rng = np.random.Generator(np.random.PCG64(n))
    a, b = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    nb = min(kernels.blocks(), (n // 4 + 255) // 256 + 1)   # (v4blocks)
    part = np.full(nb, np.nan)
    ptr = lambda x, t: x.ctypes.data_as(ctypes.POINTER(t))
    kernels.dot(ptr(a, ctypes.c_float), ptr(b, ctypes.c_float), n, nb, ptr(part, ctypes.c_double))
    prod = (a * b).astype(np.float64)
    # at most n FP64 roundings of partial sums no larger than sum |a b|
    assert abs(math.fsum(part) - math.fsum(prod)) <= n * 2.0 ** -53 * math.fsum(abs(prod))


def test_cluster_vcycle_sums_its_dot_in_fp64():
    """r.z of a grid that the cluster kernel holds whole: each thread's sum, the warps' and the block's."""
    text = _function(_source("solvers.cu"), r"__global__ void __cluster_dims__\(kCvCtas, 1, 1\)[^;{]*\bk_cc_coarse_vcycle\(")
    assert re.findall(r"\b(\w+) dot = ", text) == ["double"]
    adds = re.findall(r"\bdot \+= ([^;]*);", text)
    assert adds == ["dot_term(w.b[c0 * w.cap + m], x0) + dot_term(w.b[(1 - c0) * w.cap + m], x1)",
                    "__shfl_down_sync(0xffffffffu, dot, o)"]
    assert re.search(r"\bps\[tid >> 5\] = dot;", text) and re.search(r"double \*bs = .*\*ps = reinterpret_cast<double \*>", text)


def test_listed_nodes_residual_norm_is_fp64():
    """|r|^2 of the nodes that a nodal pass lists: FP64 squares of the stored FP32 residuals, FP64 sums
    (k_nd_pass runs this mode with T = double; the march's own nodes are summed in FP32 within a warp)."""
    solvers = _source("solvers.cu")
    text = _function(solvers, r"__global__ void __launch_bounds__\(NT_T\) k_nd_pass\(")
    lists = text[text.index("if (listed) {"):text.index("    } else {\n        __shared__ T sx")]
    assert re.findall(r"\bvr? = T\(r\) \* T\(r\);", lists) == ["v = T(r) * T(r);"] and "vr" not in lists
    assert "kMode == ND_RES32 && !listed ? block_sum3_t<float>(vr) : block_sum3_t<T>(v)" in text
    assert re.findall(r"nd_pass<(\w+), ND_RES32>", solvers) == ["double"]


def test_krylov_apply_is_chosen_by_one_components_grid():
    """The vectorised FP32 apply sums p.q of eight cells a thread in FP32, the other one of two: a joint
    solve takes the one that each component's own solve would take."""
    text = _source("solvers.cu")
    m = re.search(r"bool vec32\(\) const\s*\{(.*?)\n    \}", text, flags=re.S)
    assert "nblocks3(apply4_grid(H->lv[0].g)) >= kVecMinBlocks" in m.group(1)
    assert not re.search(r"\bnc\b", m.group(1))


def test_vectorised_apply_sums_no_more_fp32_terms_than_the_other():
    """p.q: a thread of k_cc_apply_dot adds two FP32 terms and its warp 32 of those sums, 64 terms and seven
    additions deep (one fused with the first product).  A thread of k_cc_apply4 has eight: two to each of
    four sums, those pairwise, and then no more than 8 lanes in FP32."""
    text = _source("solvers.cu")
    k = _function(text, r"__global__ void __launch_bounds__\(256\) k_cc_apply4\(")
    assert "float v[4] = {0.f, 0.f, 0.f, 0.f};" in k and "v[e] += pc[e] * y[e];" in k
    assert "block_sum8((v[0] + v[1]) + (v[2] + v[3]))" in k
    b = _function(text, r"__device__ inline double block_sum8\(float v\)")
    steps = re.findall(r"for \(int o = (\d+); o > 0; o >>= 1\) (\w+) \+= __shfl_down_sync", b)
    assert steps == [("4", "v"), ("16", "r")] and "__shared__ double sm[32];" in b and "double r = 0.0;" in b
    depth = 2 + 2 + int(steps[0][0]).bit_length()
    assert 8 * 2 * int(steps[0][0]) <= 2 * 32 and depth <= 2 + 5
