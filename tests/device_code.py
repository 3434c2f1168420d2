"""Device functions of the CUDA sources compiled by g++ for the host, so that a test runs the code itself
rather than a copy of it. Intrinsics are stood in for by the IEEE operation they name."""
import ctypes
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_12466_gb300", "csrc")

SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
template <class A, class B> static A bits_as(B b) { static_assert(sizeof(A) == sizeof(B), ""); A a; std::memcpy(&a, &b, sizeof a); return a; }
static long long __double_as_longlong(double v) { return bits_as<long long>(v); }
static double __longlong_as_double(long long v) { return bits_as<double>(v); }
static unsigned __float_as_uint(float v) { return bits_as<unsigned>(v); }
static float __uint_as_float(unsigned v) { return bits_as<float>(v); }
static double __hiloint2double(int hi, int lo) { return bits_as<double>(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo); }
static double __dadd_rn(double a, double b) { return a + b; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static float __int2float_rn(int v) { return (float)v; }
static float __uint2float_rn(unsigned v) { return (float)v; }
static int __float2int_rz(float v) { return (int)v; }
static int __float2int_rn(float v) { return (int)std::nearbyint(v); }
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
using std::min;
using std::max;
// rcp.approx.ftz.f32: within one unit of the last place, taken as off by one, up or down by the operand's last bit
static float rcp_approx(float x) { return std::nextafterf(1.0f / x, (__float_as_uint(x) & 1u) ? INFINITY : 0.0f); }
"""


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def definition(text, start):
    """The definition that begins with `start`, up to its closing brace (and semicolon); a template line above it
    comes along."""
    at = text.index(start)
    line = text.rindex("\n", 0, at) + 1
    above = text.rindex("\n", 0, line - 1) + 1
    begin = above if text[above:line].startswith("template") else line
    depth, i = 0, text.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            break
    end = i + 1 if text[i:i + 1] == ";" else i
    return text[begin:end] + "\n"


def compile_host(tmp, body):
    """A shared object of SHIM and `body`, loaded."""
    body = re.sub(r'asm\("rcp\.approx\.ftz\.f32 [^"]*" : "=f"\((\w+)\) : "f"\(([\w.]+)\)\);', r"\1 = rcp_approx(\2);", body)
    src, lib = os.path.join(str(tmp), "dev.cpp"), os.path.join(str(tmp), "dev.so")
    with open(src, "w") as f:
        f.write(SHIM + body)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-o", lib, src], check=True)
    return ctypes.CDLL(lib)
