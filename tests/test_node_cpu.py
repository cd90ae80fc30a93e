"""The node update rounds every product where the source says so: with a number
type that remembers which values are products, no sum or difference of the
update gets one (the assembler may or may not fuse those, and not alike in
every kernel that holds the update).  Products with a power of two are exact."""
import subprocess

from paper_1806_10241_gb300 import build

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "lb_internal.h"
#define LB_NODE_FN inline
namespace lbk {
namespace {
int sums = 0, with_product = 0;
struct V {
    double v;
    bool product, power;
    static V of(double x) { return V{x, false, false}; }
    static V unit(double, double x) { return lit(x); }
    static V lit(double x) { int e; return V{x, false, std::fabs(std::frexp(x, &e)) == 0.5}; }
};
V added(double v, V a, V b) { ++sums; with_product += a.product || b.product; return V{v, false, false}; }
V operator+(V a, V b) { return added(a.v + b.v, a, b); }
V operator-(V a, V b) { return added(a.v - b.v, a, b); }
V operator*(V a, V b) { return V{a.v * b.v, a.power || b.power ? a.product || b.product : true, false}; }
V fma2(V a, V b, V c) { return V{std::fma(a.v, b.v, c.v), false, false}; }
V rcp2(V a) { return V{1.0 / a.v, false, false}; }
#include "lb_node.cuh"

template <bool kScale> void run(bool explicit_src)
{
    NodeConst<double> c;
    double *p = reinterpret_cast<double *>(&c);
    for (unsigned i = 0; i < sizeof(c) / sizeof(double); ++i) p[i] = 0.3 + 0.01 * i;
    V f[9], g[5], h[5], d[5];
    for (int q = 0; q < 9; ++q) f[q] = V::of(0.1 + 0.01 * q);
    for (int q = 0; q < 5; ++q) g[q] = V::of(0.02 * q), h[q] = V::of(0.3 - 0.02 * q), d[q] = V::of(0.001 * q);
    NodeVals<V> o;
    update_node2<kScale>(c, explicit_src, geo_of(c, V::of(0.2)), f, g, h, d[0], d[1], d[2], d[3], d[4], o);
    for (int q = 0; q < NQ; ++q) with_product += o.v[q].product || !std::isfinite(o.v[q].v);
}
}
}
int main()
{
    for (int e = 0; e < 2; ++e) lbk::run<false>(e), lbk::run<true>(e);
    std::printf("%d %d\n", lbk::sums, lbk::with_product);
}
"""


def test_no_product_is_an_operand_of_a_sum(tmp_path):
    src = tmp_path / "node.cu"
    src.write_text(PROGRAM)
    subprocess.run([build.NVCC, "-std=c++17", "-I", build.CSRC, "-o", str(tmp_path / "node"), str(src)], check=True)
    out = subprocess.run([str(tmp_path / "node")], check=True, capture_output=True, text=True).stdout
    sums, with_product = map(int, out.split())
    assert sums > 200 and with_product == 0
