// lbm_ordered.cuh -- FP64 arithmetic whose roundings the source fixes.
#pragma once
#include <cuda_runtime.h>

namespace tlv {

using ::expm1;  // the overloads below add to these
using ::fabs;
using ::fmax;
using ::hypot;
using ::log1p;

// A double whose sums, products and quotients round as written, whatever the
// code around them: a product that is one term of a sum or difference goes
// into a fused multiply-add (the right one, if both terms are products), any
// other is rounded by itself. Plain doubles leave that choice to the compiler,
// which makes it anew in every kernel that inlines the code. The sums are the
// intrinsics that the compiler never contracts, so a plain product can only
// meet them rounded, and one with a constant 1 (a seed of Dual) still folds.
struct Ordered {
    double v;
    Ordered() = default;
    __device__ __forceinline__ explicit Ordered(double x) : v(x) {}
};

// a product before it is rounded
struct OrderedProduct {
    double a, b;
    __device__ __forceinline__ operator Ordered() const { return Ordered(a * b); }
};

#define TLV_OP __device__ __forceinline__
TLV_OP Ordered operator-(Ordered x) { return Ordered(-x.v); }
TLV_OP Ordered operator+(Ordered x, Ordered y) { return Ordered(__dadd_rn(x.v, y.v)); }
TLV_OP Ordered operator-(Ordered x, Ordered y) { return Ordered(__dsub_rn(x.v, y.v)); }
TLV_OP Ordered operator/(Ordered x, Ordered y) { return Ordered(__ddiv_rn(x.v, y.v)); }
TLV_OP OrderedProduct operator*(Ordered x, Ordered y) { return {x.v, y.v}; }
TLV_OP OrderedProduct operator-(OrderedProduct p) { return {-p.a, p.b}; }
TLV_OP Ordered operator+(OrderedProduct p, Ordered y) { return Ordered(__fma_rn(p.a, p.b, y.v)); }
TLV_OP Ordered operator+(Ordered x, OrderedProduct p) { return p + x; }
TLV_OP Ordered operator-(OrderedProduct p, Ordered y) { return p + -y; }
TLV_OP Ordered operator-(Ordered x, OrderedProduct p) { return -p + x; }
TLV_OP Ordered operator+(OrderedProduct p, OrderedProduct q) { return Ordered(p) + q; }
TLV_OP Ordered operator-(OrderedProduct p, OrderedProduct q) { return Ordered(p) - q; }
TLV_OP OrderedProduct operator*(OrderedProduct p, Ordered y) { return Ordered(p) * y; }
TLV_OP OrderedProduct operator*(Ordered x, OrderedProduct p) { return x * Ordered(p); }
TLV_OP OrderedProduct operator*(OrderedProduct p, OrderedProduct q) { return Ordered(p) * Ordered(q); }
TLV_OP Ordered operator/(OrderedProduct p, Ordered y) { return Ordered(p) / y; }
TLV_OP Ordered operator/(Ordered x, OrderedProduct p) { return x / Ordered(p); }
TLV_OP Ordered &operator+=(Ordered &x, Ordered y) { return x = x + y; }
TLV_OP Ordered &operator+=(Ordered &x, OrderedProduct p) { return x = x + p; }
TLV_OP Ordered &operator*=(Ordered &x, Ordered y) { return x = x * y; }
TLV_OP bool operator<(Ordered x, Ordered y) { return x.v < y.v; }
TLV_OP bool operator>(Ordered x, Ordered y) { return x.v > y.v; }
TLV_OP bool operator<=(Ordered x, Ordered y) { return x.v <= y.v; }
TLV_OP Ordered fabs(Ordered x) { return Ordered(::fabs(x.v)); }
TLV_OP Ordered fmax(Ordered x, Ordered y) { return Ordered(::fmax(x.v, y.v)); }
TLV_OP Ordered hypot(Ordered x, Ordered y) { return Ordered(::hypot(x.v, y.v)); }
TLV_OP Ordered log1p(Ordered x) { return Ordered(::log1p(x.v)); }
TLV_OP Ordered expm1(Ordered x) { return Ordered(::expm1(x.v)); }
TLV_OP Ordered rcp_rn(Ordered x) { return Ordered(__drcp_rn(x.v)); }
#undef TLV_OP

} // namespace tlv
