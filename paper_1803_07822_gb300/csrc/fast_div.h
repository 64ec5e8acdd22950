// Division of node indices by lattice extents as a multiplication.
#pragma once

#if defined(__CUDACC__)
#define CSLBM_DIV_HD __host__ __device__ __forceinline__
#else
#define CSLBM_DIV_HD inline
#endif

namespace cslbm {

// v / d for v < 2^28 (a context holds fewer nodes): q = v m >> s with m =
// ceil(2^s / d), s = 28 + ceil(log2 d), exact since m d - 2^s < d <= 2^(s - 28).
// (A division by a kernel argument is about twenty instructions, this three.)
struct Div {
    unsigned m, s;
};
inline Div make_div(unsigned d)
{
    unsigned b = 0;
    while ((1ull << b) < d) b++;
    Div q;
    q.s = 28 + b;
    q.m = (unsigned)(((1ull << q.s) + d - 1) / d);
    return q;
}
CSLBM_DIV_HD unsigned div_by(unsigned v, const Div& q) { return (unsigned)(((unsigned long long)v * q.m) >> q.s); }

}  // namespace cslbm
