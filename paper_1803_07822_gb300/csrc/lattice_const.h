// Constants of a lattice (relaxation, temperature, body force) as the kernels
// take them, at both precisions.
#pragma once

namespace cslbm {

// A constant of the lattice, kept in FP64 and rounded to FP32 on the host:
// R(c) takes the one of the kernel's arithmetic.  (A conversion in the kernel
// is an FP64-pipe instruction per thread; six of them were 10 % of the FP64
// pipe's time in the FP32 gather pass, 23 % in the D2Q9 march.)
struct Cst {
    double d;
    float f;
    Cst& operator=(double v)
    {
        d = v;
        f = (float)v;
        return *this;
    }
    __host__ __device__ __forceinline__ explicit operator double() const { return d; }
    __host__ __device__ __forceinline__ explicit operator float() const { return f; }
};

}  // namespace cslbm
