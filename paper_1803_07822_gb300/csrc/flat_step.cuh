// LBM step as two flat passes per time step.
//
// The forcing moment C^ij (Eq. forcing-C) needs the lattice gradient of
// rho u at time t on the 18 neighbours of every node (App. D).  The first
// pass forms rho u of every node (one float4 per node, a field small enough
// to stay in L2); the second pass steps every node independently: pull
// gather, moments, stress, gradient from the neighbours' rho u, forcing
// moments, collision, store.  No barriers, so the SMs run at the occupancy
// the registers allow; the price over the one-pass ideal is one extra read
// of the populations per step (about 430 B per node against 332).
//
// What bounds them (GB300, FP32, 128 x 256 x 128): the momentum pass the
// memory, 63 us for 418 MB, the measured copy rate; the step pass the latency
// of its loads at 16 warps per SM, 288 us for 1,433 MB (0.73 of the copy
// rate, 41 % of issue slots).  The split into short chains is what made it
// so: geometry and history travel to shared memory asynchronously while the
// populations and the stencil load (64x128x64: 76.6 -> 46 us per step, 91 x
// 77 x 93: 94 -> 60, 256^3: 1,717 -> 1,334 with the following), face nodes
// run in blocks of their own ahead of the others instead of on a slow branch
// of every warp (rho u of a face node in closed form where that keeps the bits,
// momentum_by_rule), blocks shrink
// until every SM has four (16 x 32 x 16: 22.6 -> 13.3 us per step, FP64 106
// -> 51), and each kernel's blocks come up while the previous one drains.
// Measured without effect: five blocks per SM, blocks of 64 or 160 nodes,
// descending order, evict-first stores; an L2 prefetch one wave ahead costs
// 10 to 30 %.
#pragma once

#include <mutex>
#include <type_traits>

#include "fast_div.h"
#include "step_math.cuh"

namespace cslbm {

template <class R> struct alignas(4 * sizeof(R)) Mom4 {
    R x, y, z, w;
};

// 32-bit element offsets of a node's pull sources / stencil sites for
// c in {-1, 0, +1} per axis (the host guarantees 25 N < 2^32)
struct Nbr {
    unsigned xs[3], ys[3], zs[3];
};
__device__ __forceinline__ Nbr nbr_index(const Lat& L, int x, int y, int z, int sign)
{
    Nbr p;
    const unsigned n0 = L.n[0], n01 = (unsigned)L.n[0] * L.n[1];
#pragma unroll
    for (int c = -1; c <= 1; c++) {
        p.xs[c + 1] = (unsigned)wrapc(x + sign * c, L.n[0]);
        p.ys[c + 1] = (unsigned)wrapc(y + sign * c, L.n[1]) * n0;
        p.zs[c + 1] = (unsigned)wrapc(z + sign * c, L.n[2]) * n01;
    }
    return p;
}
__device__ __forceinline__ unsigned nbr_off(const Nbr& p, int cx, int cy, int cz)
{
    return p.zs[cz + 1] + p.ys[cy + 1] + p.xs[cx + 1];
}

// rho u of a node into jf[v].  With FACES every node, a face node's from its
// inner node without the boundary rule's populations: a wall or inflow node
// takes rho_i u_w (the first moment of f^eq(rho_i, u_w) plus that of the inner
// node's non-equilibrium part, which vanishes), an outflow node takes j_i.  So
// every node makes the same gather, a face node at its inner node.  Without,
// nodes on no face only.
template <class S, class R, bool FACES>
__device__ __forceinline__ void momentum_node(const Lat& L, const S* __restrict__ P, const R* __restrict__ hist,
                                              const R* __restrict__ geo, Mom4<R>* __restrict__ jf, int x, int y,
                                              int z, unsigned v)
{
    const unsigned N = (unsigned)L.N;
    const int r[3] = {x, y, z};
    int in[3] = {x, y, z}, axis = 0, side = 0, bc = BC_OUTFLOW;
    if (FACES && on_boundary(L, x, y, z)) bc = classify(L, r, axis, side, in);
    const Nbr src = nbr_index(L, in[0], in[1], in[2], -1);
    R s[Q];
#pragma unroll
    for (int l = 0; l < Q; l++)
        s[l] = R(Store<S>::ld(P + (unsigned)pslot(l) * N + nbr_off(src, cvec(l, 0), cvec(l, 1), cvec(l, 2))));
    const unsigned vi = nbr_off(src, 0, 0, 0);
    const R sg = __ldg(geo + vi);
    Mom4<R> j;
    j.x = __ldg(hist + 1 * N + vi);
    j.y = __ldg(hist + 2 * N + vi);
    j.z = __ldg(hist + 3 * N + vi);
    j.w = R(0);
    PairSums<R> Ps;
    pair_sums(s, Ps);
    R m1[3];
    first_moment(Ps, m1);
    j.x = fmad(sg, m1[0], R(0.5) * j.x);
    j.y = fmad(sg, m1[1], R(0.5) * j.y);
    j.z = fmad(sg, m1[2], R(0.5) * j.z);
    if (FACES && bc != BC_OUTFLOW) {
        R m0 = s[0];
#pragma unroll
        for (int k = 0; k < 9; k++) m0 += Ps.p[k];
        const R rho = fmad(sg, m0 + R(1), R(0.5) * __ldg(hist + vi));
        R u[3];
        face_velocity(L, axis, side, r, u);
        j.x = rho * u[0];
        j.y = rho * u[1];
        j.z = rho * u[2];
    }
    jf[v] = j;
}

// rho u of a face node as the first moment of the boundary rule's populations
template <class S, class R>
__device__ __noinline__ void momentum_boundary(const Lat& L, const S* __restrict__ P, const R* __restrict__ hist,
                                               const R* __restrict__ geo, int x, int y, int z, Mom4<R>* jf)
{
    R s[Q];
    boundary_pops<S, R>(L, P, hist, geo, x, y, z, s);
    PairSums<R> Ps;
    pair_sums(s, Ps);
    R m1[3];
    first_moment(Ps, m1);
    const long long v = nidx(L, x, y, z);
    const R sg = geo[v];
    Mom4<R> j;
    j.x = fmad(sg, m1[0], R(0.5) * hist[1 * L.N + v]);
    j.y = fmad(sg, m1[1], R(0.5) * hist[2 * L.N + v]);
    j.z = fmad(sg, m1[2], R(0.5) * hist[3 * L.N + v]);
    j.w = R(0);
    jf[v] = j;
}

// Both passes run over consecutive nodes of the lattice, one thread each, in
// blocks of FB threads or fewer (flat_block).
constexpr int FB = 128;

struct Plane {
    Div n0, n01;
};
__device__ __forceinline__ void flat_coords(const Lat& L, const Plane& pl, unsigned v, int& x, int& y, int& z)
{
    const unsigned n0 = L.n[0], zu = div_by(v, pl.n01), r = v - zu * (n0 * (unsigned)L.n[1]), yu = div_by(r, pl.n0);
    x = (int)(r - yu * n0);
    y = (int)yu;
    z = (int)zu;
}

// The kernels of a step follow one another with programmatic launches: the
// next kernel's blocks come up while the last blocks of this one still run
// and wait here for its completion before they touch memory.
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <class S, class R>
__global__ void __launch_bounds__(FB) k_momentum_flat(const __grid_constant__ Lat L, const __grid_constant__ Plane pl,
                                                      const S* __restrict__ P, const R* __restrict__ hist,
                                                      const R* __restrict__ geo, Mom4<R>* __restrict__ jf)
{
    const unsigned v = blockIdx.x * blockDim.x + threadIdx.x;
    int x, y, z;
    flat_coords(L, pl, v, x, y, z);
    wait_previous();
    launch_next();
    if (v >= (unsigned)L.N) return;
    momentum_node<S, R, true>(L, P, hist, geo, jf, x, y, z, v);
}

// The nodes on non-periodic faces as up to six boxes without overlap: the
// faces of axis 2 whole, those of axis 1 without the axis-2 face nodes, those
// of axis 0 without the face nodes of axes 1 and 2.
struct FaceList {
    int nseg;
    int lo[6][3], len[6][3];
    long long start[7];
};

inline FaceList face_list(const cslbm_ctx* c)
{
    FaceList f{};
    long long total = 0;
    bool done[3] = {false, false, false};
    for (int a = 2; a >= 0; a--) {
        if (c->p.bc_lo[a] == CSLBM_PERIODIC) continue;
        for (int side = 0; side < 2; side++) {
            const int k = f.nseg++;
            for (int b = 0; b < 3; b++) {
                if (b == a) {
                    f.lo[k][b] = side ? c->n[b] - 1 : 0;
                    f.len[k][b] = 1;
                } else if (done[b]) {
                    f.lo[k][b] = 1;
                    f.len[k][b] = c->n[b] - 2;
                } else {
                    f.lo[k][b] = 0;
                    f.len[k][b] = c->n[b];
                }
            }
            f.start[k] = total;
            total += (long long)f.len[k][0] * f.len[k][1] * f.len[k][2];
        }
        done[a] = true;
    }
    f.start[f.nseg] = total;
    return f;
}

// nodes on non-periodic faces
inline long long face_count(const cslbm_params& p)
{
    long long all = 1, inner = 1;
    for (int a = 0; a < 3; a++) {
        all *= p.n[a];
        inner *= p.bc_lo[a] == CSLBM_PERIODIC ? p.n[a] : p.n[a] - 2;
    }
    return all - inner;
}

// node i of the list; false past its end.  (Selects over the six segments: an
// index of f by a runtime value would copy it to local memory; face nodes
// number fewer than 2^31.)
__device__ __forceinline__ bool face_coords(const FaceList& f, int i, int& x, int& y, int& z)
{
    if (i >= (int)f.start[f.nseg]) return false;
    int lo0 = 0, lo1 = 0, lo2 = 0, len0 = 1, len1 = 1, st = 0;
#pragma unroll
    for (int k = 0; k < 6; k++)
        if (k < f.nseg && i >= (int)f.start[k]) {
            lo0 = f.lo[k][0];
            lo1 = f.lo[k][1];
            lo2 = f.lo[k][2];
            len0 = f.len[k][0];
            len1 = f.len[k][1];
            st = (int)f.start[k];
        }
    const int r = i - st, q = r / len0;
    x = lo0 + (r - q * len0);
    y = lo1 + q % len1;
    z = lo2 + q / len1;
    return true;
}

// The same with the boundary rule on face nodes (momentum_by_rule), which the
// first nfb blocks take.  MINB: eight blocks per SM (64 registers, the rule
// spills 48 bytes) where the memory bounds the pass, one (80 registers) where
// the rule's chain of loads does (us per step, closed form / one / eight: 21 x
// 33 x 17 8.9, 9.5, 10.3; 91 x 77 x 93 55.0, 55.3, 54.8; 257 x 128 x 128 334,
// 341, 336).
template <class S, class R, int MINB>
__global__ void __launch_bounds__(FB, MINB)
    k_momentum_rule(const __grid_constant__ Lat L, const __grid_constant__ Plane pl, const __grid_constant__ FaceList f,
                    unsigned nfb, const S* __restrict__ P, const R* __restrict__ hist, const R* __restrict__ geo,
                    Mom4<R>* __restrict__ jf)
{
    int x, y, z;
    if (blockIdx.x < nfb) {
        const bool ok = face_coords(f, (int)(blockIdx.x * blockDim.x + threadIdx.x), x, y, z);
        wait_previous();
        launch_next();
        if (ok) momentum_boundary<S, R>(L, P, hist, geo, x, y, z, jf);
        return;
    }
    const unsigned v = (blockIdx.x - nfb) * blockDim.x + threadIdx.x;
    flat_coords(L, pl, v, x, y, z);
    wait_previous();
    launch_next();
    if (v >= (unsigned)L.N || on_boundary(L, x, y, z)) return;
    momentum_node<S, R, false>(L, P, hist, geo, jf, x, y, z, v);
}

// rho u at a stencil site that may lie one step outside a non-periodic face:
// linear extrapolation 2 j(face) - j(face - normal) per out-of-range axis
// (tensor product over the axes).  Each axis contributes one or two
// (coordinate, weight) terms; the 2 x 2 x 2 sum is unrolled with the loads of
// zero-weight terms predicated off, so that all loads can be in flight at once.
__device__ __forceinline__ void site_axis(int r, int n, bool per_lo, bool per_hi, int& c0, int& c1, float& w0, float& w1)
{
    if (r >= 0 && r < n) { c0 = c1 = r; w0 = 1.0f; w1 = 0.0f; }
    else if (r < 0 && per_lo) { c0 = c1 = r + n; w0 = 1.0f; w1 = 0.0f; }
    else if (r >= n && per_hi) { c0 = c1 = r - n; w0 = 1.0f; w1 = 0.0f; }
    else if (r < 0) { c0 = 0; c1 = 1; w0 = 2.0f; w1 = -1.0f; }
    else { c0 = n - 1; c1 = n - 2; w0 = 2.0f; w1 = -1.0f; }
}
template <class R>
__device__ __forceinline__ Mom4<R> mom_site(const Lat& L, const Mom4<R>* __restrict__ jf, int x, int y, int z)
{
    // most sites of a face node's stencil are lattice nodes (after a periodic
    // wrap): one load, the value the weighted sum below would give
    {
        const int r[3] = {x, y, z};
        int w[3];
        bool ghost = false;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            w[a] = r[a];
            if (r[a] < 0) {
                if (L.bclo[a] == BC_PERIODIC) w[a] += L.n[a];
                else ghost = true;
            } else if (r[a] >= L.n[a]) {
                if (L.bchi[a] == BC_PERIODIC) w[a] -= L.n[a];
                else ghost = true;
            }
        }
        if (!ghost) return jf[((unsigned)w[2] * L.n[1] + w[1]) * (unsigned)L.n[0] + w[0]];
    }
    int x0, x1, y0, y1, z0, z1;
    float wx0, wx1, wy0, wy1, wz0, wz1;
    site_axis(x, L.n[0], L.bclo[0] == BC_PERIODIC, L.bchi[0] == BC_PERIODIC, x0, x1, wx0, wx1);
    site_axis(y, L.n[1], L.bclo[1] == BC_PERIODIC, L.bchi[1] == BC_PERIODIC, y0, y1, wy0, wy1);
    site_axis(z, L.n[2], L.bclo[2] == BC_PERIODIC, L.bchi[2] == BC_PERIODIC, z0, z1, wz0, wz1);
    Mom4<R> acc;
    acc.x = acc.y = acc.z = acc.w = R(0);
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int k = 0; k < 2; k++)
#pragma unroll
            for (int m = 0; m < 2; m++) {
                const float w = (i ? wx1 : wx0) * (k ? wy1 : wy0) * (m ? wz1 : wz0);
                if (w != 0.0f) {
                    const Mom4<R> j = jf[nidx(L, i ? x1 : x0, k ? y1 : y0, m ? z1 : z0)];
                    acc.x += R(w) * j.x;
                    acc.y += R(w) * j.y;
                    acc.z += R(w) * j.z;
                }
            }
    return acc;
}

// The rho u differences d_l = j(x + c_l) - j(x - c_l) of a face node over the
// nine opposite pairs, sites beyond a non-periodic face by the extrapolation
// of mom_site.  Per axis each of the offsets -1, 0, 1 is one term (o, 1) or,
// past a face, two terms (face, 2), (inner, -1); a site displaced along two
// axes is their product.  Second terms are predicated loads instead of
// branches, so that the 18 sites' loads are in flight together: a face node's
// step is a chain of such latencies (16 x 32 x 16 FP32: 13.3 -> 8.3 us per step,
// k_step_faces at 256^3 64 -> 39 us).
template <class R>
__device__ __forceinline__ void ghost_differences(const Lat& L, const Mom4<R>* jf, int x, int y, int z, R d[9][3])
{
    unsigned o[3][3], g[3][3];  // first and second term's offset of axis a at c = -1, 0, 1
    bool two[3][3];
    const int r[3] = {x, y, z};
    unsigned stride = 1;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int n = L.n[a];
#pragma unroll
        for (int c = -1; c <= 1; c++) {
            const int q = r[a] + c;
            const bool out = q < 0 || q >= n;
            const bool per = (q < 0 ? L.bclo[a] : L.bchi[a]) == BC_PERIODIC;
            two[a][c + 1] = out && !per;
            // past a face: the face node itself (r), then the node one step inward
            o[a][c + 1] = (unsigned)(out ? (per ? wrapc(q, n) : r[a]) : q) * stride;
            g[a][c + 1] = (unsigned)(r[a] - c) * stride;
        }
        stride *= (unsigned)n;
    }
    auto add = [&](R (&acc)[3], bool on, R w, unsigned off) {
        if (on) {
            const Mom4<R> j = jf[off];
            acc[0] = fmad(w, j.x, acc[0]);
            acc[1] = fmad(w, j.y, acc[1]);
            acc[2] = fmad(w, j.z, acc[2]);
        }
    };
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const int l = 2 * k + 1;
        R site[2][3];  // rho u at x + c_l and at x - c_l, each summed in mom_site's order
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int sg = 1 - 2 * s, c[3] = {sg * cvec(l, 0), sg * cvec(l, 1), sg * cvec(l, 2)};
            // the (one or two) displaced axes a, b; the others contribute their own coordinate
            const int a = c[0] ? 0 : (c[1] ? 1 : 2), b = c[2] ? 2 : (c[1] ? 1 : 0);
            unsigned rest = 0;
#pragma unroll
            for (int q = 0; q < 3; q++)
                if (q != a && q != b) rest += o[q][1];
            const int ia = c[a] + 1, ib = c[b] + 1;
            const bool ta = two[a][ia], tb = a != b && two[b][ib];
            const unsigned o0 = rest + o[a][ia], ob = a != b ? o[b][ib] : 0u, gb = a != b ? g[b][ib] : 0u;
            const R wa = ta ? R(2) : R(1), wb = tb ? R(2) : R(1);
            R(&acc)[3] = site[s];
            acc[0] = acc[1] = acc[2] = R(0);
            add(acc, true, wa * wb, o0 + ob);
            if (a != b) add(acc, tb, -wa, o0 + gb);
            add(acc, ta, -wb, rest + g[a][ia] + ob);
            if (a != b) add(acc, ta && tb, R(1), rest + g[a][ia] + gb);
        }
#pragma unroll
        for (int i = 0; i < 3; i++) d[k][i] = site[0][i] - site[1][i];
    }
}

// L2 eviction policies (createpolicy): data read or written once per step
// goes out of L2 first; data read again within the step stays longer
__device__ __forceinline__ unsigned long long policy_evict_first()
{
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
__device__ __forceinline__ unsigned long long policy_evict_last()
{
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
// a store carrying an L2 eviction policy
__device__ __forceinline__ void st_hint(float* p, float v, unsigned long long pol)
{
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;\n" ::"l"(p), "f"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_hint(double* p, double v, unsigned long long pol)
{
    asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;\n" ::"l"(p), "d"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_hint(__half* p, float v, unsigned long long pol)
{
    const unsigned short b = __half_as_ushort(__float2half_rn(v));
    asm volatile("st.global.L2::cache_hint.b16 [%0], %1, %2;\n" ::"l"(p), "h"(b), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_hint(__nv_bfloat16* p, float v, unsigned long long pol)
{
    const unsigned short b = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    asm volatile("st.global.L2::cache_hint.b16 [%0], %1, %2;\n" ::"l"(p), "h"(b), "l"(pol) : "memory");
}

// the step of one node from its populations s (h - w), geometry and history
// at element offset v, and the rho u differences d across the nine opposite
// stencil pairs; stores the new populations and forcing coefficients (with
// the L2 policy pol when HINT)
template <class S, class R, bool HINT = false>
__device__ __forceinline__ void step_core(const Lat& L, const R s[Q], const GeoT<R>& G, const HistT<R>& Hp,
                                          const R d[9][3], S* __restrict__ Pout, R* __restrict__ hout, unsigned v,
                                          unsigned N, unsigned long long pol = 0)
{
    PairSums<R> Ps;
    pair_sums(s, Ps);
    R m0, m1[3], m2[6];
    all_moments(s, Ps, m0, m1, m2);
    const R rho = fmad(G.sg, m0 + R(1), R(0.5) * Hp.A);
    const R ir = recip(rho);
    R j[3];
#pragma unroll
    for (int a = 0; a < 3; a++) j[a] = fmad(G.sg, m1[a], R(0.5) * Hp.B[a]);
    R Tt[6];
    stress_t<R, R>(R(L.theta), R(L.kvisc), G, rho, ir, j, m2, Hp, Tt);
    R D[3][3];
    gradient_from_pairs(d, D);
    const R fext[3] = {R(L.fext[0]), R(L.fext[1]), R(L.fext[2])};
    HistT<R> H;
    forcing_t<R, R>(R(L.theta), fext, G, j, Tt, D, H);
    R out[Q];
    collide_t<R, R>(R(L.omega), R(L.theta), G, s, m0, rho, ir, j, Hp, H, out);
    if constexpr (HINT) {
        st_hint(hout + v, H.A, pol);
#pragma unroll
        for (int a = 0; a < 3; a++) st_hint(hout + (1 + a) * N + v, H.B[a], pol);
#pragma unroll
        for (int a = 0; a < 6; a++) st_hint(hout + (4 + a) * N + v, H.C[a], pol);
#pragma unroll
        for (int l = 0; l < Q; l++) st_hint(Pout + (unsigned)pslot(l) * N + v, out[l], pol);
    } else {
        hout[v] = H.A;
#pragma unroll
        for (int a = 0; a < 3; a++) hout[(1 + a) * N + v] = H.B[a];
#pragma unroll
        for (int a = 0; a < 6; a++) hout[(4 + a) * N + v] = H.C[a];
#pragma unroll
        for (int l = 0; l < Q; l++) Store<S>::st(Pout + (unsigned)pslot(l) * N + v, out[l]);
    }
}

template <class R>
__device__ __forceinline__ void load_geo_hist(const R* __restrict__ geo, const R* __restrict__ hist, unsigned v,
                                              unsigned N, GeoT<R>& G, HistT<R>& Hp)
{
    G.sg = __ldg(geo + v);
    G.isg = recip(G.sg);
#pragma unroll
    for (int a = 0; a < 6; a++) G.gi[a] = __ldg(geo + (1 + a) * N + v);
#pragma unroll
    for (int a = 0; a < 18; a++) G.gam[a] = __ldg(geo + (7 + a) * N + v);
#pragma unroll
    for (int k = 0; k < 3; k++) G.gc[k] = (G.gam[0 * 6 + s6(k, 0)] + G.gam[1 * 6 + s6(k, 1)]) + G.gam[2 * 6 + s6(k, 2)];
    Hp.A = __ldg(hist + v);
#pragma unroll
    for (int a = 0; a < 3; a++) Hp.B[a] = __ldg(hist + (1 + a) * N + v);
#pragma unroll
    for (int a = 0; a < 6; a++) Hp.C[a] = __ldg(hist + (4 + a) * N + v);
}

// the step of a node on a non-periodic face (boundary rule, ghost stencil)
template <class S, class R>
__device__ __forceinline__ void step_boundary_body(const Lat& L, const S* __restrict__ Pin, S* __restrict__ Pout,
                                                   const R* __restrict__ hin, R* __restrict__ hout,
                                                   const R* __restrict__ geo, const Mom4<R>* jf, int x,
                                                   int y, int z)
{
    const unsigned N = (unsigned)L.N, v = (unsigned)nidx(L, x, y, z);
    GeoT<R> G;
    HistT<R> Hp;
    load_geo_hist(geo, hin, v, N, G, Hp);
    // the boundary rule with the node's own metric and history as loaded
    Geo<R> Gw;
    Gw.sg = G.sg;
    Gw.isg = G.isg;
#pragma unroll
    for (int a = 0; a < 6; a++) Gw.gi[a] = G.gi[a];
    Hist<R> Hw;
    Hw.A = Hp.A;
#pragma unroll
    for (int a = 0; a < 3; a++) Hw.B[a] = Hp.B[a];
#pragma unroll
    for (int a = 0; a < 6; a++) Hw.C[a] = Hp.C[a];
    R s[Q];
    boundary_pops_w<S, R>(L, Pin, hin, geo, x, y, z, Gw, Hw, s);
    R d[9][3];
    ghost_differences<R>(L, jf, x, y, z, d);
    step_core<S, R>(L, s, G, Hp, d, Pout, hout, v, N);
}

// the same out of line, where one kernel runs face nodes among others (jf may
// be written by the same launch: plain loads)
template <class S, class R>
__device__ __noinline__ void step_face(const Lat& L, const S* __restrict__ Pin, S* __restrict__ Pout,
                                       const R* __restrict__ hin, R* __restrict__ hout, const R* __restrict__ geo,
                                       const Mom4<R>* jf, int x, int y, int z)
{
    step_boundary_body<S, R>(L, Pin, Pout, hin, hout, geo, jf, x, y, z);
}

// one step of the face nodes only (the interior comes from the row-staged pass)
template <class S, class R>
__global__ void __launch_bounds__(128) k_step_faces(const __grid_constant__ Lat L, const __grid_constant__ FaceList f,
                                                    const S* __restrict__ Pin, S* __restrict__ Pout,
                                                    const R* __restrict__ hin, R* __restrict__ hout,
                                                    const R* __restrict__ geo, const Mom4<R>* __restrict__ jf)
{
    int x, y, z;
    if (!face_coords(f, blockIdx.x * 128 + threadIdx.x, x, y, z)) return;
    step_boundary_body<S, R>(L, Pin, Pout, hin, hout, geo, jf, x, y, z);
}

template <class S, class R>
int launch_faces(const cslbm_ctx* c, const Lat& L, const S* Pin, S* Pout, const R* hin, R* hout, const R* geo,
                 cudaStream_t stream)
{
    const FaceList f = face_list(c);
    const long long total = f.start[f.nseg];
    if (total == 0) return 0;
    k_step_faces<S, R><<<(unsigned)((total + 127) / 128), 128, 0, stream>>>(L, f, Pin, Pout, hin, hout, geo,
                                                                               (const Mom4<R>*)c->jf);
    return 1;
}

// asynchronous copy of one value into shared memory (with an L2 policy)
__device__ __forceinline__ void copy_async(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async(double* dst, const double* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async(float* dst, const float* src, unsigned long long pol)
{
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, %2;\n" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void copy_async(double* dst, const double* src, unsigned long long pol)
{
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 8, %2;\n" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// values of a node that step_interior stages in shared memory: geometry,
// history and, on one lattice in FP32, the populations (a copy moves 4 bytes
// at least, and FP64's would not fit)
template <class S, bool ONE> constexpr bool kStagePops = ONE && sizeof(S) == 4;
template <class S, bool ONE> constexpr int kStaged = NGEO + NHIST + (kStagePops<S, ONE> ? Q : 0);

// The step of an interior node.  The staged values travel to shared memory
// (sm[k * ST], the thread's own column: no barrier) while the rho u stencil
// loads into registers, so that all of the node's reads are in flight at
// once.  With ONE (a step of a single lattice) the geometry, read once per
// step, leaves L2 first and the new populations and history, which the next
// step reads twice, last: 91 x 77 x 93 FP16 49.0 -> 47.1 us per step, FP32 58.0
// -> 55.3, 64 x 128 x 64 45.9 -> 43.3; 256^3 the same within 1 %.  In a batch
// the same costs 2 to 7 % (its channels leave L2 whatever the policy, and the
// persistent kernel's loops want the shared memory as L1).
template <class S, class R, int ST, bool ONE>
__device__ __forceinline__ void step_interior(const Lat& L, const S* __restrict__ Pin, S* __restrict__ Pout,
                                              const R* __restrict__ hin, R* __restrict__ hout,
                                              const R* __restrict__ geo, const Mom4<R>* jf, int x, int y, int z,
                                              unsigned v, R* sm)
{
    constexpr bool POPS = kStagePops<S, ONE>;
    const unsigned N = (unsigned)L.N;
    {
        const R* g = geo + v;
        const R* h = hin + v;
        const unsigned long long once = ONE ? policy_evict_first() : 0;
#pragma unroll
        for (int k = 0; k < NGEO; k++) {
            if constexpr (ONE) copy_async(sm + k * ST, g + (size_t)k * N, once);
            else copy_async(sm + k * ST, g + (size_t)k * N);
        }
#pragma unroll
        for (int k = 0; k < NHIST; k++) copy_async(sm + (NGEO + k) * ST, h + (size_t)k * N);
    }
    const Nbr src = nbr_index(L, x, y, z, -1);
    R s[Q];
#pragma unroll
    for (int l = 0; l < Q; l++) {
        const S* p = Pin + (unsigned)pslot(l) * N + nbr_off(src, cvec(l, 0), cvec(l, 1), cvec(l, 2));
        if constexpr (POPS) copy_async(sm + (NGEO + NHIST + l) * ST, p);
        else s[l] = R(Store<S>::ld(p));
    }
    R d[9][3];
#pragma unroll
    for (int k = 0; k < 9; k++) {
        // site x + c is the pull source of -c
        const int l = 2 * k + 1, cx = cvec(l, 0), cy = cvec(l, 1), cz = cvec(l, 2);
        const Mom4<R> p = jf[nbr_off(src, -cx, -cy, -cz)], m = jf[nbr_off(src, cx, cy, cz)];
        d[k][0] = p.x - m.x;
        d[k][1] = p.y - m.y;
        d[k][2] = p.z - m.z;
    }
    copies_landed();
    if constexpr (POPS) {
#pragma unroll
        for (int l = 0; l < Q; l++) s[l] = sm[(NGEO + NHIST + l) * ST];
    }
    GeoT<R> G;
    HistT<R> Hp;
    G.sg = sm[0];
    G.isg = recip(G.sg);
#pragma unroll
    for (int a = 0; a < 6; a++) G.gi[a] = sm[(1 + a) * ST];
#pragma unroll
    for (int a = 0; a < 18; a++) G.gam[a] = sm[(7 + a) * ST];
#pragma unroll
    for (int k = 0; k < 3; k++) G.gc[k] = (G.gam[0 * 6 + s6(k, 0)] + G.gam[1 * 6 + s6(k, 1)]) + G.gam[2 * 6 + s6(k, 2)];
    Hp.A = sm[NGEO * ST];
#pragma unroll
    for (int a = 0; a < 3; a++) Hp.B[a] = sm[(NGEO + 1 + a) * ST];
#pragma unroll
    for (int a = 0; a < 6; a++) Hp.C[a] = sm[(NGEO + 4 + a) * ST];
    step_core<S, R, ONE>(L, s, G, Hp, d, Pout, hout, v, N, ONE ? policy_evict_last() : 0);
}

// The step of every node: the first nfb blocks take the face nodes (the
// longest chains of loads, so they start first), the others the nodes of the
// planes between non-periodic faces of axis 2, v = v0 ..
template <class S, class R>
__global__ void __launch_bounds__(FB, sizeof(R) == 8 ? 3 : 4)
    k_step_flat(const __grid_constant__ Lat L, const __grid_constant__ Plane pl, const __grid_constant__ FaceList f,
                unsigned nfb, unsigned v0, unsigned v1, const S* __restrict__ Pin, S* __restrict__ Pout,
                const R* __restrict__ hin, R* __restrict__ hout, const R* __restrict__ geo,
                const Mom4<R>* __restrict__ jf)
{
    __shared__ R sm[kStaged<S, true> * FB];
    int x, y, z;
    if (blockIdx.x < nfb) {
        const bool ok = face_coords(f, (int)(blockIdx.x * blockDim.x + threadIdx.x), x, y, z);
        wait_previous();
        launch_next();
        if (ok) step_boundary_body<S, R>(L, Pin, Pout, hin, hout, geo, jf, x, y, z);
        return;
    }
    const unsigned v = v0 + (blockIdx.x - nfb) * blockDim.x + threadIdx.x;
    flat_coords(L, pl, v, x, y, z);
    wait_previous();
    launch_next();
    if (v >= v1 || on_boundary(L, x, y, z)) return;
    step_interior<S, R, FB, true>(L, Pin, Pout, hin, hout, geo, jf, x, y, z, v, sm + threadIdx.x);
}

// The dynamic shared memory of a kernel beyond 48 KB (bytes, or 0 for all the
// device allows a kernel without static shared memory), set once per device:
// the attribute belongs to the context of the device current when it is set.
template <auto kernel>
inline void set_smem_optin_once(int device, int bytes = 0)
{
    static std::mutex mu;
    static bool done[64] = {};
    if (device < 0 || device >= 64) return;
    std::lock_guard<std::mutex> lock(mu);
    if (done[device]) return;
    if (!bytes) cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done[device] = true;
}

// threads per block: FB, fewer where that would leave multiprocessors idle
inline unsigned flat_block(const cslbm_ctx* c)
{
    unsigned tb = FB;
    while (tb > 32 && c->N < (long long)tb * 4 * c->n_sm) tb /= 2;
    return tb;
}

inline Plane make_plane(const Lat& L)
{
    Plane p;
    p.n0 = make_div((unsigned)L.n[0]);
    p.n01 = make_div((unsigned)L.n[0] * (unsigned)L.n[1]);
    return p;
}

// a kernel whose blocks may come up before the previous one has ended (it
// waits for that itself)
template <class... A>
inline void launch_after(void (*kernel)(A...), unsigned grid, unsigned block, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Which lattices take rho u of their face nodes from the boundary rule (one
// more rounding of numbers that cancel, but the rounding these lattices have
// always had): FP32 arithmetic, unless AUTO may take the fused pass, which has
// the closed form; then the gather pass gives the fused pass's bits.  The value
// of a wall-force objective is a sum of terms hundreds of times larger, so
// another rounding of the state moves it by several times its error either way
// (FP32, 22 x 101 x 29, 23 steps from rest: 1.7e-7 with the rule, 5.5e-7 with
// the closed form; over 16 channels neither is better).
inline bool momentum_by_rule(const cslbm_ctx* c)
{
    return c->p.storage != CSLBM_FP64 && !(c->rows.fused_ok && c->p.step_kernel == CSLBM_STEP_AUTO);
}

template <class S, class R>
void launch_momentum(const cslbm_ctx* c, const Lat& L, const S* P, const R* hin, const R* geo, bool rule)
{
    const unsigned tb = flat_block(c), nb = (unsigned)((c->N + tb - 1) / tb);
    if constexpr (!std::is_same<R, double>::value) {
        const FaceList f = face_list(c);
        const unsigned nfb = (unsigned)((f.start[f.nseg] + tb - 1) / tb);
        if (rule && nfb) {
            launch_after(tb < FB ? k_momentum_rule<S, R, 1> : k_momentum_rule<S, R, 8>, nfb + nb, tb, c->stream, L,
                         make_plane(L), f, nfb, P, hin, geo, (Mom4<R>*)c->jf);
            return;
        }
    }
    launch_after(k_momentum_flat<S, R>, nb, tb, c->stream, L, make_plane(L), P, hin, geo, (Mom4<R>*)c->jf);
}

// one time step: momentum pass, then the step pass
template <class S, class R>
void launch_flat_step(const cslbm_ctx* c, const Lat& L, const S* Pin, S* Pout, const R* hin, R* hout, const R* geo)
{
    launch_momentum<S, R>(c, L, Pin, hin, geo, momentum_by_rule(c));
    const unsigned tb = flat_block(c);
    const FaceList f = face_list(c);
    const unsigned nfb = (unsigned)((f.start[f.nseg] + tb - 1) / tb), n01 = (unsigned)c->n[0] * c->n[1];
    const bool zper = c->p.bc_lo[2] == CSLBM_PERIODIC;
    const unsigned v0 = zper ? 0 : n01, v1 = zper ? (unsigned)c->N : (unsigned)c->N - n01;
    launch_after(k_step_flat<S, R>, nfb + (v1 - v0 + tb - 1) / tb, tb, c->stream, L, make_plane(L), f, nfb, v0, v1, Pin,
                 Pout, hin, hout, geo, (const Mom4<R>*)c->jf);
}

}  // namespace cslbm
