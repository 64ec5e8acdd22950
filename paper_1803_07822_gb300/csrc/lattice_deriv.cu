// Isotropic lattice derivatives of FP64 fields (App. D) on the device, and
// the geometry of a context from its metric alone.
//
// With the D3Q19 weights w_l and velocities c_l (lattice units):
//   G_i f(x) = (1/c_s^2) sum_l w_l c_l^i f(x + c_l)            second order
//   L f(x)   = (2/c_s^2) sum_l w_l (f(x + c_l) - f(x))         second order
//   d_i f(x) = G_i[f - (c_s^2/2) L f](x)                        fourth order
// (the third-order term of G_i is (c_s^2/2) d_i Lap f: the fourth moment of
// the D3Q19 weights is isotropic).  Beyond a non-periodic face the field is
// continued by the polynomial of degree `order` through the order + 1 nodes
// nearest the face, axis by axis (tensor product at edges and corners).
//
// Two kernels: the first writes F / 12, F = f - (c_s^2/2) L f (order 4,
// k_correct), or the continued f itself (order 2, k_pad: its bits, so that
// differences of close values stay exact), on the lattice padded by one site
// along every axis with a non-periodic face; k_grad forms G_i F at every node.  FP64 throughout, which is what bounds both: the FP64 pipe issues two
// lanes per clock and SM, so only the number of FP64 instructions counts.
// Written out per node, the stencils take 22 and 24 of them; both factor into
// sums along one axis that neighbours share, which leaves 10 and 16: blocks
// march along axis 2 with one plane of a 32 x 8 tile (and its rim) in shared
// memory, in-plane sums exchanged there, sums along the march kept in
// registers.  Six fields on 128 x 256 x 128, order 4: 1,359 + 1,150 -> 1,562 us for both.
// Lattices that fill the tiles badly keep a thread per site (see
// gradient_marches).
#include <cstdint>
#include <string>

#include "ctx.h"
#include "lbm_device.cuh"
#include "march_tiles.cuh"

cslbm_status cslbm_record_error(cslbm_status s, const char* msg);

namespace cslbm {
namespace lder {

constexpr int TBL = 256;

struct Box {
    int n[3];
    int plo[3], phi[3];  // low / high face periodic
    int pad[3];          // 1 on an axis with a non-periodic face
    int ne[3];           // padded extents n + 2 pad
    long long N, Ne;
};

// Weight of node k (k = 0 the face node, counting inward) in the value t = 1
// or 2 sites beyond the face: the polynomial of degree `order` through the
// nodes 0..order, evaluated at -t (Lagrange form, worked out).
__device__ __forceinline__ double cont_weight(int order, int t, int k)
{
    if (order == 2) {
        const double a[3] = {3.0, -3.0, 1.0}, b[3] = {6.0, -8.0, 3.0};
        return t == 1 ? a[k] : b[k];
    }
    const double a[5] = {5.0, -10.0, 10.0, -5.0, 1.0}, b[5] = {15.0, -40.0, 45.0, -24.0, 5.0};
    return t == 1 ? a[k] : b[k];
}

__device__ __forceinline__ bool wrap(const Box& B, int a, int& r)
{
    if (r < 0 && B.plo[a]) r += B.n[a];
    else if (r >= B.n[a] && B.phi[a]) r -= B.n[a];
    return r >= 0 && r < B.n[a];
}

// the continued field at a site up to two steps beyond a face: the terms of
// every out-of-range axis multiplied out
__device__ __noinline__ double site_far(const Box& B, const double* __restrict__ f, int order, int x, int y, int z)
{
    int c[3][5], m[3];
    double w[3][5];
    const int r[3] = {x, y, z};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        int ra = r[a];
        if (wrap(B, a, ra)) {
            m[a] = 1;
            c[a][0] = ra;
            w[a][0] = 1.0;
            continue;
        }
        const bool lo = ra < 0;
        const int t = lo ? -ra : ra - (B.n[a] - 1);
        m[a] = order + 1;
        for (int k = 0; k <= order; k++) {
            c[a][k] = lo ? k : B.n[a] - 1 - k;
            w[a][k] = cont_weight(order, t, k);
        }
    }
    double v = 0.0;
    for (int k = 0; k < m[2]; k++)
        for (int j = 0; j < m[1]; j++) {
            double row = 0.0;
            const long long base = ((long long)c[2][k] * B.n[1] + c[1][j]) * B.n[0];
            for (int i = 0; i < m[0]; i++) row += w[0][i] * f[base + c[0][i]];
            v += w[2][k] * w[1][j] * row;
        }
    return v;
}

__device__ __forceinline__ double site(const Box& B, const double* __restrict__ f, int order, int x, int y, int z)
{
    int xs = x, ys = y, zs = z;
    if (wrap(B, 0, xs) && wrap(B, 1, ys) && wrap(B, 2, zs))
        return __ldg(f + ((long long)zs * B.n[1] + ys) * B.n[0] + xs);
    return site_far(B, f, order, x, y, z);
}

// a site whose whole stencil resolves without continuation (periodic wrap only)
__device__ __forceinline__ bool inner(const Box& B, int a, int r)
{
    return r >= 0 && r < B.n[a] && (r >= 1 || B.plo[a]) && (r <= B.n[a] - 2 || B.phi[a]);
}
// The fields and the weights.  The faces of G_i weigh w_1 / c_s^2 = 1/6, its
// edges w_7 / c_s^2 = 1/12; with order 4 the scratch holds F / 12, so that the
// gradient below needs no products but by two.
constexpr double kEdge = 1.0 / 12.0;

// order 2: the continued field at every site of the padded lattice, component blockIdx.y
__global__ void __launch_bounds__(TBL) k_pad(const __grid_constant__ Box B, const double* __restrict__ f,
                                             double* __restrict__ F)
{
    // 32-bit site arithmetic (the padded lattice has fewer than 2^32 sites)
    const unsigned s = blockIdx.x * TBL + threadIdx.x;
    if (s >= (unsigned)B.Ne) return;
    const unsigned ne0 = B.ne[0], ne1 = B.ne[1], row = s / ne0, zr = row / ne1;
    F[(long long)blockIdx.y * B.Ne + s] =
        site(B, f + (long long)blockIdx.y * B.N, 2, (int)(s - row * ne0) - B.pad[0],
             (int)(row - zr * ne1) - B.pad[1], (int)zr - B.pad[2]);
}

// Order 4: F / 12 on the padded lattice, F = f - (c_s^2/2) L f = f0 - sum_l w_l
// (f_l - f0) with sum_{l>0} w_l = 2/3, w = 1/18 on the six faces, 1/36 on the
// twelve edges.  With the in-plane sums q = s_x + s_y (s_a = f(a + 1) + f(a -
// 1)) and e = s_x(y + 1) + s_x(y - 1), and u = f + q/2,
//   F = (5/3) f - (q + e/2) / 18 - (u(z + 1) + u(z - 1)) / 18.
// Values beyond a face are continued as a plane is loaded, so that every site
// takes these sums: a constant field's gradient is exactly zero, as for sums
// written out per site.  (Sites next to a face of axis 0 or 1 in a path of
// their own, 19 continued sites each, one after the other: 128 x 256 x 128, six
// fields, both kernels, walls across axis 0 5,553 us against 1,890, across axes
// 1 and 2 2,628 against 1,599.)
__global__ void __launch_bounds__(TX* TY) k_correct(const __grid_constant__ Box B, const __grid_constant__ Tiles T,
                                                    const double* __restrict__ f, double* __restrict__ F)
{
    __shared__ double fs[TY + 2][TX + 2], ss[TY + 2][TX];
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * TX + tx;
    int x0, y0, za, zb;
    tile_of(T, -B.pad[0], -B.pad[1], x0, y0, za, zb);
    const int x = x0 + tx, y = y0 + ty;
    const double* fc = f + (long long)blockIdx.y * B.N;
    double* Fc = F + (long long)blockIdx.y * B.Ne;
    const bool mine = x < B.n[0] + B.pad[0] && y < B.n[1] + B.pad[1];
    // the tile's entries this thread loads: in-plane offset; beyond one face of
    // the plane that of the face node, with the step inward and the distance
    // `gone`; kCorner beyond two, kNone for none
    constexpr int kNone = -1, kCorner = -2;
    int off[2], step[2], gone[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int i = t + k * TX * TY, ly = i / (TX + 2), lx = i - ly * (TX + 2);
        int rx = x0 - 1 + lx, ry = y0 - 1 + ly;
        off[k] = kNone;
        step[k] = gone[k] = 0;
        if (i < (TX + 2) * (TY + 2) && rx <= B.n[0] + B.pad[0] && ry <= B.n[1] + B.pad[1]) {
            const bool inx = wrap(B, 0, rx), iny = wrap(B, 1, ry);
            const int r = inx ? ry : rx, n = B.n[inx ? 1 : 0], dir = r < 0 ? 1 : -1;
            if (!inx && !iny) {
                off[k] = kCorner;
            } else {
                if (!inx || !iny) {
                    step[k] = dir * (inx ? B.n[0] : 1);
                    gone[k] = r < 0 ? -r : r - (n - 1);
                    (inx ? ry : rx) = r < 0 ? 0 : n - 1;
                }
                off[k] = ry * B.n[0] + rx;
            }
        }
    }
    const unsigned n01 = (unsigned)B.n[0] * B.n[1];
    // u and the in-plane part w of F at plane p (every thread of the block); a
    // plane one or two beyond a face is continued as it is loaded.  (To
    // continue u and w, which are linear in f, doubles the error next to the
    // face: their rounding is multiplied by the weights.)
    auto plane = [&](int p, double& u, double& w) {
        int pz = p;
        const bool in = wrap(B, 2, pz);
        const double* fp = fc + (in ? (unsigned)pz * n01 : 0u);
#pragma unroll
        for (int k = 0; k < 2; k++) {
            if (off[k] == kNone) continue;
            const int i = t + k * TX * TY;
            double v = 0.0;
            if (off[k] == kCorner || (!in && step[k])) {
                v = site_far(B, fc, 4, x0 - 1 + i % (TX + 2), y0 - 1 + i / (TX + 2), p);
            } else if (!in || step[k]) {
                const int s = in ? step[k] : (p < 0 ? 1 : -1) * (int)n01, g = in ? gone[k] : (p < 0 ? -p : p - (B.n[2] - 1));
                const double* q = in ? fp + off[k] : fc + (p < 0 ? 0u : (unsigned)(B.n[2] - 1) * n01) + off[k];
#pragma unroll
                for (int m = 0; m <= 4; m++) v = fma(cont_weight(4, g, m), __ldg(q + (long long)m * s), v);
            } else {
                v = __ldg(fp + off[k]);
            }
            (&fs[0][0])[i] = v;
        }
        __syncthreads();
        const double sx = fs[ty + 1][tx] + fs[ty + 1][tx + 2];
        ss[ty + 1][tx] = sx;
        if (ty < 2) ss[ty * (TY + 1)][tx] = fs[ty * (TY + 1)][tx] + fs[ty * (TY + 1)][tx + 2];
        const double f0 = fs[ty + 1][tx + 1], q = sx + (fs[ty][tx + 1] + fs[ty + 2][tx + 1]);
        __syncthreads();
        const double e = ss[ty][tx] + ss[ty + 2][tx];
        u = fma(0.5, q, f0);
        w = fma(5.0 / 3.0 * kEdge, f0, (-kEdge / 18.0) * fma(0.5, e, q));
    };
    double ua = 0.0, ub = 0.0, wb = 0.0;  // u of planes p - 2 and p - 1, w of p - 1
    for (int p = za - 1; p <= zb; p++) {
        double u, w;
        plane(p, u, w);
        const int z = p - 1;
        if (p > za && mine) {
            Fc[((unsigned)(z + B.pad[2]) * B.ne[1] + (unsigned)(y + B.pad[1])) * (unsigned)B.ne[0] +
               (unsigned)(x + B.pad[0])] = fma(-kEdge / 18.0, ua + u, wb);
        }
        ua = ub;
        ub = u;
        wb = w;
    }
}

// The same per site, for lattices whose tiles would be mostly empty or repeated
// (correct_marches): 19 loads, those beyond a face one after the other
__global__ void __launch_bounds__(TBL) k_correct_sites(const __grid_constant__ Box B, const double* __restrict__ f,
                                                       double* __restrict__ F)
{
    const unsigned s = blockIdx.x * TBL + threadIdx.x;
    if (s >= (unsigned)B.Ne) return;
    const double* fc = f + (long long)blockIdx.y * B.N;
    const unsigned ne0 = B.ne[0], ne1 = B.ne[1], row = s / ne0, zr = row / ne1;
    const int x = (int)(s - row * ne0) - B.pad[0], y = (int)(row - zr * ne1) - B.pad[1], z = (int)zr - B.pad[2];
    double f0, sf = 0.0, se = 0.0;
    if (inner(B, 0, x) && inner(B, 1, y) && inner(B, 2, z)) {
        unsigned o[3][3];
        const int r[3] = {x, y, z};
        const unsigned st[3] = {1u, (unsigned)B.n[0], (unsigned)B.n[0] * (unsigned)B.n[1]};
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int c = -1; c <= 1; c++) {
                int q = r[a] + c;
                wrap(B, a, q);
                o[a][c + 1] = (unsigned)q * st[a];
            }
        f0 = __ldg(fc + (o[2][1] + o[1][1] + o[0][1]));
#pragma unroll
        for (int l = 1; l < Q; l++) {
            const double fl = __ldg(fc + (o[2][cvec(l, 2) + 1] + o[1][cvec(l, 1) + 1] + o[0][cvec(l, 0) + 1]));
            if (l <= 6) sf += fl;
            else se += fl;
        }
    } else {
        f0 = site(B, fc, 4, x, y, z);
#pragma unroll
        for (int l = 1; l < Q; l++) {
            const double fl = site(B, fc, 4, x + cvec(l, 0), y + cvec(l, 1), z + cvec(l, 2));
            if (l <= 6) sf += fl;
            else se += fl;
        }
    }
    F[(long long)blockIdx.y * B.Ne + s] = fma(5.0 / 3.0 * kEdge, f0, (-kEdge / 18.0) * fma(0.5, se, sf));
}

// d_k f_c = G_k F at every node, out[(k ncomp + c) N + v].  With the
// differences d_x = F(x + 1) - F(x - 1), d_y, d_z and their sums over the
// neighbours across,
//   D_x = 2 d_x + (d_x(y + 1) + d_x(y - 1)) + (d_x(z + 1) + d_x(z - 1)),
//   D_y and D_z likewise, in units of F / 12 (EDGE: F itself is given, the
// sums are scaled here).  Differences come before every sum: the fields vary
// little from node to node, and a difference of sums 2 F + s_x + s_y (one
// instruction less) doubled the error of D_z against 64-bit significands.
// d_z of the plane before the newest is exchanged beside that plane, from the
// entries each thread kept of the two planes before.
template <bool EDGE>
__global__ void __launch_bounds__(TX* TY) k_grad(const __grid_constant__ Box B, const __grid_constant__ Tiles T, int ncomp,
                                                 const double* __restrict__ F, double* __restrict__ out)
{
    __shared__ double fs[TY + 2][TX + 2], dzs[TY + 2][TX + 2], dxs[TY + 2][TX], dys[TY][TX + 2];
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * TX + tx;
    int x0, y0, za, zb;
    tile_of(T, 0, 0, x0, y0, za, zb);
    const int x = x0 + tx, y = y0 + ty;
    const int c = blockIdx.y;
    const double* Fc = F + (long long)c * B.Ne;
    const bool mine = x < B.n[0] && y < B.n[1];
    int off[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int i = t + k * TX * TY, ly = i / (TX + 2), lx = i - ly * (TX + 2);
        int rx = x0 - 1 + lx, ry = y0 - 1 + ly;
        off[k] = -1;
        if (i < (TX + 2) * (TY + 2) && rx <= B.n[0] && ry <= B.n[1]) {
            wrap(B, 0, rx);
            wrap(B, 1, ry);
            off[k] = (ry + B.pad[1]) * B.ne[0] + (rx + B.pad[0]);
        }
    }
    const unsigned ne01 = (unsigned)B.ne[0] * B.ne[1];
    double dxa = 0.0, dxb = 0.0, rxb = 0.0, dya = 0.0, dyb = 0.0, ryb = 0.0;
    double fa[2] = {0.0, 0.0}, fb[2] = {0.0, 0.0};  // this thread's entries of planes p - 2 and p - 1
    for (int p = za - 1; p <= zb; p++) {
        int pz = p;
        wrap(B, 2, pz);
        const double* fp = Fc + (unsigned)(pz + B.pad[2]) * ne01;
#pragma unroll
        for (int k = 0; k < 2; k++)
            if (off[k] >= 0) {
                const double v = __ldg(fp + off[k]);
                (&fs[0][0])[t + k * TX * TY] = v;
                (&dzs[0][0])[t + k * TX * TY] = v - fa[k];
                fa[k] = fb[k];
                fb[k] = v;
            }
        __syncthreads();
        const double e = fs[ty + 1][tx + 2], w = fs[ty + 1][tx], n = fs[ty + 2][tx + 1], s = fs[ty][tx + 1];
        const double dx = e - w, dy = n - s;
        dxs[ty + 1][tx] = dx;
        dys[ty][tx + 1] = dy;
        // the rims: d_x of the rows beside the tile, d_y of the columns
        if (ty < 2) dxs[ty * (TY + 1)][tx] = fs[ty * (TY + 1)][tx + 2] - fs[ty * (TY + 1)][tx];
        else if (ty == 2 && tx < 2 * TY) {
            const int r = tx >> 1, col = (tx & 1) * (TX + 1);
            dys[r][col] = fs[r + 2][col] - fs[r][col];
        }
        const double rz = fma(2.0, dzs[ty + 1][tx + 1],
                              (dzs[ty + 1][tx + 2] + dzs[ty + 1][tx]) + (dzs[ty + 2][tx + 1] + dzs[ty][tx + 1]));
        __syncthreads();
        const double rx = fma(2.0, dx, dxs[ty][tx] + dxs[ty + 2][tx]);
        const double ry = fma(2.0, dy, dys[ty][tx] + dys[ty][tx + 2]);
        if (p > za && mine) {
            const unsigned v = ((unsigned)(p - 1) * B.n[1] + (unsigned)y) * (unsigned)B.n[0] + (unsigned)x;
            double* o = out + (long long)c * B.N + v;
            const long long comp = (long long)ncomp * B.N;
            const double gx = rxb + (dxa + dx), gy = ryb + (dya + dy);
            o[0] = EDGE ? kEdge * gx : gx;
            o[comp] = EDGE ? kEdge * gy : gy;
            o[2 * comp] = EDGE ? kEdge * rz : rz;
        }
        dxa = dxb;
        dxb = dx;
        rxb = rx;
        dya = dyb;
        dyb = dy;
        ryb = ry;
    }
}

// The same per node, from the nine opposite pairs (gradient_marches)
template <bool EDGE>
__global__ void __launch_bounds__(TBL) k_grad_nodes(const __grid_constant__ Box B, int ncomp, const double* __restrict__ F,
                                                    double* __restrict__ out)
{
    const unsigned v = blockIdx.x * TBL + threadIdx.x;
    if (v >= (unsigned)B.N) return;
    const int c = blockIdx.y;
    const double* Fc = F + (long long)c * B.Ne;
    const unsigned n0 = B.n[0], n1 = B.n[1], row = v / n0, zr = row / n1;
    // offsets of the sites r + c per axis in the padded lattice
    unsigned o[3][3];
    {
        const int r[3] = {(int)(v - row * n0), (int)(row - zr * n1), (int)zr};
        const unsigned st[3] = {1u, (unsigned)B.ne[0], (unsigned)B.ne[0] * (unsigned)B.ne[1]};
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int cc = -1; cc <= 1; cc++) {
                int q = r[a] + cc;
                wrap(B, a, q);
                o[a][cc + 1] = (unsigned)(q + B.pad[a]) * st[a];
            }
    }
    double g[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const int l = 2 * k + 1;
        const double d = __ldg(Fc + (o[2][cvec(l, 2) + 1] + o[1][cvec(l, 1) + 1] + o[0][cvec(l, 0) + 1])) -
                         __ldg(Fc + (o[2][1 - cvec(l, 2)] + o[1][1 - cvec(l, 1)] + o[0][1 - cvec(l, 0)]));
        const double wd = (l <= 6 ? 2.0 : 1.0) * (EDGE ? kEdge : 1.0);
#pragma unroll
        for (int a = 0; a < 3; a++)
            if (cvec(l, a)) g[a] = fma(cvec(l, a) * wd, d, g[a]);
    }
#pragma unroll
    for (int a = 0; a < 3; a++) out[((long long)a * ncomp + c) * B.N + v] = g[a];
}

Box box_of(const cslbm_ctx* c, int order)
{
    Box B;
    B.N = c->N;
    B.Ne = 1;
    for (int a = 0; a < 3; a++) {
        B.n[a] = c->n[a];
        B.plo[a] = c->p.bc_lo[a] == CSLBM_PERIODIC;
        B.phi[a] = c->p.bc_hi[a] == CSLBM_PERIODIC;
        B.pad[a] = (B.plo[a] && B.phi[a]) ? 0 : 1;
        B.ne[a] = B.n[a] + 2 * B.pad[a];
        B.Ne *= B.ne[a];
    }
    return B;
}

cslbm_status lfail(cslbm_status s, const std::string& m) { return cslbm_record_error(s, m.c_str()); }

cslbm_status check_order(const cslbm_ctx* c, int order)
{
    if (order != 2 && order != 4) return lfail(CSLBM_EINVAL, "order must be 2 or 4");
    for (int a = 0; a < 3; a++)
        if (c->n[a] < 2) return lfail(CSLBM_EINVAL, "every axis needs at least 2 nodes");
    for (int a = 0; a < 3; a++)
        if ((c->p.bc_lo[a] != CSLBM_PERIODIC || c->p.bc_hi[a] != CSLBM_PERIODIC) && c->n[a] < order + 1)
            return lfail(CSLBM_EINVAL, "an axis with a non-periodic face needs at least order + 1 nodes");
    return CSLBM_OK;
}

size_t pad_bytes(const cslbm_ctx* c, int ncomp, int order)
{
    return (size_t)ncomp * (size_t)box_of(c, order).Ne * sizeof(double);
}

// Where the marching kernels pay.  A march takes 0.53 (k_correct), 0.76 (k_grad)
// or 0.87 (k_grad with the scaling of order 2) of a per-site kernel's time per
// site it visits, and it visits march_sites: whole tiles, and two planes more
// per chunk, which are short where the lattice has few tiles.  us, six fields,
// per-site kernels both / marches both / as chosen here:
//                        order 2             order 4
//   48 x 48 x 48          43   61   43        69   82   68   (periodic)
//   33 x 129 x 65         94  186   94       152  255  153   (periodic)
//   65 x 129 x 65        183  270  180       291  359  292   (periodic)
//   64 x 128 x 64        182  193  178       403  248  248   (walls across axis 2)
//   128 x 256 x 128     1355 1263 1262      2513 1565 1562   (walls across axis 2)
long long march_sites(const Tiles& T)
{
    const int planes = T.last - T.first;
    return (long long)T.nx * TX * T.ny * TY * (planes + 2 * ((planes + T.chunk - 1) / T.chunk));
}
bool gradient_marches(const Tiles& T, const Box& B, int order)
{
    return 100 * march_sites(T) <= (order == 2 ? 115 : 130) * B.N;
}
// A continued site of k_correct_sites costs 40 others (axes 1 and 2; across
// axis 0, where every warp has some, several hundred); without faces the march
// needs 3/4 2^20 sites to fill the device (64 x 128 x 64, one field: 57 us
// against 55, 96^3: 79 against 85).
bool correct_marches(const Tiles& T, const Box& B, int ncomp)
{
    long long in = 1;
    for (int a = 0; a < 3; a++) in *= B.n[a] - 2 * B.pad[a];
    const long long far = B.Ne - in;
    if (B.pad[0]) return true;
    return 10 * march_sites(T) <= 17 * B.Ne + 400 * far && (far || B.Ne * ncomp >= 3LL << 18);
}

cslbm_status gradient(cslbm_ctx* c, const double* f, int ncomp, int order, double* out, void* scratch, size_t bytes)
{
    if (!c || !f || !out || ncomp < 1 || ncomp > 65535) return lfail(CSLBM_EINVAL, "bad argument");
    if (cslbm_status s = check_order(c, order)) return s;
    const size_t need = pad_bytes(c, ncomp, order);
    if (!scratch || bytes < need) return lfail(CSLBM_ENOMEM, "scratch smaller than required");
    if (!cslbm_is_device_memory(f) || !cslbm_is_device_memory(out) || !cslbm_is_device_memory(scratch))
        return lfail(CSLBM_EINVAL, "fields, output and scratch must be device memory");
    const Box B = box_of(c, order);
    double* F = (double*)scratch;
    const dim3 sites((unsigned)((B.Ne + TBL - 1) / TBL), (unsigned)ncomp);
    if (order == 2) {
        k_pad<<<sites, TBL, 0, c->stream>>>(B, f, F);
    } else {
        const Tiles T = tiles_of(c->n_sm, B.ne[0], B.ne[1], -B.pad[2], B.n[2] + B.pad[2], ncomp);
        if (correct_marches(T, B, ncomp)) k_correct<<<tile_grid(T, ncomp), dim3(TX, TY), 0, c->stream>>>(B, T, f, F);
        else k_correct_sites<<<sites, TBL, 0, c->stream>>>(B, f, F);
    }
    const Tiles T = tiles_of(c->n_sm, B.n[0], B.n[1], 0, B.n[2], ncomp);
    const dim3 nodes((unsigned)((B.N + TBL - 1) / TBL), (unsigned)ncomp);
    if (gradient_marches(T, B, order)) {
        if (order == 4) k_grad<false><<<tile_grid(T, ncomp), dim3(TX, TY), 0, c->stream>>>(B, T, ncomp, F, out);
        else k_grad<true><<<tile_grid(T, ncomp), dim3(TX, TY), 0, c->stream>>>(B, T, ncomp, F, out);
    } else {
        if (order == 4) k_grad_nodes<false><<<nodes, TBL, 0, c->stream>>>(B, ncomp, F, out);
        else k_grad_nodes<true><<<nodes, TBL, 0, c->stream>>>(B, ncomp, F, out);
    }
    c->launches += 2;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return lfail(CSLBM_ECUDA, std::string("lattice gradient: ") + cudaGetErrorString(e));
    return CSLBM_OK;
}

}  // namespace lder
}  // namespace cslbm

using namespace cslbm::lder;

extern "C" {

cslbm_status cslbm_lattice_gradient_scratch_bytes(const cslbm_ctx* c, int ncomp, int order, size_t* bytes)
{
    if (!c || !bytes || ncomp < 1) return lfail(CSLBM_EINVAL, "bad argument");
    if (cslbm_status s = check_order(c, order)) return s;
    *bytes = pad_bytes(c, ncomp, order);
    return CSLBM_OK;
}

cslbm_status cslbm_lattice_gradient(cslbm_ctx* c, const double* f, int ncomp, int order, double* grad, void* scratch,
                                    size_t scratch_bytes)
{
    return gradient(c, f, ncomp, order, grad, scratch, scratch_bytes);
}

cslbm_status cslbm_metric_lattice_scratch_bytes(const cslbm_ctx* c, int order, size_t* bytes)
{
    if (!c || !bytes) return lfail(CSLBM_EINVAL, "bad argument");
    if (cslbm_status s = check_order(c, order)) return s;
    *bytes = 18 * (size_t)c->N * sizeof(double) + pad_bytes(c, 6, order);
    return CSLBM_OK;
}

cslbm_status cslbm_set_metric_lattice(cslbm_ctx* c, const double* g6, int order, void* scratch, size_t scratch_bytes)
{
    size_t need = 0;
    if (cslbm_status s = cslbm_metric_lattice_scratch_bytes(c, order, &need)) return s;
    if (!g6 || !scratch || scratch_bytes < need) return lfail(CSLBM_ENOMEM, "scratch smaller than required");
    double* dg = (double*)scratch;
    const size_t dg_bytes = 18 * (size_t)c->N * sizeof(double);
    if (cslbm_status s = gradient(c, g6, 6, order, dg, (char*)scratch + dg_bytes, scratch_bytes - dg_bytes)) return s;
    return cslbm_set_metric(c, g6, dg, 1);
}

cslbm_status cslbm_update_metric_lattice(cslbm_ctx* c, const double* g6, const double* Jnew9, int order, void* scratch,
                                         size_t scratch_bytes)
{
    size_t need = 0;
    if (cslbm_status s = cslbm_metric_lattice_scratch_bytes(c, order, &need)) return s;
    if (!g6 || !Jnew9 || !scratch || scratch_bytes < need) return lfail(CSLBM_ENOMEM, "scratch smaller than required");
    if (!cslbm_is_device_memory(Jnew9)) return lfail(CSLBM_EINVAL, "Jnew9 must be device memory");
    double* dg = (double*)scratch;
    const size_t dg_bytes = 18 * (size_t)c->N * sizeof(double);
    if (cslbm_status s = gradient(c, g6, 6, order, dg, (char*)scratch + dg_bytes, scratch_bytes - dg_bytes)) return s;
    return cslbm_update_metric(c, g6, dg, Jnew9, 1);
}

}  // extern "C"
