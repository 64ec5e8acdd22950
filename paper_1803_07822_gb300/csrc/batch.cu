// Batched form: many independent channels of uneven sizes advanced together,
// FP32 storage.
//
// Each channel is an ordinary context (its own workspace slice, metric,
// boundary velocities; every single-channel call works on it).  A time step
// of the whole batch is ONE persistent launch: a grid of CTAs, all resident
// at once (cooperative launch), takes work items -- runs of `item` nodes of
// one channel -- in turn (CTA b items b, b + grid, ...), first the momentum
// field rho u of each (the gather pass's per-node code), then, after a grid
// barrier, the step: the items of the face nodes, whose chains of loads are
// the longest, then the interior nodes.  The warps of a CTA share nothing but
// the channel tables, so none waits for another between the barriers.  A CTA
// finds an item's channel by binary search in the channels' first items, held
// in shared memory; the channel's lattice, buffers and ping-pong parities
// come from a table in device memory.  Two steps are captured once as a CUDA
// graph (barrier reset, launch, barrier reset, launch) on the batch's own
// stream and replayed; the table is re-uploaded only when a channel's buffers
// moved (a metric update, a single-channel step).  The tile shape -- nodes
// per block, nodes per work item, blocks per SM -- is picked by
// cslbm_batch_tune, which times every candidate on the batch itself with the
// same step repeated from the same input (the state does not advance).  The
// grid barrier's wait is bounded (half a second); a wait that runs out sets
// the batch's error flag, which cslbm_batch_check reports as CSLBM_ETIMEOUT.
//
// 64 channels of 32..96 per side (17.4 million nodes), us per step: items
// drawn from an atomic queue by whole blocks (two block barriers each), face
// nodes on a branch, geometry through registers (168 of them), 1,736; this,
// 1,627.  (One queue for both passes, a channel's step a little behind its
// momentum so that the populations are still in L2: 2,224.)
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <string>
#include <vector>

#include "ctx.h"
#include "make_lat.h"
#include "flat_step.cuh"

namespace cslbm {
namespace batch {

struct Chan {
    Lat L;
    float* P[2];
    float* H[2];
    const float* G;
    Mom4<float>* jf;
    Plane pl;
    FaceList f;
    int pc0, hc0;  // the context's buffers when the table was made
};

constexpr int kMaxChan = 4096;

__device__ __forceinline__ int find_chan(const unsigned* blk0, int nchan, unsigned blk)
{
    int lo = 0, hi = nchan - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (blk0[mid] <= blk) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

constexpr unsigned long long kWaitNs = 500000000ull;
constexpr int kTB[3] = {128, 256, 512};       // nodes per block
constexpr int kItemMul[3] = {1, 4, 16};       // nodes per work item, in blocks
constexpr int kItems[7] = {128, 256, 512, 1024, 2048, 4096, 8192};

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}

// every CTA of the grid here before any goes on (bounded; *err |= 1 when
// the wait ran out): the momentum field is complete for the step phase
__device__ __forceinline__ void grid_barrier(unsigned* count, int* err)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        const unsigned long long t0 = now_ns();
        unsigned v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
            if (v >= gridDim.x) break;
            if (now_ns() - t0 > kWaitNs) {
                atomicOr(err, 1);
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
}

// the step of an interior node through registers, nothing staged
__device__ __forceinline__ void step_plain(const Lat& L, const float* __restrict__ Pin, float* __restrict__ Pout,
                                           const float* __restrict__ hin, float* __restrict__ hout,
                                           const float* __restrict__ geo, const Mom4<float>* jf, int x, int y, int z,
                                           unsigned v)
{
    const unsigned N = (unsigned)L.N;
    const Nbr src = nbr_index(L, x, y, z, -1);
    float s[Q];
#pragma unroll
    for (int l = 0; l < Q; l++)
        s[l] = Store<float>::ld(Pin + (unsigned)pslot(l) * N + nbr_off(src, cvec(l, 0), cvec(l, 1), cvec(l, 2)));
    GeoT<float> G;
    HistT<float> Hp;
    load_geo_hist(geo, hin, v, N, G, Hp);
    float d[9][3];
#pragma unroll
    for (int k = 0; k < 9; k++) {
        // site x + c is the pull source of -c
        const int l = 2 * k + 1, cx = cvec(l, 0), cy = cvec(l, 1), cz = cvec(l, 2);
        const Mom4<float> p = jf[nbr_off(src, -cx, -cy, -cz)], m = jf[nbr_off(src, cx, cy, cz)];
        d[k][0] = p.x - m.x;
        d[k][1] = p.y - m.y;
        d[k][2] = p.z - m.z;
    }
    step_core<float, float>(L, s, G, Hp, d, Pout, hout, v, N);
}

// One persistent launch per LBM step of every channel (see the top of the
// file).  first[c] = first work item of channel c's nodes (items of `item`
// nodes), first[nchan] = all of them; first[nchan + 1 + c] the same for its
// face nodes; q the barrier count, zero at launch; k the parity of the step in
// the two-step cycle.
// STAGED: geometry and history through shared memory (step_interior), 512
// threads per SM at 128 registers; else step_plain, 384 at 168, which is the
// faster of the two where the nodes hardly fill one round of blocks (eight
// channels of 16..40 per side: walls 33 against 31 us per step, periodic 29
// against 25; 64 channels of 32..96: 1,634 against 1,749).  The tuner picks.
template <int TB, bool STAGED>
__global__ void __launch_bounds__(TB, (STAGED ? 512 : 384) / TB)
    k_batch_persistent(const Chan* __restrict__ tab, const unsigned* __restrict__ first, int nchan, int item, int k,
                       unsigned* q, int* err)
{
    extern __shared__ __align__(16) unsigned char smem_batch[];
    float* stage = reinterpret_cast<float*>(smem_batch);
    unsigned* sb = reinterpret_cast<unsigned*>(stage + kStaged<float, false> * TB);
    for (int i = threadIdx.x; i < 2 * (nchan + 1); i += TB) sb[i] = first[i];
    __syncthreads();
    const unsigned* sf = sb + nchan + 1;
    const unsigned nitems = sb[nchan], nfaces = sf[nchan];
    for (unsigned w = blockIdx.x; w < nitems; w += gridDim.x) {
        const int c = find_chan(sb, nchan, w);
        const Chan& C = tab[c];
        const unsigned v0 = (w - sb[c]) * (unsigned)item, v1 = min(v0 + (unsigned)item, (unsigned)C.L.N);
        const int pi = (C.pc0 + k) & 1, hi = (C.hc0 + k) & 1;
        for (unsigned v = v0 + threadIdx.x; v < v1; v += TB) {
            int x, y, z;
            flat_coords(C.L, C.pl, v, x, y, z);
            momentum_node<float, float, true>(C.L, C.P[pi], C.H[hi], C.G, C.jf, x, y, z, v);
        }
    }
    grid_barrier(q, err);
    for (unsigned w = blockIdx.x; w < nfaces; w += gridDim.x) {
        const int c = find_chan(sf, nchan, w);
        const Chan& C = tab[c];
        const unsigned i0 = (w - sf[c]) * (unsigned)item;
        const int pi = (C.pc0 + k) & 1, hi = (C.hc0 + k) & 1;
        int x, y, z;
        for (unsigned i = i0 + threadIdx.x; i < i0 + (unsigned)item && face_coords(C.f, (int)i, x, y, z); i += TB)
            step_face<float, float>(C.L, C.P[pi], C.P[pi ^ 1], C.H[hi], C.H[hi ^ 1], C.G, C.jf, x, y, z);
    }
    // (the block's turn continues where the faces left it)
    for (unsigned u = (blockIdx.x + gridDim.x - nfaces % gridDim.x) % gridDim.x; u < nitems; u += gridDim.x) {
        const unsigned w = nitems - 1 - u;  // the momentum pass's last populations are still in L2
        const int c = find_chan(sb, nchan, w);
        const Chan& C = tab[c];
        const unsigned v0 = (w - sb[c]) * (unsigned)item, v1 = min(v0 + (unsigned)item, (unsigned)C.L.N);
        const int pi = (C.pc0 + k) & 1, hi = (C.hc0 + k) & 1;
        for (unsigned v = v0 + threadIdx.x; v < v1; v += TB) {
            int x, y, z;
            flat_coords(C.L, C.pl, v, x, y, z);
            if (on_boundary(C.L, x, y, z)) continue;
            if constexpr (STAGED)
                step_interior<float, float, TB, false>(C.L, C.P[pi], C.P[pi ^ 1], C.H[hi], C.H[hi ^ 1], C.G, C.jf, x, y, z,
                                                       v, stage + threadIdx.x);
            else
                step_plain(C.L, C.P[pi], C.P[pi ^ 1], C.H[hi], C.H[hi ^ 1], C.G, C.jf, x, y, z, v);
        }
    }
}

template <int TB> size_t smem_bytes(int nchan)
{
    return (size_t)kStaged<float, false> * TB * sizeof(float) + 2 * (size_t)(nchan + 1) * sizeof(unsigned);
}

}  // namespace batch
}  // namespace cslbm

using cslbm::batch::Chan;

struct Shape {
    int tb;    // index into kTB
    int item;  // nodes per work item
    int bps;   // blocks per SM; with 128 threads three are those of the kernel that stages nothing
};

struct cslbm_batch {
    int nb;
    std::vector<cslbm_ctx*> ctx;
    cudaStream_t user;    // the caller's stream
    cudaStream_t stream;  // the batch's own stream (graphs are captured on it)
    cudaEvent_t ev_in, ev_out, t0, t1;
    Chan* d_tab;          // [nb] in the workspace
    unsigned* d_first;    // [7][2][nb + 1]: first work item of each channel's nodes and faces, per item size of kItems
    unsigned* d_q;        // [4]: barrier count, unused
    int* d_err;           // grid-barrier timeout flag
    std::vector<Chan> h_tab;
    std::vector<unsigned> h_first;
    int n_sm;
    Shape shape;
    std::vector<Shape> cand;  // the tuner's candidates, and their times
    std::vector<float> cand_ms;
    cudaGraphExec_t graph;    // two steps
    Shape graph_shape;
    int have_table;
    long long launches;
};

namespace {

size_t al(size_t x) { return (x + 255) & ~size_t(255); }

cslbm_status bfail(cslbm_status s, const std::string& m) { return cslbm_record_error(s, m.c_str()); }

#define BCUDA(x)                                                                                          \
    do {                                                                                                  \
        cudaError_t e_ = (x);                                                                             \
        if (e_ != cudaSuccess) return bfail(CSLBM_ECUDA, std::string(#x ": ") + cudaGetErrorString(e_)); \
    } while (0)

bool same(const Shape& a, const Shape& b) { return a.tb == b.tb && a.item == b.item && a.bps == b.bps; }

int item_index(int item)
{
    for (int i = 0; i < 7; i++)
        if (cslbm::batch::kItems[i] == item) return i;
    return 0;
}

bool table_current(const cslbm_batch* b)
{
    if (!b->have_table) return false;
    for (int i = 0; i < b->nb; i++) {
        const cslbm_ctx* c = b->ctx[i];
        const Chan& t = b->h_tab[i];
        if (t.pc0 != c->pc || t.hc0 != c->hc || t.G != (const float*)c->G[c->gc]) return false;
    }
    return true;
}

cslbm_status upload_table(cslbm_batch* b)
{
    for (int i = 0; i < b->nb; i++) {
        const cslbm_ctx* c = b->ctx[i];
        Chan& t = b->h_tab[i];
        t.L = cslbm::make_lat(c);
        for (int k = 0; k < 2; k++) {
            t.P[k] = (float*)c->P[k];
            t.H[k] = (float*)c->H[k];
        }
        t.G = (const float*)c->G[c->gc];
        t.jf = (cslbm::Mom4<float>*)c->jf;
        t.pl = cslbm::make_plane(t.L);
        t.f = cslbm::face_list(c);
        t.pc0 = c->pc;
        t.hc0 = c->hc;
    }
    BCUDA(cudaMemcpyAsync(b->d_tab, b->h_tab.data(), b->nb * sizeof(Chan), cudaMemcpyHostToDevice, b->stream));
    BCUDA(cudaStreamSynchronize(b->stream));
    b->have_table = 1;
    return CSLBM_OK;
}

template <int TB, bool STAGED = true>
cudaError_t launch_tb(cslbm_batch* b, const Shape& sh, int k, cudaStream_t s)
{
    const unsigned* first = b->d_first + item_index(sh.item) * 2 * (b->nb + 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(sh.bps * b->n_sm));
    cfg.blockDim = dim3(TB);
    cfg.dynamicSmemBytes = cslbm::batch::smem_bytes<TB>(b->nb);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cslbm::batch::k_batch_persistent<TB, STAGED>, (const Chan*)b->d_tab, first,
                              b->nb, sh.item, k, b->d_q, b->d_err);
}

// one LBM step of every channel: the barrier reset, then one persistent launch
cudaError_t launch_step(cslbm_batch* b, const Shape& sh, int k, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(b->d_q, 0, 4 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    switch (sh.tb) {
    case 0: return sh.bps == 3 ? launch_tb<128, false>(b, sh, k, s) : launch_tb<128>(b, sh, k, s);
    case 1: return launch_tb<256>(b, sh, k, s);
    default: return launch_tb<512>(b, sh, k, s);
    }
}

template <int TB, bool STAGED> int occupancy_tb(const cslbm_batch* b)
{
    // (the most channels a batch can have, so that the attribute serves every batch)
    cslbm::set_smem_optin_once<cslbm::batch::k_batch_persistent<TB, STAGED>>(
        b->ctx[0]->device, (int)cslbm::batch::smem_bytes<TB>(cslbm::batch::kMaxChan));
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, cslbm::batch::k_batch_persistent<TB, STAGED>, TB,
                                                  cslbm::batch::smem_bytes<TB>(b->nb));
    return occ;
}
int occupancy(const cslbm_batch* b, int tb)
{
    switch (tb) {
    case 0: return occupancy_tb<128, true>(b);
    case 1: return occupancy_tb<256, true>(b);
    default: return occupancy_tb<512, true>(b);
    }
}
// may the batch launch with this shape's block size and blocks per SM?
bool resident(const cslbm_batch* b, int tb, int bps)
{
    return bps >= 1 && bps <= occupancy(b, tb) && (tb != 0 || bps != 3 || occupancy_tb<128, false>(b) >= 3);
}

cslbm_status make_graph(cslbm_batch* b)
{
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    cudaGraph_t g;
    BCUDA(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t e0 = launch_step(b, b->shape, 0, b->stream);
    cudaError_t e1 = e0 == cudaSuccess ? launch_step(b, b->shape, 1, b->stream) : e0;
    cudaError_t ec = cudaStreamEndCapture(b->stream, &g);
    if (e1 != cudaSuccess || ec != cudaSuccess)
        return bfail(CSLBM_ECUDA, std::string("batch step capture: ") + cudaGetErrorString(e1 != cudaSuccess ? e1 : ec));
    cudaError_t e = cudaGraphInstantiate(&b->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return bfail(CSLBM_ECUDA, std::string("graph instantiation: ") + cudaGetErrorString(e));
    b->graph_shape = b->shape;
    return CSLBM_OK;
}

}  // namespace

extern "C" {

cslbm_status cslbm_batch_workspace_bytes(int nb, const cslbm_params* p, size_t* bytes)
{
    if (nb <= 0 || nb > cslbm::batch::kMaxChan || !p || !bytes) return bfail(CSLBM_EINVAL, "bad argument");
    size_t total = 0;
    for (int i = 0; i < nb; i++) {
        if (p[i].storage != CSLBM_FP32) return bfail(CSLBM_EINVAL, "a batch holds FP32 channels only");
        size_t w = 0;
        if (cslbm_status s = cslbm_workspace_bytes(&p[i], &w)) return s;
        total += al(w);
    }
    total += al(nb * sizeof(Chan)) + al(14 * (nb + 1) * sizeof(unsigned)) + al(4 * sizeof(unsigned) + sizeof(int));
    *bytes = total;
    return CSLBM_OK;
}

cslbm_status cslbm_batch_create(int nb, const cslbm_params* p, void* workspace, size_t bytes, void* stream,
                                cslbm_batch** out)
{
    if (!out || !workspace) return bfail(CSLBM_EINVAL, "null argument");
    size_t need = 0;
    if (cslbm_status s = cslbm_batch_workspace_bytes(nb, p, &need)) return s;
    if (bytes < need) return bfail(CSLBM_ENOMEM, "workspace smaller than cslbm_batch_workspace_bytes");
    if ((uintptr_t)workspace & 255) return bfail(CSLBM_EINVAL, "workspace must be 256-byte aligned");
    cslbm_batch* b = new cslbm_batch();
    b->nb = nb;
    b->user = (cudaStream_t)stream;
    b->graph = nullptr;
    b->graph_shape = {-1, 0, 0};
    b->have_table = 0;
    b->launches = 0;
    char* base = (char*)workspace;
    size_t o = 0;
    cslbm_status st = CSLBM_OK;
    for (int i = 0; i < nb && !st; i++) {
        size_t w = 0;
        cslbm_workspace_bytes(&p[i], &w);
        cslbm_params q = p[i];
        q.step_kernel = CSLBM_STEP_FLAT;  // a channel's own steps take the same gather pass
        cslbm_ctx* c = nullptr;
        st = cslbm_create(&q, base + o, w, stream, &c);
        if (!st) b->ctx.push_back(c);
        o += al(w);
    }
    b->d_tab = (Chan*)(base + o);
    o += al(nb * sizeof(Chan));
    b->d_first = (unsigned*)(base + o);
    o += al(14 * (nb + 1) * sizeof(unsigned));
    b->d_q = (unsigned*)(base + o);
    b->d_err = (int*)(b->d_q + 4);
    b->h_tab.resize(nb);
    b->h_first.assign(14 * (nb + 1), 0);
    for (int t = 0; t < 7 && !st; t++)
        for (int kind = 0; kind < 2; kind++) {
            unsigned* f = b->h_first.data() + (2 * t + kind) * (nb + 1);
            const int item = cslbm::batch::kItems[t];
            for (int i = 0; i < nb; i++) {
                const long long n = kind ? cslbm::face_count(p[i]) : b->ctx[i]->N;
                f[i + 1] = f[i] + (unsigned)((n + item - 1) / item);
            }
        }
    bool have_stream = false;
    if (!st) {
        cudaDeviceGetAttribute(&b->n_sm, cudaDevAttrMultiProcessorCount, b->ctx[0]->device);
        b->shape = {1, 1024, 1};
        const int occ = occupancy(b, 1);
        if (occ < 1) st = bfail(CSLBM_ECUDA, "the batch kernel cannot be resident");
        else b->shape.bps = occ;
        // (an untuned batch that would leave blocks without an item: two periodic
        // channels of 16..24 per side 31 -> 15 us per step)
        long long nodes = 0;
        for (const cslbm_ctx* c : b->ctx) nodes += c->N;
        if (nodes < 1024LL * occ * b->n_sm) b->shape.item = 256;
    }
    if (!st) {
        if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess)
            st = bfail(CSLBM_ECUDA, "stream creation failed");
        else
            have_stream = true;
    }
    if (!st && (cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreate(&b->t0) != cudaSuccess || cudaEventCreate(&b->t1) != cudaSuccess))
        st = bfail(CSLBM_ECUDA, "event creation failed");
    if (!st && cudaMemcpyAsync(b->d_first, b->h_first.data(), 14 * (nb + 1) * sizeof(unsigned), cudaMemcpyHostToDevice,
                               b->stream) != cudaSuccess)
        st = bfail(CSLBM_ECUDA, "table upload failed");
    if (!st && cudaMemsetAsync(b->d_q, 0, 4 * sizeof(unsigned) + sizeof(int), b->stream) != cudaSuccess)
        st = bfail(CSLBM_ECUDA, "barrier reset failed");
    if (!st && cudaStreamSynchronize(b->stream) != cudaSuccess) st = bfail(CSLBM_ECUDA, "table upload failed");
    if (st) {
        if (have_stream) cudaStreamDestroy(b->stream);
        for (cslbm_ctx* c : b->ctx) cslbm_destroy(c);
        delete b;
        return st;
    }
    *out = b;
    return CSLBM_OK;
}

cslbm_status cslbm_batch_context(cslbm_batch* b, int i, cslbm_ctx** out)
{
    if (!b || !out || i < 0 || i >= b->nb) return bfail(CSLBM_EINVAL, "bad argument");
    *out = b->ctx[i];
    return CSLBM_OK;
}

cslbm_status cslbm_batch_step(cslbm_batch* b, int nsteps)
{
    if (!b || nsteps < 0) return bfail(CSLBM_EINVAL, "bad argument");
    for (cslbm_ctx* c : b->ctx)
        if (!c->has_state) return bfail(CSLBM_ESTATE, "a channel of the batch has no state");
    if (nsteps == 0) return CSLBM_OK;
    // the batch stream starts after the caller's queued work
    BCUDA(cudaEventRecord(b->ev_in, b->user));
    BCUDA(cudaStreamWaitEvent(b->stream, b->ev_in, 0));
    if (!table_current(b))
        if (cslbm_status s = upload_table(b)) return s;
    if (!b->graph || !same(b->graph_shape, b->shape))
        if (cslbm_status s = make_graph(b)) return s;
    for (int t = 0; t + 1 < nsteps; t += 2) {
        BCUDA(cudaGraphLaunch(b->graph, b->stream));
        b->launches += 2;
    }
    if (nsteps & 1) {
        BCUDA(launch_step(b, b->shape, 0, b->stream));
        b->launches += 1;
    }
    for (cslbm_ctx* c : b->ctx) {
        c->pc ^= nsteps & 1;
        c->hc ^= nsteps & 1;
    }
    // the caller's stream waits for the batch
    BCUDA(cudaEventRecord(b->ev_out, b->stream));
    BCUDA(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CSLBM_OK;
}

cslbm_status cslbm_batch_tune(cslbm_batch* b, int reps, int* shape3, float* ms)
{
    if (!b || reps <= 0) return bfail(CSLBM_EINVAL, "bad argument");
    for (cslbm_ctx* c : b->ctx)
        if (!c->has_state) return bfail(CSLBM_ESTATE, "a channel of the batch has no state");
    BCUDA(cudaEventRecord(b->ev_in, b->user));
    BCUDA(cudaStreamWaitEvent(b->stream, b->ev_in, 0));
    if (!table_current(b))
        if (cslbm_status s = upload_table(b)) return s;
    // candidates: block size x work-item size x blocks per SM (the resident
    // maximum, half of it, and three of 128 threads); the same step (parity 0) repeated, so every
    // repetition reads the current state and writes the spare buffers
    b->cand.clear();
    b->cand_ms.clear();
    for (int t = 0; t < 3; t++) {
        const int occ = occupancy(b, t);
        if (occ < 1) continue;
        const int bps_c[3] = {occ, occ / 2, t == 0 ? 3 : 0};
        for (int u = 0; u < 3; u++) {
            if (!resident(b, t, bps_c[u]) || (u && bps_c[u] == occ)) continue;
            for (int mi = 0; mi < 3; mi++) b->cand.push_back({t, cslbm::batch::kTB[t] * cslbm::batch::kItemMul[mi], bps_c[u]});
        }
    }
    float best = 1e30f;
    Shape best_s = b->shape;
    for (const Shape& sh : b->cand) {
        BCUDA(launch_step(b, sh, 0, b->stream));  // warm
        BCUDA(cudaEventRecord(b->t0, b->stream));
        for (int r = 0; r < reps; r++) BCUDA(launch_step(b, sh, 0, b->stream));
        BCUDA(cudaEventRecord(b->t1, b->stream));
        BCUDA(cudaEventSynchronize(b->t1));
        float e = 0.0f;
        BCUDA(cudaEventElapsedTime(&e, b->t0, b->t1));
        b->cand_ms.push_back(e / reps);
        if (e < best) {
            best = e;
            best_s = sh;
        }
    }
    b->shape = best_s;
    if (shape3) {
        shape3[0] = cslbm::batch::kTB[best_s.tb];
        shape3[1] = best_s.item;
        shape3[2] = best_s.bps;
    }
    if (ms) *ms = best / reps;
    BCUDA(cudaEventRecord(b->ev_out, b->stream));
    BCUDA(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CSLBM_OK;
}

cslbm_status cslbm_batch_set_shape(cslbm_batch* b, const int* shape3)
{
    if (!b || !shape3) return bfail(CSLBM_EINVAL, "bad argument");
    int t = -1;
    for (int k = 0; k < 3; k++)
        if (cslbm::batch::kTB[k] == shape3[0]) t = k;
    bool item_ok = false;
    for (int k = 0; k < 7; k++)
        if (cslbm::batch::kItems[k] == shape3[1]) item_ok = true;
    if (t < 0 || !item_ok || shape3[1] % shape3[0] != 0 || !resident(b, t, shape3[2]))
        return bfail(CSLBM_EINVAL, "nodes per block 128, 256 or 512; nodes per work item a multiple of it in "
                                   "128..8192 (powers of two); blocks per SM from 1 to the resident maximum");
    b->shape = {t, shape3[1], shape3[2]};
    return CSLBM_OK;
}

cslbm_status cslbm_batch_tune_results(const cslbm_batch* b, int max, int* shapes, float* ms, int* count)
{
    if (!b || !count || max < 0 || (max > 0 && (!shapes || !ms))) return bfail(CSLBM_EINVAL, "bad argument");
    const int n = (int)b->cand.size();
    *count = n;
    for (int i = 0; i < n && i < max; i++) {
        shapes[3 * i] = cslbm::batch::kTB[b->cand[i].tb];
        shapes[3 * i + 1] = b->cand[i].item;
        shapes[3 * i + 2] = b->cand[i].bps;
        ms[i] = b->cand_ms[i];
    }
    return CSLBM_OK;
}

cslbm_status cslbm_batch_check(cslbm_batch* b)
{
    if (!b) return bfail(CSLBM_EINVAL, "batch is null");
    int e = 0;
    BCUDA(cudaMemcpyAsync(&e, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
    BCUDA(cudaStreamSynchronize(b->stream));
    if (e) {
        BCUDA(cudaMemsetAsync(b->d_err, 0, sizeof(int), b->stream));
        BCUDA(cudaStreamSynchronize(b->stream));
        return bfail(CSLBM_ETIMEOUT, "the batch step's grid barrier ran out of time");
    }
    return CSLBM_OK;
}

cslbm_status cslbm_batch_launches(const cslbm_batch* b, long long* launches)
{
    if (!b || !launches) return bfail(CSLBM_EINVAL, "bad argument");
    *launches = b->launches;
    return CSLBM_OK;
}

cslbm_status cslbm_batch_destroy(cslbm_batch* b)
{
    if (!b) return bfail(CSLBM_EINVAL, "batch is null");
    cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    cudaEventDestroy(b->ev_in);
    cudaEventDestroy(b->ev_out);
    cudaEventDestroy(b->t0);
    cudaEventDestroy(b->t1);
    cudaStreamDestroy(b->stream);
    for (cslbm_ctx* c : b->ctx) cslbm_destroy(c);
    delete b;
    return CSLBM_OK;
}

}  // extern "C"
