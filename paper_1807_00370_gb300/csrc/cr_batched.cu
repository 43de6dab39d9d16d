// cr_batched.cu -- many independent systems of uneven N, m, k in one
// persistent launch (the paper notes that the block formulas of a level are
// independent across blocks, Sec. 2; independent systems are independent a
// fortiori).
//
// Design.  The grid is one persistent CTA per workspace slot.  A CTA takes the
// next system from an atomic counter (systems ordered by decreasing cost, the
// longest-processing-time-first rule, so that the big systems do not start
// last) and runs the whole classic cyclic reduction of that system: for every
// level the factor chunks and the down-sweep chunks, then the up sweep, with
// the same per-chunk device functions as the level kernels (cr_core.cuh).
// Because one CTA runs the chunks of a level in order, chunk-boundary even
// blocks are completed in place (inline_fix) and no fix-up launch is needed;
// no CTA ever waits for another.  Each slot holds the stored factors of its
// current system and two ping-pong buffers for the transient level systems
// and right-hand sides, and is reused by the slot's next system.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "crsolve.h"
#include "cr_batch.cuh"

using crs::z2;

struct crsolve_batch_s {
    int32_t nsys = 0;
    std::vector<crs::SysDesc> sys;
    std::vector<int32_t> order;
    crs::BatchTiles tiles{};
    int threads = 256, device = 0, nsm = 0;
    int64_t slot_bytes = 0, nA = 0, nB = 0, nY = 0;
    int32_t nslots = 0;
    size_t smem = 0;
    size_t offSys = 0, offOrder = 0, offCounter = 0, offStatus = 0, offDbg = 0, offSlots = 0, total = 0;
    char *ws = nullptr;
    bool uploaded = false;
    cudaGraphExec_t gexec = nullptr;
    cudaGraph_t graph = nullptr;
    const void *gptr[4] = {nullptr, nullptr, nullptr, nullptr};
};

namespace {

const int kMtList[5] = {4, 8, 16, 32, 64};

void (*batch_kernel(int threads))(crs::BatchArgs) { return threads == 512 ? crs::batch_kernel512() : crs::k_batch<256>; }

// Largest dynamic shared memory k_batch may use: the device's opt-in limit
// minus the kernel's static shared memory; also raises the kernel's limit.
int batch_smem_limit(int device, int threads, size_t *limit) {
    int optin = 0;
    cudaFuncAttributes fa{};
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, batch_kernel(threads)) != cudaSuccess)
        return CRSOLVE_ECUDA;
    const int dyn = optin - (int)fa.sharedSizeBytes;
    if (dyn <= 0 || cudaFuncSetAttribute(batch_kernel(threads), cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) != cudaSuccess)
        return CRSOLVE_ECUDA;
    *limit = (size_t)dyn;
    return CRSOLVE_OK;
}

size_t batch_smem(const crsolve_batch_s *b) {
    size_t smem = 0;
    bool present[5] = {false, false, false, false, false};
    for (const auto &d : b->sys) present[d.mt == 4 ? 0 : d.mt == 8 ? 1 : d.mt == 16 ? 2 : d.mt == 32 ? 3 : 4] = true;
    for (int i = 0; i < 5; ++i) {
        if (!present[i]) continue;
        smem = std::max(smem, crs::factor_smem_bytes(kMtList[i], b->tiles.nbf[i], 8));
        smem = std::max(smem, crs::solve_smem_bytes(kMtList[i], b->tiles.nbs[i], b->tiles.kc[i], 3, 8));
    }
    return smem;
}

void release_graph(crsolve_batch_s *b) {
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->gexec = nullptr;
    b->graph = nullptr;
}

// Workspace: descriptors, order, counter, per-system status, then the slots.
void layout(crsolve_batch_s *b, int32_t nslots) {
    size_t cur = 0;
    auto take = [&](size_t bytes) { size_t o = cur; cur += (bytes + 255) & ~(size_t)255; return o; };
    b->offSys = take(b->sys.size() * sizeof(crs::SysDesc));
    b->offOrder = take(b->order.size() * sizeof(int32_t));
    b->offCounter = take(sizeof(int32_t));
    b->offStatus = take(b->sys.size() * sizeof(unsigned long long));
    b->offDbg = take(sizeof(unsigned long long));
    b->offSlots = take(0);
    b->nslots = nslots;
    b->total = b->offSlots + (size_t)nslots * (size_t)b->slot_bytes;
}

int enqueue(crsolve_batch_s *b, const z2 *A, const z2 *B, const z2 *y, z2 *x, cudaStream_t s) {
    if (cudaMemsetAsync(b->ws + b->offCounter, 0, sizeof(int32_t), s) != cudaSuccess) return CRSOLVE_ECUDA;
    if (cudaMemsetAsync(b->ws + b->offStatus, 0xFF, b->sys.size() * sizeof(unsigned long long), s) != cudaSuccess)
        return CRSOLVE_ECUDA;
    crs::BatchArgs ba{};
    ba.sys = reinterpret_cast<const crs::SysDesc *>(b->ws + b->offSys);
    ba.order = reinterpret_cast<const int32_t *>(b->ws + b->offOrder);
    ba.nsys = b->nsys;
    ba.counter = reinterpret_cast<int32_t *>(b->ws + b->offCounter);
    ba.A = A; ba.B = B; ba.y = y; ba.x = x;
    ba.slots = b->ws + b->offSlots;
    ba.slot_bytes = b->slot_bytes;
    ba.status = reinterpret_cast<unsigned long long *>(b->ws + b->offStatus);
    ba.tiles = b->tiles;
    ba.dbg = reinterpret_cast<unsigned long long *>(b->ws + b->offDbg);
#ifdef CRSOLVE_DEBUG_BOUNDS
    if (cudaMemsetAsync(ba.dbg, 0xFF, sizeof(unsigned long long), s) != cudaSuccess) return CRSOLVE_ECUDA;
#endif
    batch_kernel(b->threads)<<<b->nslots, b->threads, b->smem, s>>>(ba);
    return cudaGetLastError() == cudaSuccess ? CRSOLVE_OK : CRSOLVE_ECUDA;
}

int prepare(crsolve_batch_s *b) {
    if (b->uploaded) return CRSOLVE_OK;
    size_t limit = 0;
    int rc = batch_smem_limit(b->device, b->threads, &limit);
    if (rc) return rc;
    if (b->smem > limit) return CRSOLVE_EINVAL;
    if (cudaMemcpy(b->ws + b->offSys, b->sys.data(), b->sys.size() * sizeof(crs::SysDesc), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(b->ws + b->offOrder, b->order.data(), b->order.size() * sizeof(int32_t), cudaMemcpyHostToDevice) !=
            cudaSuccess)
        return CRSOLVE_ECUDA;
    b->uploaded = true;
    return CRSOLVE_OK;
}

bool ok_ptrs(const crsolve_batch_s *b, const void *A, const void *B, const void *y, const void *x) {
    if (!A || !y || !x || (b->nB > 0 && !B)) return false;
    return ((((uintptr_t)A | (uintptr_t)B | (uintptr_t)y | (uintptr_t)x) & 15u) == 0) && x != y;
}

}  // namespace

extern "C" {

int crsolve_batch_create(int32_t nsys, const int64_t *N, const int32_t *m, const int32_t *k, crsolve_batch *out) {
    if (!out) return CRSOLVE_EINVAL;
    *out = nullptr;
    if (nsys < 1 || !N || !m || !k) return CRSOLVE_EINVAL;
    for (int32_t i = 0; i < nsys; ++i) {
        if (N[i] < 1 || m[i] < 1 || k[i] < 1) return CRSOLVE_EINVAL;
        if (m[i] > CRSOLVE_MAX_M || k[i] > CRSOLVE_MAX_K) return CRSOLVE_EUNSUPPORTED;
    }
    crsolve_batch_s *b = new (std::nothrow) crsolve_batch_s();
    if (!b) return CRSOLVE_ENOMEM;
    b->nsys = nsys;
    b->sys.resize(nsys);
    std::vector<double> cost(nsys);
    int64_t oA = 0, oB = 0, oY = 0;
    for (int32_t i = 0; i < nsys; ++i) {
        crs::SysDesc &d = b->sys[i];
        d.N = N[i]; d.m = m[i]; d.k = k[i]; d.mt = crs::pick_mt(m[i]); d.pad = 0;
        d.offA = oA; d.offB = oB; d.offY = oY;
        oA += N[i] * (int64_t)m[i] * m[i];
        oB += (N[i] - 1) * (int64_t)m[i] * m[i];
        oY += N[i] * (int64_t)m[i] * k[i];
        const double md = m[i];
        cost[i] = (double)N[i] * (25.33 * md * md * md + 40.0 * md * md * k[i]);
        b->slot_bytes = std::max(b->slot_bytes, crs::slot_layout(N[i], m[i], k[i], -1, nullptr));
    }
    b->nA = oA; b->nB = oB; b->nY = oY;
    b->order.resize(nsys);
    std::iota(b->order.begin(), b->order.end(), 0);
    std::stable_sort(b->order.begin(), b->order.end(), [&](int32_t a, int32_t c) { return cost[a] > cost[c]; });
    // default tiles per block-size class: odd blocks per chunk (factor, solve), rhs columns
    const int nbf[5] = {16, 8, 4, 2, 1}, nbs[5] = {16, 8, 4, 2, 1}, kc[5] = {16, 16, 16, 16, 16};
    for (int i = 0; i < 5; ++i) { b->tiles.nbf[i] = nbf[i]; b->tiles.nbs[i] = nbs[i]; b->tiles.kc[i] = kc[i]; }
    if (cudaGetDevice(&b->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&b->nsm, cudaDevAttrMultiProcessorCount, b->device) != cudaSuccess) {
        delete b;
        return CRSOLVE_ECUDA;
    }
    // A system runs in one CTA, so a batch lasts at least as long as its largest
    // system.  Where that system has more than its share of 2 CTAs per SM, the
    // batch runs CTAs of 512 threads, one per SM, with chunks of twice the blocks
    // where they fit: 512 systems of N <= 4096, m = 4 .. 32 took 479 ms at 256 threads
    // and 246 so (263 since small results take FMAs).
    const double total = std::accumulate(cost.begin(), cost.end(), 0.0);
    const double largest = *std::max_element(cost.begin(), cost.end());
    if (largest * 2 * b->nsm > total) {
        b->threads = 512;
        const int nb2[5] = {16, 16, 8, 4, 1};
        for (int i = 0; i < 5; ++i) b->tiles.nbf[i] = b->tiles.nbs[i] = nb2[i];
    }
    b->smem = batch_smem(b);
    *out = b;
    return CRSOLVE_OK;
}

int crsolve_batch_tile_set(crsolve_batch b, int32_t mt, int32_t nb_factor, int32_t nb_solve, int32_t kc) {
    if (!b || b->ws) return CRSOLVE_EINVAL;
    int i = -1;
    for (int j = 0; j < 5; ++j)
        if (kMtList[j] == mt) i = j;
    if (i < 0 || nb_factor < 1 || nb_solve < 1 || kc < 1 || kc > CRSOLVE_MAX_K) return CRSOLVE_EINVAL;
    b->tiles.nbf[i] = nb_factor; b->tiles.nbs[i] = nb_solve; b->tiles.kc[i] = kc;
    b->smem = batch_smem(b);
    size_t limit = 0;
    const int rc = batch_smem_limit(b->device, b->threads, &limit);
    if (rc) return rc;
    return b->smem <= limit ? CRSOLVE_OK : CRSOLVE_EINVAL;
}

int crsolve_batch_workspace_bytes(crsolve_batch b, size_t max_bytes, size_t *bytes, int32_t *nslots) {
    if (!b || !bytes) return CRSOLVE_EINVAL;
    int per_sm = 0;
    size_t limit = 0;
    int rc = batch_smem_limit(b->device, b->threads, &limit);
    if (rc) return rc;
    if (b->smem > limit) return CRSOLVE_EINVAL;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel(b->threads), b->threads, b->smem) != cudaSuccess)
        return CRSOLVE_ECUDA;
    if (per_sm < 1) return CRSOLVE_EINVAL;
    int64_t want = std::min<int64_t>((int64_t)per_sm * b->nsm, b->nsys);
    layout(b, 0);
    if (max_bytes) {
        const int64_t fit = ((int64_t)max_bytes - (int64_t)b->offSlots) / b->slot_bytes;
        if (fit < 1) return CRSOLVE_ENOMEM;
        want = std::min(want, fit);
    }
    layout(b, (int32_t)want);
    *bytes = b->total;
    if (nslots) *nslots = b->nslots;
    return CRSOLVE_OK;
}

int crsolve_batch_set_workspace(crsolve_batch b, void *dev_ptr, size_t bytes) {
    if (!b || !dev_ptr || ((uintptr_t)dev_ptr & 255u) || b->nslots < 1) return CRSOLVE_EINVAL;
    if (bytes < b->total) return CRSOLVE_ENOMEM;
    b->ws = static_cast<char *>(dev_ptr);
    b->uploaded = false;
    release_graph(b);
    return CRSOLVE_OK;
}

int crsolve_batch_offsets(crsolve_batch b, int64_t *offA, int64_t *offB, int64_t *offY, int64_t *totals) {
    if (!b) return CRSOLVE_EINVAL;
    for (int32_t i = 0; i < b->nsys; ++i) {
        if (offA) offA[i] = b->sys[i].offA;
        if (offB) offB[i] = b->sys[i].offB;
        if (offY) offY[i] = b->sys[i].offY;
    }
    if (totals) { totals[0] = b->nA; totals[1] = b->nB; totals[2] = b->nY; }
    return CRSOLVE_OK;
}

int crsolve_batch_solve(crsolve_batch b, const crsolve_z *A, const crsolve_z *B, const crsolve_z *y, crsolve_z *x,
                        void *stream) {
    if (!b || !ok_ptrs(b, A, B, y, x)) return CRSOLVE_EINVAL;
    if (!b->ws) return CRSOLVE_ENOMEM;
    int rc = prepare(b);
    if (rc) return rc;
    return enqueue(b, reinterpret_cast<const z2 *>(A), reinterpret_cast<const z2 *>(B),
                   reinterpret_cast<const z2 *>(y), reinterpret_cast<z2 *>(x), static_cast<cudaStream_t>(stream));
}

int crsolve_batch_graph_launch(crsolve_batch b, const crsolve_z *A, const crsolve_z *B, const crsolve_z *y,
                               crsolve_z *x, void *stream) {
    if (!b || !ok_ptrs(b, A, B, y, x)) return CRSOLVE_EINVAL;
    if (!b->ws) return CRSOLVE_ENOMEM;
    int rc = prepare(b);
    if (rc) return rc;
    const void *ptrs[4] = {A, B, y, x};
    if (!b->gexec || memcmp(ptrs, b->gptr, sizeof(ptrs)) != 0) {
        release_graph(b);
        cudaStream_t cs;
        if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return CRSOLVE_ECUDA;
        rc = CRSOLVE_OK;
        if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) rc = CRSOLVE_ECUDA;
        if (!rc) rc = enqueue(b, reinterpret_cast<const z2 *>(A), reinterpret_cast<const z2 *>(B),
                              reinterpret_cast<const z2 *>(y), reinterpret_cast<z2 *>(x), cs);
        cudaGraph_t g = nullptr;
        if (cudaStreamEndCapture(cs, &g) != cudaSuccess && !rc) rc = CRSOLVE_ECUDA;
        cudaStreamDestroy(cs);
        if (!rc && cudaGraphInstantiate(&b->gexec, g, 0) != cudaSuccess) rc = CRSOLVE_ECUDA;
        b->graph = g;
        if (rc) { release_graph(b); return rc; }
        memcpy(b->gptr, ptrs, sizeof(ptrs));
    }
    return cudaGraphLaunch(b->gexec, static_cast<cudaStream_t>(stream)) == cudaSuccess ? CRSOLVE_OK : CRSOLVE_ECUDA;
}

int crsolve_batch_debug_bounds(crsolve_batch b, uint64_t *record, void *stream) {
    if (!b || !record) return CRSOLVE_EINVAL;
#ifdef CRSOLVE_DEBUG_BOUNDS
    if (!b->ws) return CRSOLVE_ENOMEM;
    unsigned long long v = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&v, b->ws + b->offDbg, sizeof(v), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return CRSOLVE_ECUDA;
    *record = v;
    return CRSOLVE_OK;
#else
    (void)stream;
    *record = ~0ull;
    return CRSOLVE_EUNSUPPORTED;
#endif
}

int crsolve_batch_info(crsolve_batch b, crsolve_info *out, void *stream) {
    if (!b || !out) return CRSOLVE_EINVAL;
    if (!b->ws) return CRSOLVE_ENOMEM;
    std::vector<unsigned long long> st(b->nsys);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(st.data(), b->ws + b->offStatus, st.size() * sizeof(unsigned long long),
                        cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return CRSOLVE_ECUDA;
    for (int32_t i = 0; i < b->nsys; ++i) {
        if (st[i] == CRS_NO_FAIL) {
            out[i] = crsolve_info{CRSOLVE_OK, 0, 0, 0};
        } else {
            const int level = (int)(st[i] >> 40);
            const int64_t block = (int64_t)(st[i] & ((1ull << 40) - 1));
            out[i] = crsolve_info{CRSOLVE_NOT_PD, level, block, block << level};
        }
    }
    return CRSOLVE_OK;
}

int crsolve_batch_destroy(crsolve_batch b) {
    if (!b) return CRSOLVE_EINVAL;
    release_graph(b);
    delete b;
    return CRSOLVE_OK;
}

}  // extern "C"
