// md_noalloc.cu -- md_forces_noalloc: forces, potential energy and virial of
// one configuration with no device allocation at all.
//
// Who needs it: callers that may not allocate device memory themselves --
// code running inside a memory pool or budget it does not own, or on a
// path where cudaMalloc/cudaFree must not run because they synchronise the
// device and would stall other streams.  They pass input and output buffers;
// every working array lives in one fixed scratch area compiled into this
// library (a file-scope __device__ array), which each GPU that loads the
// library keeps until the process exits.
//
// The computation is the FP64 form of the pair-force step: wrap, bin into
// cells of width >= r_c (counting sort, deterministic order inside each
// cell), then forces from the 27 neighbouring cells with Eq. (1) plus the
// shift, and the sums U and W.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <string>

#include "../../include/md.h"
#include "md_common.cuh"

namespace md {
// Records the message md_last_error(NULL) returns (defined with the rest of
// the C ABI; not exported).
void set_call_error(const char* msg);
}  // namespace md

namespace {

constexpr int kThreads = 256;
constexpr int kMaxAtoms = MD_NOALLOC_MAX_ATOMS;
constexpr int kMaxCells = MD_NOALLOC_MAX_CELLS;
// Lanes per atom of the force kernel, and atoms per block.
constexpr int kLanes = 8;
constexpr int kAtoms = kThreads / kLanes;
constexpr int kMaxBlocks = (kMaxAtoms + kAtoms - 1) / kAtoms;
// Pairs that one atom queues before they are evaluated (a multiple of
// kLanes, at least two of them; a fluid's atom has about five).
constexpr int kQueue = 16;
static_assert(kLanes == 8 && kQueue % kLanes == 0 && kQueue >= 2 * kLanes, "");
// Cells per block of the scan.
constexpr int kTile = 2048;
// Sizes up to which one block does all the binning (its counts and order
// fit 32 KB of shared memory).
constexpr int kSmallAtoms = 4096;
constexpr int kSmallCells = 4096;

// Byte layout of the scratch area.  The FP32 coordinates take the place of
// the counts, cells and ranks, which are no longer needed when they are
// written.
constexpr size_t kOffStart = 0;                                                          // int[kMaxCells + 1]
constexpr size_t kOffOrder = kOffStart + sizeof(int) * (kMaxCells + 64);                 // int[kMaxAtoms]
constexpr size_t kOffPosF = (kOffOrder + sizeof(int) * kMaxAtoms + 255) & ~size_t(255);  // float4[kMaxAtoms]
constexpr size_t kOffCount = kOffPosF;                                                   // int[kMaxCells]
constexpr size_t kOffCell = kOffCount + sizeof(int) * kMaxCells;                         // int[kMaxAtoms]
constexpr size_t kOffRank = kOffCell + sizeof(int) * kMaxAtoms;                          // int[kMaxAtoms]
constexpr size_t kOffPart = kOffPosF + sizeof(float4) * kMaxAtoms;                       // double[2 kMaxBlocks]
constexpr size_t kOffPos = (kOffPart + sizeof(double) * 2 * kMaxBlocks + 255) & ~size_t(255);  // double4[kMaxAtoms]
constexpr size_t kOffFlag = kOffPos + sizeof(double) * 4 * kMaxAtoms;  // int: a non-finite input was seen; ticket
constexpr size_t kScratchBytes = kOffFlag + 256;
static_assert(kOffRank + sizeof(int) * kMaxAtoms <= kOffPart, "counts, cells and ranks fit the FP32 coordinates");
static_assert(kScratchBytes <= MD_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds the declared size");

__device__ __align__(256) unsigned char g_scratch[MD_NOALLOC_SCRATCH_BYTES];

struct Geo {
    int n, ncells;
    int G[3];
    double L[3], hL[3], invL[3], invW[3];
    double rc2, ushift, irc;
    float Lf[3];    // box edges in units of r_c
    float near2;    // FP32 bound on (r / r_c)^2 that no pair inside r_c exceeds
};

struct Scratch {
    int* count;
    int* start;
    int* cell;
    int* rank;
    int* order;
    double* part;
    double* pos;    // x, y, z and (index, cell) per atom in cell order
    float4* posf;   // x, y, z in units of r_c, in cell order
    int* bad;       // set when a position is not finite
    unsigned* ticket;  // blocks of the force kernel that have finished
};

__device__ __forceinline__ int gid() { return blockIdx.x * blockDim.x + threadIdx.x; }

// Wrap one component into [-L/2, L/2) and return its cell coordinate (same
// operation order as the handle-based path).
__device__ __forceinline__ int wrap_bin(double& x, const Geo& g, int d) {
    // |x| below L/2 by more than one part in 2^21 (high words that differ by two
    // or more: by one, and x may be the number next to L/2, whose x + L/2 rounds
    // to L): neither the wrap nor the folding at the faces applies, and
    // truncation is the floor (the FP64 pipe bounds these conversions)
    if ((__double2hiint(x) & 0x7fffffff) < __double2hiint(g.hL[d]) - 1)
        return __double2int_rz(__dmul_rn(__dadd_rn(x, g.hL[d]), g.invW[d]));
    double s = floor(__dmul_rn(__dadd_rn(x, g.hL[d]), g.invL[d]));
    x = __dsub_rn(x, __dmul_rn(s, g.L[d]));
    int c = (int)floor(__dmul_rn(__dadd_rn(x, g.hL[d]), g.invW[d]));
    // a coordinate rounded onto a face belongs to the cell across it; move
    // it with its cell so the periodic shifts stay consistent
    if (c >= g.G[d]) { c -= g.G[d]; x = __dsub_rn(x, g.L[d]); }
    if (c < 0) { c += g.G[d]; x = __dadd_rn(x, g.L[d]); }
    if (c < 0 || c >= g.G[d]) c = 0;  // non-finite input; keeps indices in range
    return c;
}

__global__ void nz_zero(Geo g, Scratch s) {
    for (int c = gid(); c < g.ncells; c += gridDim.x * blockDim.x) s.count[c] = 0;
    if (gid() == 0) {
        *s.bad = 0;
        *s.ticket = 0u;
    }
}

// Cell of atom i's wrapped position; clears `finite` on a non-finite one.
__device__ __forceinline__ int bin_atom(const Geo& g, const double* __restrict__ pos, int i, bool& finite) {
    int c[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        double x = pos[3 * (size_t)i + d];
        finite = finite && isfinite(x);
        c[d] = wrap_bin(x, g, d);
    }
    return (c[2] * g.G[1] + c[1]) * g.G[0] + c[0];
}

// Writes the wrapped position of atom i to slot k of the cell order.
__device__ __forceinline__ void place_atom(const Geo& g, const Scratch& s, const double* __restrict__ pos, int i, int k) {
    double x[3];
    int c[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        x[d] = pos[3 * (size_t)i + d];
        c[d] = wrap_bin(x[d], g, d);
    }
    double2* q = reinterpret_cast<double2*>(s.pos + 4 * (size_t)k);
    q[0] = make_double2(x[0], x[1]);
    q[1] = make_double2(x[2], __hiloint2double((c[2] * g.G[1] + c[1]) * g.G[0] + c[0], i));
    s.posf[k] = make_float4((float)(x[0] * g.irc), (float)(x[1] * g.irc), (float)(x[2] * g.irc), 0.0f);
}

// Ascending order of the atom indices order[beg, end) of one cell
// (deterministic summation order).
__device__ __forceinline__ void sort_cell(int* order, int beg, int end) {
    for (int k = beg + 1; k < end; k++) {
        const int key = order[k];
        int t = k - 1;
        while (t >= beg && order[t] > key) {
            order[t + 1] = order[t];
            t--;
        }
        order[t + 1] = key;
    }
}

__global__ void __launch_bounds__(kThreads) nz_bin(Geo g, Scratch s, const double* __restrict__ pos) {
    int i = gid();
    if (i >= g.n) return;
    bool finite = true;
    const int cl = bin_atom(g, pos, i, finite);
    if (!finite) atomicExch(s.bad, 1);
    s.cell[i] = cl;
    s.rank[i] = atomicAdd(&s.count[cl], 1);
}

// Exclusive scan of one value per thread over a block of 1024.
__device__ __forceinline__ int block_scan(int v, int* warp_tot, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = warp_tot[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    total = warp_tot[31];
    return x - v + (warp > 0 ? warp_tot[warp - 1] : 0);
}

// Exclusive scan of the counts, kTile cells a block; each block first adds
// up the counts of the tiles below its own (at most 62k integers, read from
// L2 by 1024 threads at once: one block that walked all the tiles in turn
// took 51 us for 55k cells, this 5 us).
__global__ void __launch_bounds__(1024) nz_scan(Geo g, Scratch s) {
    __shared__ int warp_tot[32];
    const int below = blockIdx.x * kTile;
    int pre = 0;
    const int4* c4 = reinterpret_cast<const int4*>(s.count);
    for (int k = threadIdx.x; k < below / 4; k += 1024) {
        const int4 v = c4[k];
        pre += v.x + v.y + v.z + v.w;
    }
    int before, total;
    block_scan(pre, warp_tot, before);
    __syncthreads();
    const int c0 = below + 2 * (int)threadIdx.x;
    const int v0 = c0 < g.ncells ? s.count[c0] : 0, v1 = c0 + 1 < g.ncells ? s.count[c0 + 1] : 0;
    const int e = before + block_scan(v0 + v1, warp_tot, total);
    if (c0 < g.ncells) s.start[c0] = e;
    if (c0 + 1 < g.ncells) s.start[c0 + 1] = e + v0;
    if (blockIdx.x == 0 && threadIdx.x == 0) s.start[g.ncells] = g.n;
}

__global__ void __launch_bounds__(kThreads) nz_scatter(Geo g, Scratch s) {
    int i = gid();
    if (i >= g.n) return;
    int slot = s.start[s.cell[i]] + s.rank[i];
    if (slot >= 0 && slot < g.n) s.order[slot] = i;
}

// Sorts each cell, a thread per cell, and writes the block's slots out in cell
// order, a thread per slot (18 us for 55k cells when the cells' threads also
// wrote their atoms out).
__global__ void __launch_bounds__(kThreads) nz_place(Geo g, Scratch s, const double* __restrict__ pos) {
    const int c0 = blockIdx.x * kThreads, c = c0 + threadIdx.x;
    if (c < g.ncells) {
        const int beg = s.start[c], end = min(s.start[c + 1], g.n);
        if (end - beg > 1) sort_cell(s.order, beg, end);
    }
    __syncthreads();
    const int end = min(s.start[min(c0 + kThreads, g.ncells)], g.n);
    for (int k = s.start[c0] + threadIdx.x; k < end; k += kThreads) place_atom(g, s, pos, s.order[k], k);
}

// All of the binning in one block, for boxes of at most kSmallAtoms atoms
// and kSmallCells cells: the five launches above cost more than their work
// there.
__global__ void __launch_bounds__(1024) nz_bin_small(Geo g, Scratch s, const double* __restrict__ pos) {
    __shared__ int s_start[kSmallCells];
    __shared__ int s_order[kSmallAtoms];
    __shared__ int warp_tot[32];
    const int tid = threadIdx.x;
    if (tid == 0) *s.ticket = 0u;
    for (int c = tid; c < kSmallCells; c += 1024) s_start[c] = 0;
    __syncthreads();
    constexpr int kPer = kSmallAtoms / 1024;
    int cl[kPer], rank[kPer];
    bool finite = true;
#pragma unroll
    for (int u = 0; u < kPer; u++) {
        const int i = u * 1024 + tid;
        cl[u] = 0;
        rank[u] = 0;
        if (i < g.n) {
            cl[u] = bin_atom(g, pos, i, finite);
            rank[u] = atomicAdd(&s_start[cl[u]], 1);
        }
    }
    const int bad = __syncthreads_or(!finite);
    if (tid == 0) *s.bad = bad ? 1 : 0;
    constexpr int kCells = kSmallCells / 1024;
    int v[kCells], sum = 0, total;
#pragma unroll
    for (int u = 0; u < kCells; u++) {
        v[u] = s_start[kCells * tid + u];
        sum += v[u];
    }
    int e = block_scan(sum, warp_tot, total);
#pragma unroll
    for (int u = 0; u < kCells; u++) {
        const int c = kCells * tid + u;
        s_start[c] = e;
        if (c < g.ncells) s.start[c] = e;
        e += v[u];
    }
    if (tid == 0) s.start[g.ncells] = g.n;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; u++) {
        const int i = u * 1024 + tid;
        if (i < g.n) s_order[s_start[cl[u]] + rank[u]] = i;
    }
    __syncthreads();
    for (int c = tid; c < g.ncells; c += 1024) {
        const int end = c + 1 < kSmallCells ? s_start[c + 1] : g.n;
        if (end - s_start[c] > 1) sort_cell(s_order, s_start[c], end);
    }
    __syncthreads();
    for (int k = tid; k < g.n; k += 1024) place_atom(g, s, pos, s_order[k], k);
}

// Forces on every atom from the 27 cells around its cell, and the sums of
// 1/2 sum_j u and 1/2 sum_j r.f (each pair is seen from both atoms).
//
// What bounds it is the FP64 pipe, which takes 16 clocks for a warp's
// instruction however few of its lanes are active, and for small boxes the
// chain of dependent loads.  So kLanes lanes share an atom.  They first test
// its candidates in FP32, on coordinates in units of r_c with a bound
// (Geo::near2) that no pair inside r_c exceeds, and queue the survivors in
// shared memory, in a fixed order; then they evaluate the queued pairs in
// FP64, one a lane, with the exact test.  The three cells of a row along x
// are one run of the cell order; the cell across the periodic face, when
// there is one, is a second run.  A thread per atom doing everything in FP64
// as it went took 226 us for 65000 atoms and 123 us for 500 (the length of
// one thread's chain).
__global__ void __launch_bounds__(kThreads, 4) nz_force(Geo g, Scratch s, double* __restrict__ f, double* __restrict__ out) {
    __shared__ int s_queue[kAtoms * kQueue];
    __shared__ double s_sum[5][kThreads];
    __shared__ double s_uw[2][kAtoms];
    __shared__ int s_last;
    constexpr unsigned kFull = 0xffffffffu;
    const int sub = threadIdx.x % kLanes, al = threadIdx.x / kLanes;
    const int k0 = blockIdx.x * kAtoms + al;
    const bool in = k0 < g.n;
    const int k = in ? k0 : g.n - 1;
    const unsigned gshift = (threadIdx.x & 31) / kLanes * kLanes;
    const unsigned below = (1u << sub) - 1u;
    int* queue = s_queue + al * kQueue;
    const double2* qi = reinterpret_cast<const double2*>(s.pos + 4 * (size_t)k);
    const double2 q0 = qi[0], q1 = qi[1];
    const double xi = q0.x, yi = q0.y, zi = q1.x;
    const float4 qf = s.posf[k];
    const int i = __double2loint(q1.y);
    const int cl = __double2hiint(q1.y);
    const int cx = cl % g.G[0], cyz = cl / g.G[0];
    const int cy = cyz % g.G[1], cz = cyz / g.G[1];
    double fx = 0.0, fy = 0.0, fz = 0.0, uu = 0.0, ww = 0.0;

    // evaluates the first nq queued pairs of this atom, one a lane
    auto evaluate = [&](int nq) {
        __syncwarp();
        for (int p = sub; __any_sync(kFull, p < nq); p += kLanes) {
            if (p >= nq) continue;
            const int rec = queue[p];
            const int t = rec & 0xffff, r = (rec >> 16) & 15, wrapped = rec >> 20;
            const double2* qj = reinterpret_cast<const double2*>(s.pos + 4 * (size_t)t);
            const double2 p0 = qj[0], p1 = qj[1];
            double ex = xi - p0.x, ey = yi - p0.y, ez = zi - p1.x;
            const int y = cy + r % 3 - 1, z = cz + r / 3 - 1;
            if (wrapped) ex += cx == 0 ? g.L[0] : -g.L[0];
            if (y < 0 || y >= g.G[1]) ey += y < 0 ? g.L[1] : -g.L[1];
            if (z < 0 || z >= g.G[2]) ez += z < 0 ? g.L[2] : -g.L[2];
            const double r2 = fma(ez, ez, fma(ey, ey, ex * ex));
            if (r2 < g.rc2) {
                const double ir2 = md::reciprocal(r2);
                const double ir6 = ir2 * ir2 * ir2;
                const double fr = fma(48.0, ir6, -24.0) * ir6 * ir2;
                fx = fma(fr, ex, fx);
                fy = fma(fr, ey, fy);
                fz = fma(fr, ez, fz);
                uu += fma(fma(4.0, ir6, -4.0), ir6, g.ushift);
                ww = fma(fr, r2, ww);
            }
        }
        __syncwarp();
    };

    int nq = 0;
    // tests candidate t of row r and queues it; flushes a queue that the next
    // kLanes candidates might overflow
    auto test = [&](int t, bool have, const float4& c, int r, int wrapped, float bx, float by, float bz) {
        const float ex = (qf.x - c.x) + bx, ey = (qf.y - c.y) + by, ez = (qf.z - c.z) + bz;
        const bool keep = have && t != k && fmaf(ex, ex, fmaf(ey, ey, ez * ez)) < g.near2;
        const unsigned m = (__ballot_sync(kFull, keep) >> gshift) & ((1u << kLanes) - 1u);
        if (keep) queue[nq + __popc(m & below)] = t | (r << 16) | (wrapped << 20);
        nq += __popc(m);
        if (__any_sync(kFull, nq > kQueue - kLanes)) {
            evaluate(nq);
            nq = 0;
        }
    };

    // wrapped = 0: cells max(cx - 1, 0) .. min(cx + 1, G - 1); 1: the cell
    // across the face, for the atoms of the first and last cell
    const bool edge = cx == 0 || cx == g.G[0] - 1;
    for (int wrapped = 0; wrapped < 2; wrapped++) {
        if (wrapped && !__any_sync(kFull, edge)) break;
        const int x0 = wrapped ? (cx == 0 ? g.G[0] - 1 : 0) : max(cx - 1, 0);
        const int x1 = wrapped ? x0 : min(cx + 1, g.G[0] - 1);
        const float bx = wrapped ? (cx == 0 ? g.Lf[0] : -g.Lf[0]) : 0.0f;
        // a plane of three rows at a time, all its loads first
        for (int dz = -1; dz <= 1; dz++) {
            int z = cz + dz;
            float bz = 0.0f;
            if (z >= g.G[2]) { z -= g.G[2]; bz = -g.Lf[2]; }
            if (z < 0) { z += g.G[2]; bz = g.Lf[2]; }
            int lo[3], hi[3];
            float by[3];
#pragma unroll
            for (int r = 0; r < 3; r++) {
                int y = cy + r - 1;
                by[r] = 0.0f;
                if (y >= g.G[1]) { y -= g.G[1]; by[r] = -g.Lf[1]; }
                if (y < 0) { y += g.G[1]; by[r] = g.Lf[1]; }
                const int row = (z * g.G[1] + y) * g.G[0];
                lo[r] = s.start[row + x0];
                hi[r] = min(s.start[row + x1 + 1], g.n);
                if (wrapped && !edge) hi[r] = lo[r];
            }
            float4 c[3];
#pragma unroll
            for (int r = 0; r < 3; r++) {
                const int t = lo[r] + sub;
                c[r] = t < hi[r] ? s.posf[t] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int r = 0; r < 3; r++) {
                const int row = 3 * (dz + 1) + r;
                test(lo[r] + sub, lo[r] + sub < hi[r], c[r], row, wrapped, bx, by[r], bz);
                // rows longer than kLanes (few)
                for (int t = lo[r] + sub + kLanes; __any_sync(kFull, t - sub < hi[r]); t += kLanes) {
                    const bool have = t < hi[r];
                    const float4 d = have ? s.posf[t] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    test(t, have, d, row, wrapped, bx, by[r], bz);
                }
            }
        }
    }
    evaluate(nq);

    // the lanes' partial sums: lane v of an atom adds up component v
    s_sum[0][threadIdx.x] = fx;
    s_sum[1][threadIdx.x] = fy;
    s_sum[2][threadIdx.x] = fz;
    s_sum[3][threadIdx.x] = uu;
    s_sum[4][threadIdx.x] = ww;
    __syncwarp();
    if (sub < 5) {
        const double* p = s_sum[sub] + al * kLanes;
        double t = p[0];
#pragma unroll
        for (int l = 1; l < kLanes; l++) t += p[l];
        if (sub < 3) {
            if (in) f[3 * (size_t)i + sub] = t;
        } else {
            s_uw[sub - 3][al] = in ? 0.5 * t : 0.0;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // the block's sums of U and W
        static_assert(kAtoms == 32, "one lane per atom");
        double u = s_uw[0][threadIdx.x], w = s_uw[1][threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) {
            u += __shfl_xor_sync(kFull, u, o);
            w += __shfl_xor_sync(kFull, w, o);
        }
        if (threadIdx.x == 0) {
            s.part[2 * blockIdx.x + 0] = u;
            s.part[2 * blockIdx.x + 1] = w;
            __threadfence();
            s_last = atomicAdd(s.ticket, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    // the last block adds up all blocks' sums, in a fixed order
    __threadfence();
    double u = 0.0, w = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads) {
        u += __ldcg(s.part + 2 * b + 0);
        w += __ldcg(s.part + 2 * b + 1);
    }
    for (int o = 16; o > 0; o >>= 1) {
        u += __shfl_xor_sync(kFull, u, o);
        w += __shfl_xor_sync(kFull, w, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_uw[0][threadIdx.x >> 5] = u;
        s_uw[1][threadIdx.x >> 5] = w;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < kThreads / 32; v++) {
            u += s_uw[0][v];
            w += s_uw[1][v];
        }
        out[0] = u;
        out[1] = w;
    }
}

// Address of g_scratch on the current device.  Looked up on every call (a
// cheap query): a cached address would go stale if the caller reset the
// device and the module were loaded again.
int scratch_for_current_device(void** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        md::set_call_error("no current CUDA device");
        return MD_ENODEV;
    }
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p) {
        md::set_call_error((std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e)).c_str());
        return MD_ECUDA;
    }
    *out = p;
    return MD_OK;
}

}  // namespace

extern "C" int md_forces_noalloc(const double box[3], int64_t n, double rc, double ushift, const double* pos,
                                 double* f, double* pe_vir, void* stream) {
    if (!box || !pos || !f || !pe_vir) {
        md::set_call_error("NULL argument");
        return MD_EINVAL;
    }
    if (n <= 0 || n > kMaxAtoms) {
        md::set_call_error("n must be in [1, MD_NOALLOC_MAX_ATOMS]");
        return MD_EINVAL;
    }
    if (!(rc > 0.0) || !std::isfinite(rc)) {
        md::set_call_error("rc must be positive and finite");
        return MD_EINVAL;
    }
    Geo g;
    std::memset(&g, 0, sizeof(g));
    g.n = (int)n;
    int64_t nc = 1;
    for (int d = 0; d < 3; d++) {
        if (!(box[d] > 0.0) || !std::isfinite(box[d])) {
            md::set_call_error("box edges must be positive and finite");
            return MD_EINVAL;
        }
        double gd = std::floor(box[d] / rc);
        if (gd < 3.0) {
            md::set_call_error("box edge below 3 r_c: the 27-cell neighbourhood would alias");
            return MD_EINVAL;
        }
        if (gd > (double)kMaxCells) gd = (double)kMaxCells;
        g.G[d] = (int)gd;
        nc *= g.G[d];
        g.L[d] = box[d];
        g.hL[d] = 0.5 * box[d];
        g.invL[d] = 1.0 / box[d];
        g.invW[d] = (double)g.G[d] / box[d];
    }
    if (nc > kMaxCells) {
        md::set_call_error("more cells than MD_NOALLOC_MAX_CELLS (box too large for r_c)");
        return MD_EINVAL;
    }
    g.ncells = (int)nc;
    g.rc2 = rc * rc;
    g.irc = 1.0 / rc;
    // FP32 coordinates in units of r_c: two roundings of values up to half
    // the longest edge and one of their difference put each component of a
    // separation within 3 L 2^-24 of the FP64 one
    const double delta = 3.0 * std::fmax(box[0], std::fmax(box[1], box[2])) * g.irc * 0x1p-24;
    g.near2 = (float)(1.0 + 4.0 * delta + 3.0 * delta * delta + 1e-5);
    for (int d = 0; d < 3; d++) g.Lf[d] = (float)(box[d] * g.irc);
    if (std::isnan(ushift)) ushift = std::fabs(rc - std::pow(2.0, 1.0 / 6.0)) <= 1e-12 * rc ? 1.0 : 0.0;
    g.ushift = ushift;

    void* base = nullptr;
    int r = scratch_for_current_device(&base);
    if (r) return r;
    unsigned char* b = (unsigned char*)base;
    Scratch s;
    s.count = (int*)(b + kOffCount);
    s.start = (int*)(b + kOffStart);
    s.cell = (int*)(b + kOffCell);
    s.rank = (int*)(b + kOffRank);
    s.order = (int*)(b + kOffOrder);
    s.part = (double*)(b + kOffPart);
    s.pos = (double*)(b + kOffPos);
    s.posf = (float4*)(b + kOffPosF);
    s.bad = (int*)(b + kOffFlag);
    s.ticket = (unsigned*)(b + kOffFlag + 128);

    cudaStream_t st = (cudaStream_t)stream;
    int ga = (g.n + kThreads - 1) / kThreads;
    int gc = (g.ncells + kThreads - 1) / kThreads;
    if (g.n <= kSmallAtoms && g.ncells <= kSmallCells) {
        nz_bin_small<<<1, 1024, 0, st>>>(g, s, pos);
    } else {
        nz_zero<<<gc, kThreads, 0, st>>>(g, s);
        nz_bin<<<ga, kThreads, 0, st>>>(g, s, pos);
        nz_scan<<<(g.ncells + kTile - 1) / kTile, 1024, 0, st>>>(g, s);
        nz_scatter<<<ga, kThreads, 0, st>>>(g, s);
        nz_place<<<gc, kThreads, 0, st>>>(g, s, pos);
    }
    nz_force<<<(g.n + kAtoms - 1) / kAtoms, kThreads, 0, st>>>(g, s, f, pe_vir);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        md::set_call_error((std::string("launch: ") + cudaGetErrorString(e)).c_str());
        return MD_ECUDA;
    }
    // the non-finite check: a 4-byte read of the flag into this stack
    // variable, after the call's own work on the stream
    int bad = 0;
    e = cudaMemcpyAsync(&bad, s.bad, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        md::set_call_error((std::string("flag read: ") + cudaGetErrorString(e)).c_str());
        return MD_ECUDA;
    }
    if (bad) {
        md::set_call_error("non-finite position");
        return MD_EUNSTABLE;
    }
    return MD_OK;
}
