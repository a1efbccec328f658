// md_run.cuh -- the steps of a small system in one cooperative launch.
//
// What bounds a small system is latency: at 2048 atoms a graph's step kernel,
// its closing kernel and a third of a conditional node took about 11 us per
// step and a rebuild's eight kernels 50 us, for work of about a microsecond.
// k_run keeps one system's whole step loop (Sec. 3.1 (a)-(e)) on the chip:
// four lanes share an atom, every thread keeps its part of the atom's state
// and list in registers from step to step, and the blocks meet at one grid
// barrier per step, which also says whether the lists are still good.  A step is
// then one gather of pair coordinates from L2, the pair terms, and the
// barrier.  The mixed form's force sums are integers, so the trajectory is
// the one of the step kernels, bit for bit.
//
// k_run_cells does the same for the cell-list-only variant, in both forms: its
// rebuild at every step leaves nothing to keep in registers, but saves the ten
// launches of a step.
//
// Included by md_kernels.cuh.
#pragma once

namespace md {

constexpr int kRunRegs = 4;    // entries a lane keeps in registers: 16 per atom (12 in a fluid's list)
constexpr int kRunStage = 10;  // candidates a lane of the build stages (an atom's four lanes: 40)
static_assert(kRunRegs % 2 == 0, "entries are evaluated in pairs");
static_assert(kRunLanes * kRunStage < 256, "one byte per shell bin in a 64-bit word");

// What the blocks tell one another at a barrier.
constexpr int kRunFar = 1;   // some atom has moved skin/2: rebuild
constexpr int kRunStop = 2;  // an error: end the run

// The grid barrier.  Barrier number `epoch` has the 64-bit word
// words[epoch mod 4] (a line each, zero before its use): every block adds 1
// to the low 16 bits on arrival, 1 to the next 16 for kRunFar and to the
// next for kRunStop, and waits until the low 16 have reached the number of
// blocks, so that one word read tells it everything.  Block 0 clears the
// word of the barrier before the one just passed, which every block has left;
// it is used again three barriers later.  (A word per block, polled by all
// blocks, took 3.7 us at 64 blocks and 6.5 us at 209: the polls queue at the
// few lines that hold the words.)  The wait is bounded (0.33 s): a
// block that gives up records kErrWait and sees kRunStop, at which it leaves
// the loop without another barrier.
struct RunBarrier {
    unsigned long long* words;
    unsigned epoch;
    // The union of `say` over the grid; every thread of every block must call
    // it.  Writes before it are visible to all threads after it.
    __device__ __forceinline__ int sync(int say, int* sh, Counters* C) {
        epoch++;
        int any = __syncthreads_or(say);
        if (any) any = (__syncthreads_or(say & kRunFar) ? kRunFar : 0) | (__syncthreads_or(say & kRunStop) ? kRunStop : 0);
        if (threadIdx.x == 0) {
            unsigned long long* w = words + (epoch & 3u) * kRunWordStride;
            unsigned long long x = 1ull | ((any & kRunFar) ? 1ull << 16 : 0ull) | ((any & kRunStop) ? 1ull << 32 : 0ull);
            asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"(x) : "memory");
            int it = 0;
            do {
                asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w) : "memory");
            } while (((unsigned)x & 0xffffu) != gridDim.x && ++it < kRunPolls);
            int got = ((unsigned)x >> 16 ? kRunFar : 0) | ((unsigned)(x >> 32) ? kRunStop : 0);
            if (((unsigned)x & 0xffffu) != gridDim.x) {
                atomicOr(&C->error, kErrWait);
                got = kRunStop;
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if (blockIdx.x == 0) words[((epoch - 1u) & 3u) * kRunWordStride] = 0ull;
            *sh = got;
        }
        __syncthreads();
        return *sh;  // (next written after the next barrier's first __syncthreads_or)
    }
};

// The gate at the start of a loop: true in all blocks once all of them have
// begun to run, false in all of them if that takes longer than a bounded wait
// (the GPU is busy with other work and has room for some of the blocks only);
// nothing has been done then, and the host takes the graphs.  *gate (zero at
// the launch) counts the blocks that have come; the block that gives up sets
// the top bit in the same atomic operation in which it finds the count short,
// so every block sees either a full count without the bit or the bit.  Every
// thread of the block must call it.  closed: Counters::run_closed when the host
// queued the loop; a loop behind one that has not started, of the same call,
// does not start either, at once.  (A block that reads the count after another
// of its own launch has shut the gate finds it shut either way.)
__device__ __forceinline__ bool run_gate(unsigned* gate, int* sh, Counters* C, long long closed) {
    constexpr unsigned kShut = 0x80000000u;
    __syncthreads();  // the block's threads have all read the counters, which other blocks may write behind the gate
    if (threadIdx.x == 0) {
        long long now;
        asm volatile("ld.relaxed.gpu.global.s64 %0, [%1];" : "=l"(now) : "l"(&C->run_closed) : "memory");
        unsigned v = now != closed ? kShut : atomicAdd(gate, 1u) + 1u;
        for (int it = 0; it < kRunGatePolls && !(v & kShut) && v != gridDim.x; it++)
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(gate) : "memory");
        while (!(v & kShut) && v != gridDim.x) {  // (ends: another block came or this one shuts the gate)
            const unsigned w = atomicCAS(gate, v, v | kShut);
            if (w == v) atomicAdd((unsigned long long*)&C->run_closed, 1ull);
            v = w == v ? kShut : w;
        }
        *sh = !(v & kShut);
    }
    __syncthreads();
    return *sh != 0;
}

// One tile (kScanTile cells) of the exclusive scan of the cell counts, by one
// block of any size (k_scan_apply with fewer threads).
template <class P>
__device__ __forceinline__ void run_scan_tile(const Args<P>& a, int tile, int* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int carry = 0;  // atoms in the tiles below
    for (int t = lane; t < tile; t += 32) carry += __ldcg(a.tile_sum + t);
    for (int o = 16; o > 0; o >>= 1) carry += __shfl_xor_sync(0xffffffffu, carry, o);
    int mx = 0;
    const int end = min((tile + 1) * kScanTile, a.ncells);
    for (int base = tile * kScanTile; base < end; base += 4 * (int)blockDim.x) {
        const int c = base + 4 * (int)threadIdx.x;
        int v[4], tot = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            v[k] = c + k < end ? __ldcg(a.count + c + k) : 0;
            tot += v[k];
            mx = max(mx, v[k]);
        }
        int x = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();  // the last round's totals have been read
        if (lane == 31) sh[warp] = x;
        __syncthreads();
        int before = carry + x - tot;
        for (int w = 0; w < nw; w++) {
            const int t = sh[w];
            if (w < warp) before += t;
            carry += t;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (c + k < end) a.cell_start[c + k] = before;
            before += v[k];
        }
    }
    if (tile == 0 && threadIdx.x == 0) a.cell_start[a.ncells] = (int)a.n;
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0 && mx > 0) atomicMax(&a.ctr->max_occ, mx);
}

// within_rn_fp64 with all twelve numbers loaded before any is used: here the
// whole grid waits for the warp that has a pair in the band.
template <class P>
__device__ __noinline__ bool run_within_rn(const Args<P>& a, int i, int j, unsigned code) {
    int ci[3];
    const int cell = a.cell[i];
    const typename P::real bi[3] = {a.pbx[i], a.pby[i], a.pbz[i]}, bj[3] = {a.pbx[j], a.pby[j], a.pbz[j]};
    const double oi[3] = {a.ox[i], a.oy[i], a.oz[i]}, oj[3] = {a.ox[j], a.oy[j], a.oz[j]};
    unpack_cell(cell, ci[0], ci[1], ci[2]);
    double e[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        int cj = ci[k] + (int)((code >> (2 * k)) & 3u) - 1;
        double s = 0.0;
        if (cj >= a.G[k]) { cj -= a.G[k]; s = -1.0; }
        else if (cj < 0) { cj += a.G[k]; s = 1.0; }
        const double xi = abs_coord(a, k, ci[k], full_offset(bi[k], oi[k]));
        const double xj = abs_coord(a, k, cj, full_offset(bj[k], oj[k]));
        e[k] = __dadd_rn(__dsub_rn(xi, xj), __dmul_rn(s, a.L[k]));
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(e[0], e[0]), __dmul_rn(e[1], e[1])), __dmul_rn(e[2], e[2])) < a.rn2;
}

// The list of the atom in cell-ordered slot s, by its four lanes (build_item's
// work dealt out).  The loop is bound by the latency of its loads and, with a
// warp or two per scheduler, of its instructions, so the lanes take a row's
// candidates in turn (the three cells of a row as one run), three rows at a
// time with all their loads first; a lane that took whole rows held up the
// others for 8 us more per rebuild.  Each lane stages its candidates, and the
// entries of all four are written out ordered by shell bin.  Returns the
// atom's entry count in every lane.  Every lane of the warp must call it (in =
// false: no atom).
// kRowsAhead: rows whose loads are issued together (fewer where registers are
// short: a spilled one costs a trip to L2 after each barrier).
template <class P, int kRowsAhead>
__device__ __forceinline__ int run_build(const Args<P>& a, int64_t s, bool in, int2* stage, int stride) {
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int kEach = 3;  // candidates of a row that a lane loads ahead: 12 per row
    const int lane = threadIdx.x & 31, sub = lane & (kRunLanes - 1), lead = lane - sub;
    Counters* C = a.ctr;
    int m = 0, i = 0;
    int* col = a.nbr;
    const int cap = a.cap;
    const int n = (int)a.n, self = (int)s;
    const float hi2 = a.rn2_hi;
    float4 ci = make_float4(0.f, 0.f, 0.f, 0.f);
    // rows sub, sub + 4, sub + 8: the run's slot of candidate t is t + at0 for
    // t < n0, t + at1 below n1, t + at2 below n2
    int n0[3] = {0, 0, 0}, n1[3] = {0, 0, 0}, n2[3] = {0, 0, 0}, at0[3], at1[3], at2[3];
    if (in) {
        ci = __ldcg(a.cand + s);
        i = __float_as_int(ci.w);
        int cx, cy, cz;
        unpack_cell(__ldcg(a.cell + i), cx, cy, cz);
        col += ((size_t)(i >> 5) * (size_t)cap) * 32 + (i & 31);
        const int xs[3] = {wrap_add(cx, -1, a.G[0]), cx, wrap_add(cx, 1, a.G[0])};
#pragma unroll
        for (int q = 0; q < 3; q++) {
            const int r = sub + kRunLanes * q;
            if (r < 9) {
                const PencilRow pr =
                    pencil_row(wrap_add(cy, r % 3 - 1, a.G[1]), wrap_add(cz, r / 3 - 1, a.G[2]), a.G);
                int lo[3], hi[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const int c = pr.base + xs[k] * pr.stride;
                    lo[k] = a.cell_start[c];
                    hi[k] = min(a.cell_start[c + 1], n);
                }
                n0[q] = hi[0] - lo[0];
                n1[q] = n0[q] + hi[1] - lo[1];
                n2[q] = n1[q] + hi[2] - lo[2];
                at0[q] = lo[0];
                at1[q] = lo[1] - n0[q];
                at2[q] = lo[2] - n1[q];
            }
        }
    }
    const float qx0 = ci.x + a.wf[0], qx1 = ci.x, qx2 = ci.x - a.wf[0];  // x seen from cells x-1, x, x+1
#pragma unroll
    for (int r0 = 0; r0 < 9; r0 += kRowsAhead) {
        int m0[kRowsAhead], m1[kRowsAhead], m2[kRowsAhead], s0[kRowsAhead], s1[kRowsAhead], s2[kRowsAhead];
        float4 pj[kRowsAhead][kEach];
#pragma unroll
        for (int w = 0; w < kRowsAhead; w++) {
            const int r = r0 + w, q = r / kRunLanes, from = lead + r % kRunLanes;
            m0[w] = __shfl_sync(kFull, n0[q], from);
            m1[w] = __shfl_sync(kFull, n1[q], from);
            m2[w] = __shfl_sync(kFull, n2[q], from);
            s0[w] = __shfl_sync(kFull, at0[q], from);
            s1[w] = __shfl_sync(kFull, at1[q], from);
            s2[w] = __shfl_sync(kFull, at2[q], from);
#pragma unroll
            for (int u = 0; u < kEach; u++) {
                const int t = sub + kRunLanes * u;
                if (t < m2[w]) pj[w][u] = a.cand[t + (t < m0[w] ? s0[w] : (t < m1[w] ? s1[w] : s2[w]))];
            }
        }
#pragma unroll
        for (int w = 0; w < kRowsAhead; w++) {
            const int r = r0 + w, dy = r % 3 - 1, dz = r / 3 - 1;
            const float qz = ci.z - (float)dz * a.wf[2];
            const float qy = ci.y - (float)dy * a.wf[1];
            const unsigned code_yz = ((unsigned)(dy + 1) << 2) | ((unsigned)(dz + 1) << 4);
            auto stage_one = [&](const float4& p, int t) {
                const int k = t < m0[w] ? 0 : (t < m1[w] ? 1 : 2);
                const int slot = t + (t < m0[w] ? s0[w] : (t < m1[w] ? s1[w] : s2[w]));
                const float ex = (t < m0[w] ? qx0 : (t < m1[w] ? qx1 : qx2)) - p.x;
                const float ey = qy - p.y, ez = qz - p.z;
                const float rr = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                const int code = (int)(((unsigned)k | code_yz) << kCodeShift);
                if (m < kRunStage) stage[m * stride] = make_int2(__float_as_int(p.w) | code, __float_as_int(rr));
                m += (rr < hi2 && slot != self) ? 1 : 0;
            };
#pragma unroll
            for (int u = 0; u < kEach; u++) {
                const int t = sub + kRunLanes * u;
                if (t < m2[w]) stage_one(pj[w][u], t);
            }
            for (int t = sub + kRunLanes * kEach; t < m2[w]; t += kRunLanes)  // a longer row
                stage_one(a.cand[t + (t < m0[w] ? s0[w] : (t < m1[w] ? s1[w] : s2[w]))], t);
        }
    }
    int total;
    const unsigned gm = ((1u << kRunLanes) - 1u) << (threadIdx.x & 31 & ~(kRunLanes - 1));
    const bool spill = (__ballot_sync(kFull, m > kRunStage) & gm) != 0u;
    if (spill) {  // rare: too long for the stage
        total = sub == 0 ? build_all<P, false>(a, s) : 0;
        total = __shfl_sync(gm, total, 0, kRunLanes);
        if (sub == 0) {
            a.nn[i] = min(total, cap);
            for (int k = 1; k < kShellBins; k++) a.lim[(size_t)(k - 1) * a.n + i] = 255;
        }
    } else {
        // as in build_item_t: FP64 test of the band entries, bins, and the
        // bin counts in the bytes of a 64-bit word -- here the lane's, then
        // those of the lanes below and of all four
        const float lo2 = a.rn2_lo;
        unsigned hlo = 0u, hhi = 0u;
        for (int t = 0; t < m; t++) {
            const int2 e = stage[t * stride];
            const float rr = __int_as_float(e.y);
            bool keep = true;
            if (!(rr < lo2)) keep = run_within_rn(a, i, e.x & kIndexMask, (unsigned)e.x >> kCodeShift);
            const int b = keep ? shell_bin(a, rr) : kShellBins;
            stage[t * stride].y = b;
            const unsigned inc = keep ? 1u << (8 * (b & 3)) : 0u;
            hlo += b < 4 ? inc : 0u;
            hhi += b < 4 ? 0u : inc;
        }
        const unsigned long long own = ((unsigned long long)hhi << 32) | hlo;
        unsigned long long upto = own;
#pragma unroll
        for (int o = 1; o < kRunLanes; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(gm, upto, o, kRunLanes);
            if (sub >= o) upto += y;
        }
        const unsigned long long all = __shfl_sync(gm, upto, kRunLanes - 1, kRunLanes);
        const unsigned long long incl = all * 0x0101010101010101ull;
        const unsigned long long first = (incl << 8) + (upto - own);  // the lane's first slot of each bin
        unsigned nlo = (unsigned)first, nhi = (unsigned)(first >> 32);
        for (int t = 0; t < m; t++) {
            const int2 e = stage[t * stride];
            const int b = e.y;
            if (b == kShellBins) continue;
            const int sh = 8 * (b & 3);
            const int dst = (int)(((b < 4 ? nlo : nhi) >> sh) & 0xffu);
            const unsigned inc = 1u << sh;
            nlo += b < 4 ? inc : 0u;
            nhi += b < 4 ? 0u : inc;
            if (dst < cap) col[(size_t)dst * 32] = e.x;
        }
        total = (int)(incl >> 56);
        if (in) {
            if (sub == 0) a.nn[i] = min(total, cap);
            for (int k = 1 + sub; k < kShellBins; k += kRunLanes)
                a.lim[(size_t)(k - 1) * a.n + i] = (unsigned char)(incl >> (8 * (k - 1)));
        }
    }
    if (in && sub == 0 && total > cap) {
        atomicOr(&C->error, kErrOverflow);
        atomicMax(&C->need_cap, total);
    }
    return in ? total : 0;
}

// The rebuild branch (k_bin .. k_rebuild_done) of the loop: seven barriers with
// a reorder, four without.  A cell's atoms keep their order of arrival unless
// the atoms are reordered: nothing in the mixed form depends on it.  Returns
// what its last barrier said.  (A function of its own, so that its
// registers do not weigh on the loop's.)
template <class P, int kB>
__device__ __noinline__ int run_rebuild(const Args<P>& a, int64_t i, int par, int reorder, RunBarrier bar, int2* stage,
                                             int* s_sync, int* s_scan) {
    constexpr unsigned kFull = 0xffffffffu;
    Counters* C = a.ctr;
    const int lane = threadIdx.x & 31, sub = lane & (kRunLanes - 1);
    const bool in = i < a.n;
    if (i == 0 && sub == 0) {
        C->max_occ = 0;
        C->max_nn = 0;
        C->list_entries = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x < kD2Buckets) a.d2b[threadIdx.x * 32] = 0u;  // displacements count from here
    int tile = -1;
    if (in && sub == 0) {
        const int c = bin_item<P>(a, i, par);
        count_item<P>(a, i, c);
        tile = c / kScanTile;
    }
    const unsigned peers = __match_any_sync(kFull, tile);
    if (tile >= 0 && lane == __ffs(peers) - 1) atomicAdd(&a.tile_sum[tile], __popc(peers));
    // (no block says anything before the last barrier: a stop is a wait that
    // ran out)
    int said = bar.sync(0, s_sync, C);
    if (said & kRunStop) return said;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) run_scan_tile(a, t, s_scan);
    said = bar.sync(0, s_sync, C);
    if (said & kRunStop) return said;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, dt = (int64_t)gridDim.x * blockDim.x;
    if (in && sub == 0) scatter_item<P>(a, i, reorder, par);
    for (int64_t c = t0; c < a.ncells; c += dt) a.count[c] = 0;
    for (int64_t c = t0; c < a.ntiles; c += dt) a.tile_sum[c] = 0;
    said = bar.sync(0, s_sync, C);
    if (said & kRunStop) return said;
    if (reorder) {
        for (int64_t c = t0; c < a.ncells; c += dt) cellsort_item<P>(a, c);
        said = bar.sync(0, s_sync, C);
        if (said & kRunStop) return said;
        if (in && sub == 0) gather_item<P>(a, i, reorder);
        said = bar.sync(0, s_sync, C);
        if (said & kRunStop) return said;
        if (in && sub == 0) commit_item<P>(a, i, par);
        said = bar.sync(0, s_sync, C);
        if (said & kRunStop) return said;
    }
    const int m = run_build<P, kB == kRunMaxBlock ? 1 : 3>(a, i, in, stage, (int)blockDim.x);
    const int wmax = __reduce_max_sync(kFull, m);
    const int wsum = __reduce_add_sync(kFull, sub == 0 ? m : 0);
    if (lane == 0) {
        atomicMax(&C->max_nn, wmax);
        atomicAdd((unsigned long long*)&C->list_entries, (unsigned long long)wsum);
    }
    // an error of the binning (recorded before an earlier barrier) or
    // of this thread's list stops the run, for all blocks alike
    return bar.sync(m > a.cap || __ldcg(&C->error) != 0 ? kRunStop : 0, s_sync, C);
}

// Up to `steps` plain steps (never a call's last one).  Cooperative launch of
// ceil(n kRunLanes / blockDim) blocks; words: the barrier's
// four and the gate's, zero.
// kB: the largest block that the instance serves (small systems have one
// block of 128 threads on an SM and need no register limit).
template <class P, int kB>
__global__ void __launch_bounds__(kB, kB == kRunMaxBlock ? 2 : 1) k_run(Args<P> a, long long steps, unsigned long long* words,
                                                                                  long long closed) {
    static_assert(!P::kFp64, "mixed form only");
    __shared__ int2 s_stage[kRunStage * kB];
    __shared__ int s_sync;
    __shared__ int s_scan[32];
    // for the functions that are not inlined: the address of a kernel
    // argument would put a copy of it in every thread's local memory
    __shared__ __align__(16) Args<P> sa;
    constexpr unsigned kFull = 0xffffffffu;
    Counters* C = a.ctr;
    RunBarrier bar{words, 0u};
    const int lane = threadIdx.x & 31, sub = lane & (kRunLanes - 1), lead = lane & ~(kRunLanes - 1);
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x / kRunLanes) + threadIdx.x / kRunLanes;
    const bool in = i < a.n;
    const bool mine = in && sub < 3;  // this lane integrates component `sub`
    // the counters, the same in every thread; block 0 writes them back
    const int err0 = C->error;
    int par = C->parity, pend = C->rebuild_flag, reorder = C->reorder_now;
    const int todo = (int)min(steps, C->steps_left - 1);  // (steps is at most kRunSteps)
    const int since0 = (int)min(C->since_reorder, (long long)INT_MAX / 2);
    int since = since0;  // steps since the last reorder
    float d2max = 0.0f;  // the largest squared displacement that this thread has seen since the last build
    if (err0 != 0 || todo <= 0) return;
    if (!run_gate(reinterpret_cast<unsigned*>(words + 4 * kRunWordStride), &s_sync, C, closed)) return;
    if (threadIdx.x == 0) sa = a;
    __syncthreads();
    int rebuilds = 0, reorders = 0;

    auto vp = [&]() { return sub == 0 ? a.vx : (sub == 1 ? a.vy : a.vz); };
    auto op = [&]() { return sub == 0 ? a.ox : (sub == 1 ? a.oy : a.oz); };
    float v = 0.0f, pb = 0.0f, p = 0.0f;
    double o = 0.0;
    int nn = 0;
    unsigned e[kRunRegs];  // entries sub, sub + 4, ...
    auto load = [&]() {
        if (in) nn = __ldcg(a.nn + i);
#pragma unroll
        for (int k = 0; k < kRunRegs; k++) {
            const int m = sub + kRunLanes * k;
            e[k] = m < nn ? (unsigned)__ldcg(a.nbr + list_base(a, i) + (size_t)m * 32) : 0u;
        }
        if (mine) {
            v = __ldcg(vp() + i);
            o = __ldcg(op() + i);
            pb = __ldcg((sub == 0 ? a.pbx : (sub == 1 ? a.pby : a.pbz)) + i);
            p = __ldcg(reinterpret_cast<const float*>((par ? a.pB : a.pA) + i) + sub);
        }
    };
    auto store = [&]() {
        if (mine) {
            vp()[i] = v;
            op()[i] = o;
        }
    };
    load();

    int done = 0;
    while (done < todo) {
        if (pend) {
            store();
            __syncwarp();
            const int said = run_rebuild<P, kB>(sa, i, par, reorder, bar, s_stage + threadIdx.x, &s_sync, s_scan);
            bar.epoch += reorder ? 7 : 4;
            rebuilds++;
            if (reorder) {
                reorders++;
                since = 0;
                reorder = 0;
            }
            pend = 0;
            d2max = 0.0f;
            load();
            if (said & kRunStop) break;
        }
        // one step: as step_atom, an atom's entries dealt out to its lanes
        const float4* pc = par ? a.pB : a.pA;
        float4* pn = par ? a.pA : a.pB;
        // (every entry is read: an atom's entries fill its lanes' registers in
        // one round whatever the shell reach, and the barrier need not carry
        // the largest displacement)
        float4 pj[kRunRegs];
#pragma unroll
        for (int k = 0; k < kRunRegs; k++)
            pj[k] = sub + kRunLanes * k < nn ? gather4<false>(pc + (e[k] & a.jmask)) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float qx = __shfl_sync(kFull, p, lead), qy = __shfl_sync(kFull, p, lead + 1),
                    qz = __shfl_sync(kFull, p, lead + 2);
        AccMixed acc;
#pragma unroll
        for (int k = 0; k < kRunRegs; k += 2)
            if (sub + kRunLanes * k < nn)
                mixed_pair2(a, qx, qy, qz, e[k], pj[k], e[k + 1], pj[k + 1], sub + kRunLanes * (k + 1) < nn, acc);
        for (int m = sub + kRunLanes * kRunRegs; m < nn; m += kRunLanes) {
            const unsigned x = (unsigned)__ldcg(a.nbr + list_base(a, i) + (size_t)m * 32);
            const float4 q = gather4<false>(pc + (x & a.jmask));
            mixed_pair2(a, qx, qy, qz, x, q, x, q, false, acc);
        }
        acc.settle();
        // the four lanes' exact partial sums
        auto total = [&](int x) {
#pragma unroll
            for (int w = 1; w < kRunLanes; w <<= 1) x += __shfl_xor_sync(kFull, x, w);
            return x;
        };
        Fix sum;  // lane d's component
        {
            const int bx = total(acc.fxy.x.b), by = total(acc.fxy.y.b), bz = total(acc.fz.b);
            const int cx = total(acc.fxy.x.c), cy = total(acc.fxy.y.c), cz = total(acc.fz.c);
            sum.b = sub == 0 ? bx : (sub == 1 ? by : bz);
            sum.c = sub == 0 ? cx : (sub == 1 ? cy : cz);
            if (__any_sync(kFull, (acc.fxy.x.a | acc.fxy.y.a | acc.fz.a) != 0)) {
                const int ax = total(acc.fxy.x.a), ay = total(acc.fxy.y.a), az = total(acc.fz.a);
                sum.a = sub == 0 ? ax : (sub == 1 ? ay : az);
            }
        }
        float disp = 0.0f;
        if (mine) {
            const float f = AccMixed::to_force(sum);
            v = kick(a, kick(a, v, f), f);
            o = drift(o, v, a.dt);
            disp = __double2float_rn(o);
            p = pb + disp;
            reinterpret_cast<float*>(pn + i)[sub] = p;
        }
        int say = 0;
        {
            const float dx = __shfl_sync(kFull, disp, lead), dy = __shfl_sync(kFull, disp, lead + 1),
                        dz = __shfl_sync(kFull, disp, lead + 2);
            const float d2 = dx * dx + dy * dy + dz * dz;
            d2max = d2 > d2max ? d2 : d2max;
            if (!(d2 < a.thr2f)) say = kRunFar;  // (a NaN asks for the rebuild, which reports it)
            if (acc.close) {
                atomicOr(&C->error, kErrClose);
                say |= kRunStop;
            }
        }
        const int said = bar.sync(say, &s_sync, C);
        par ^= 1;
        done++;
        since++;
        if (said & kRunStop) break;
        pend = (said & kRunFar) != 0;
        reorder = pend && a.reorder_interval > 0 && since >= a.reorder_interval;
    }
    store();
    // the running maximum of the displacements, for the step kernels
    warp_max_into(d2_bits(d2max), d2_word(a));
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // (no block reads the counters any more)
        C->parity = par;
        C->rebuild_flag = pend;
        C->reorder_now = reorder;
        C->steps_left -= done;
        C->step += done;
        C->run_steps += done;
        C->since_reorder = reorders > 0 ? since : C->since_reorder + done;
        C->rebuilds += rebuilds;
        C->run_rebuilds += rebuilds;
        C->reorders += reorders;
        C->far_flag = 0u;
        C->reach = kShellBins;  // the next step reads every entry; its closing kernel sets the reach again
    }
}

// Up to `steps` plain steps of the cell-list-only variant, kCellLanes lanes
// per atom in the force phase.  The phases of a step are the kernels of the
// graph, a grid barrier between them, with the same operations in the same
// order, so the results are the same bits.  Cooperative launch of
// ceil(n kCellLanes / kRunCellBlock) blocks.
template <class P>
__global__ void __launch_bounds__(kRunCellBlock, 5) k_run_cells(Args<P> a, long long steps, unsigned long long* words,
                                                             long long closed) {
    using real = typename P::real;
    __shared__ int s_queue[P::kFp64 ? kRunCellBlock / kCellLanes * kCellQueue : 1];
    __shared__ int s_sync;
    __shared__ int s_scan[32];
    Counters* C = a.ctr;
    RunBarrier bar{words, 0u};
    const int sub = threadIdx.x % kCellLanes;
    const int64_t slot = ((int64_t)blockIdx.x * kRunCellBlock + threadIdx.x) / kCellLanes;
    const int64_t t0 = (int64_t)blockIdx.x * kRunCellBlock + threadIdx.x, dt = (int64_t)gridDim.x * kRunCellBlock;
    int* queue = s_queue + (P::kFp64 ? (int)(threadIdx.x / kCellLanes) * kCellQueue : 0);
    const int err0 = C->error;
    int par = C->parity, reorder = C->reorder_now;
    const int todo = (int)min(steps, C->steps_left - 1);  // (steps is at most kRunSteps)
    int since = (int)min(C->since_reorder, (long long)INT_MAX / 2);
    if (err0 != 0 || todo <= 0) return;
    if (!run_gate(reinterpret_cast<unsigned*>(words + 4 * kRunWordStride), &s_sync, C, closed)) return;
    int reorders = 0, done = 0, stop = 0;
    while (done < todo && !stop) {
        // the rebuild (k_bin .. k_rebuild_done); the grid has a thread for
        // every atom several times over: the first n of them take one each
        if (t0 == 0) C->max_occ = 0;
        int tile = -1;
        if (t0 < a.n) {
            const int c = bin_item<P>(a, t0, par);
            count_item<P>(a, t0, c);
            tile = c / kScanTile;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, tile);
        if (tile >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&a.tile_sum[tile], __popc(peers));
        // (no block says anything before a step's last barrier: a stop is a
        // wait that ran out)
        if (bar.sync(0, &s_sync, C) & kRunStop) break;
        for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) run_scan_tile(a, t, s_scan);
        if (bar.sync(0, &s_sync, C) & kRunStop) break;
        if (t0 < a.n) scatter_item<P>(a, t0, reorder, par);
        for (int64_t c = t0; c < a.ncells; c += dt) a.count[c] = 0;
        for (int64_t c = t0; c < a.ntiles; c += dt) a.tile_sum[c] = 0;
        if (bar.sync(0, &s_sync, C) & kRunStop) break;
        if (sorts_cells<P>(reorder)) {
            for (int64_t c = t0; c < a.ncells; c += dt) {
                cellsort_item<P>(a, c);
                const int end = min(a.cell_start[c + 1], (int)a.n);
                for (int s = a.cell_start[c]; s < end; s++) gather_item<P>(a, s, reorder);
            }
            if (bar.sync(0, &s_sync, C) & kRunStop) break;
            if (reorder) {
                if (t0 < a.n) commit_item<P>(a, t0, par);
                if (bar.sync(0, &s_sync, C) & kRunStop) break;
                reorders++;
                since = 0;
            }
        }
        // forces, and the step's update of one component in each of three lanes
        const typename P::pos4* pc = par ? a.pB : a.pA;
        typename P::pos4* pn = par ? a.pA : a.pB;
        typename AccOf<P>::type acc;
        const bool in = slot < a.n;
        const int i = cell_forces_item<P, false>(a, slot, in, pc, queue, acc);
        if (in && sub < 3) {
            typename P::vel* vp = sub == 0 ? a.vx : (sub == 1 ? a.vy : a.vz);
            double* op = sub == 0 ? a.ox : (sub == 1 ? a.oy : a.oz);
            const real f = sub == 0 ? acc.force_x() : (sub == 1 ? acc.force_y() : acc.force_z());
            const real pb = (sub == 0 ? a.pbx : (sub == 1 ? a.pby : a.pbz))[i];
            const typename P::vel v = kick(a, kick(a, vp[i], f), f);
            const double o = drift(op[i], v, a.dt);
            real p;
            moved<true>(pb, o, p);
            vp[i] = v;
            op[i] = o;
            reinterpret_cast<real*>(pn + i)[sub] = p;
        }
        if (in && acc.close) atomicOr(&C->error, kErrClose);
        stop = bar.sync((in && acc.close) || __ldcg(&C->error) != 0 ? kRunStop : 0, &s_sync, C) & kRunStop;
        par ^= 1;
        done++;
        since++;
        reorder = a.reorder_interval > 0 && since >= a.reorder_interval;
    }
    if (t0 == 0) {  // (no block reads the counters any more)
        C->parity = par;
        C->rebuild_flag = 1;  // as after every step of this variant
        C->reorder_now = reorder;
        C->steps_left -= done;
        C->step += done;
        C->run_steps += done;
        C->since_reorder = reorders > 0 ? since : C->since_reorder + done;
        C->rebuilds += done;
        C->run_rebuilds += done;
        C->reorders += reorders;
        C->far_flag = 0u;
        C->max_nn = 0;
        C->list_entries = 0;
    }
}

}  // namespace md
