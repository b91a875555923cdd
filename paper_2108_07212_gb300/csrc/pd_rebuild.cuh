// pd_rebuild.cuh -- grid barriers of the cooperative kernels, and the rebuild of
// the contact candidate lists between such barriers.
#pragma once

#include "pd_device.cuh"

namespace pd {

// Grid barriers with a bounded wait.  Co-residency of all blocks is guaranteed
// by the cooperative launch.  A wait polls at most max_spins times
// (kBarrierSpins unless a test shortens it), then sets
// status[PD_STATUS_TIMEOUT] and reports failure (the kernel then returns, so
// the device never hangs); the others see the status at a later poll.
//
// The first barrier of a launch: the last block to arrive resets the arrival
// count and advances the generation that the others poll, so nothing depends
// on what an earlier launch (with another grid, or given up) left behind.
__device__ __forceinline__ bool grid_barrier_first(const DevPtrs &d, long long max_spins) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *gen = d.bar + 1;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(d.bar, 1u);
        ok = 1;
        if (arrived == gridDim.x - 1) {
            atomicExch(d.bar, 0u);
            __threadfence();
            atomicAdd(d.bar + 1, 1u);
        } else {
            long long n = 0;
            while (*gen == g) {
                if (++n > max_spins || *(volatile int *)&d.status[PD_STATUS_TIMEOUT]) {
                    atomicExch(&d.status[PD_STATUS_TIMEOUT], 1);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// The later ones: a release-increment of a counter that block 0 cleared before
// the launch's first barrier, and an acquire-poll until all arrivals of this
// barrier (the epoch-th) are in: one trip to L2 and back after the last
// arrival, where the reset and the generation above take two more.  (3.5 us a
// barrier with the latter on 304 blocks.)
__device__ __forceinline__ bool grid_barrier(const DevPtrs &d, long long max_spins, unsigned &epoch) {
    __shared__ int ok;
    ++epoch;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned *const count = d.bar + 2;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        const unsigned target = epoch * gridDim.x;
        ok = 1;
        for (long long n = 1;; ++n) {
            unsigned c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
            if ((int)(c - target) >= 0) break;
            if (n > max_spins || ((n & 63) == 0 && *(volatile int *)&d.status[PD_STATUS_TIMEOUT])) {
                atomicExch(&d.status[PD_STATUS_TIMEOUT], 1);
                ok = 0;
                break;
            }
            __nanosleep(20);
        }
    }
    __syncthreads();
    return ok != 0;
}

template <int BLOCK>
__device__ __forceinline__ int block_sum(int v, int *sm) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    int t = 0;
    if (threadIdx.x < 32) {
        t = (lane < BLOCK / 32) ? sm[lane] : 0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0) sm[32] = t;
    }
    __syncthreads();
    return sm[32];
}

// Exclusive scan of one value per thread over the block; returns the total.
template <int BLOCK>
__device__ __forceinline__ int block_scan1(int &v, int *sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    __syncthreads();
    if (lane == 31) sm[warp] = incl;
    __syncthreads();
    if (threadIdx.x < 32) {
        int w = (lane < BLOCK / 32) ? sm[lane] : 0;
        int wi = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += y;
        }
        sm[lane] = wi - w;
        if (lane == 31) sm[32] = wi;
    }
    __syncthreads();
    v = sm[warp] + incl - v;
    return sm[32];
}

// Rebuild of the candidate lists at the current positions by nblk co-resident
// blocks (this one: blk), which `barrier` (false: it gave up) brings together:
//   R1 cell counts
//   R2 per-block sums of the cell counts
//   R3 exclusive scan of the counts -> cell starts (counts cleared)
//   R4 counting-sort scatter of the node indices
//   R5 candidate lists
// Cell counts are zero on entry and on exit.  False when a barrier gave up.
template <bool PERSIST, int BLOCK, class Barrier>
__device__ __forceinline__ bool rebuild_lists(const DevPtrs &d, const KParams &k, int blk, int nblk, int *sm,
                                              Barrier barrier) {
    const int nthreads = nblk * BLOCK;
    const int gtid = blk * BLOCK + threadIdx.x;
    const unsigned T = k.T;
    const unsigned slice = (T / 4 + (unsigned)nblk - 1) / (unsigned)nblk * 4;
    const unsigned lo = min(T, (unsigned)blk * slice), hi = min(T, lo + slice);
    // R1
    for (int i = gtid; i < k.N; i += kBinBatch * nthreads) bin_nodes<PERSIST>(d, k, i, nthreads);
    if (!barrier()) return false;
    // R2 (four cells a load; T is a multiple of 4)
    int part = 0;
    for (unsigned b = lo + 4 * threadIdx.x; b < hi; b += 4 * BLOCK) {
        const int4 c = __ldcg(reinterpret_cast<const int4 *>(&d.count[b]));
        part += (c.x + c.y) + (c.z + c.w);
    }
    part = block_sum<BLOCK>(part, sm);
    if (threadIdx.x == 0) d.blocksums[(unsigned)blk] = part;
    if (!barrier()) return false;
    // R3 (kScan4 loads of four cells a thread and round)
    constexpr unsigned kScan4 = 4;
    int off = 0;
    for (int b = threadIdx.x; b < blk; b += BLOCK) off += __ldcg(&d.blocksums[b]);
    off = block_sum<BLOCK>(off, sm);
    for (unsigned b0 = lo; b0 < hi; b0 += 4 * kScan4 * BLOCK) {
        const unsigned b = b0 + 4 * kScan4 * threadIdx.x;
        int4 c[kScan4];
        int at = 0;
#pragma unroll
        for (unsigned q = 0; q < kScan4; ++q)
            c[q] = b + 4 * q < hi ? __ldcg(reinterpret_cast<const int4 *>(&d.count[b + 4 * q])) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (unsigned q = 0; q < kScan4; ++q) at += (c[q].x + c[q].y) + (c[q].z + c[q].w);
        const int tot = block_scan1<BLOCK>(at, sm);
        at += off;
#pragma unroll
        for (unsigned q = 0; q < kScan4; ++q) {
            if (b + 4 * q >= hi) break;
            *reinterpret_cast<int4 *>(&d.count[b + 4 * q]) = make_int4(0, 0, 0, 0);
            *reinterpret_cast<int4 *>(&d.start[b + 4 * q]) =
                make_int4(at, at + c[q].x, at + c[q].x + c[q].y, at + c[q].x + c[q].y + c[q].z);
            at += (c[q].x + c[q].y) + (c[q].z + c[q].w);
        }
        off += tot;
    }
    if (gtid == 0) d.start[T] = k.N;
    if (!barrier()) return false;
    // R4
    for (int i = gtid; i < k.N; i += kBinBatch * nthreads) scatter_nodes<PERSIST>(d, k, i, nthreads);
    if (!barrier()) return false;
    // R5 (every block has read the flag: clear it for the next step)
    if (gtid == 0) {
        *d.rebuild = 0;
        atomicAdd(&d.status[PD_STATUS_REBUILDS], 1);
    }
    for (int i = gtid; i < k.N; i += nthreads) build_list_node<PERSIST>(d, k, i);
    if (!barrier()) return false;
    return true;
}

}  // namespace pd
