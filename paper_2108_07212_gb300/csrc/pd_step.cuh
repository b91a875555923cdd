// pd_step.cuh -- force kernels of the multi-kernel path and the persistent
// step kernel, instantiated per precision by pd_step64.cu (no FMA
// contraction) and pd_step32.cu.
#pragma once

#include <type_traits>

#include "pd_rebuild.cuh"

namespace pd {

// Forces and update of nodes [node0, node0 + BLOCK / LANES): LANES threads per
// node compute the lane-summed bond / self-contact / contact parts, which meet
// in shared memory; then one thread per node adds the wall forces and
// integrates (FP64, converged warps).  Every thread of the block must call it.
template <bool FP32, bool PERSIST, int LANES, int BLOCK>
__device__ __forceinline__ void force_block(const DevPtrs &d, const KParams &k, int node0, int vin, int update_v) {
    constexpr int NB = BLOCK / LANES;
    using Sums = typename std::conditional<FP32, Sums32, Sums64>::type;
    __shared__ Sums sm[NB];
    const int local = threadIdx.x / LANES, lane = threadIdx.x % LANES;
    const int i = node0 + local;
    Sums f;
    [[maybe_unused]] bool contact;
    if constexpr (FP32) force_node32<PERSIST, LANES>(d, k, i, lane, i < k.N, vin, f);
    else force_node64<PERSIST, LANES, 0>(d, k, i, lane, i < k.N, vin, f, nullptr, false, contact);
    if (lane == 0) sm[local] = f;
    __syncthreads();
    if ((int)threadIdx.x < NB && node0 + (int)threadIdx.x < k.N) {
        if constexpr (FP32)
            node_epilogue32<PERSIST>(d, k, node0 + threadIdx.x, __ldg(&d.grain[node0 + threadIdx.x]), vin, update_v,
                                     sm[threadIdx.x], load_update32<PERSIST>(d, node0 + threadIdx.x, vin, update_v));
        else node_epilogue64<PERSIST>(d, k, node0 + threadIdx.x, vin, update_v, sm[threadIdx.x]);
    }
    __syncthreads();
}

// The force phase reads the candidate lists of this step: it clears the
// rebuild flag for the next one.
__device__ __forceinline__ void clear_rebuild(const DevPtrs &d) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *d.rebuild = 0;
}

// The lane sums of node i into global memory (split force phase; structure of
// arrays): six components with per-part output, else only their total (F_b +
// F_s) + F_n, as the epilogue would form it.
template <bool FP32, class Sums>
__device__ __forceinline__ void store_sums(const DevPtrs &d, const KParams &k, int i, const Sums &f) {
    const size_t N = (size_t)k.N;
    using T = typename std::conditional<FP32, float, double>::type;
    T *o = static_cast<T *>(d.fsum);
    if (k.store) {
        o[i] = f.bx, o[N + i] = f.by, o[2 * N + i] = f.sx, o[3 * N + i] = f.sy, o[4 * N + i] = f.nx, o[5 * N + i] = f.ny;
    } else if constexpr (FP32) {
        reinterpret_cast<float2 *>(o)[i] = make_float2((f.bx + f.sx) + f.nx, (f.by + f.sy) + f.ny);
    } else {
        reinterpret_cast<double2 *>(o)[i] =
            make_double2(__dadd_rn(__dadd_rn(f.bx, f.sx), f.nx), __dadd_rn(__dadd_rn(f.by, f.sy), f.ny));
    }
}

extern __shared__ __align__(16) unsigned char tile_smem[];

// One thread per node, FP64 path: the nodes [lo, hi) in bond tiles of BLOCK
// nodes (see PairTile), or without TILES as many by themselves.  All threads
// call out(i, sums, active, contact) as tile_nodes32 does.  Every thread of the
// block calls it with the same range.
template <bool PERSIST, int BLOCK, bool TILES, bool INLINE, class Out>
__device__ __forceinline__ void run_nodes64(const DevPtrs &d, const KParams &k, int lo, int hi, int vin, Out out) {
    [[maybe_unused]] float4 *slot = reinterpret_cast<float4 *>(tile_smem);
    // the pass before the run takes the nodes [lo - BLOCK, lo), of which the last kCarry have slots
    for (int node0 = TILES && lo > 0 && lo < hi ? lo - BLOCK : lo; node0 < hi; node0 += BLOCK) {
        const int i = node0 + (int)threadIdx.x;
        const bool warm = node0 < lo;
        const bool active = warm ? i >= max(0, lo - kCarry) : i < hi;
        Sums64 f;
        bool contact;
        force_node64<PERSIST, 1, TILES ? BLOCK : 0, INLINE>(d, k, i, 0, active, vin, f, slot, warm, contact);
        if (!warm) out(i, f, active, contact);
        if constexpr (TILES) {
            __syncthreads();               // the tile's slots have been read (or formed)
            PairTile<float4, BLOCK>::carry(slot);
            __syncthreads();
        }
    }
}

// The forces of the nodes [lo, hi) in bond tiles, one thread per node, by the
// calling block: sums stored (split force phase), or each node's walls and
// update behind them.
template <bool FP32, bool PERSIST, int BLOCK>
__device__ __forceinline__ void run_tiles(const DevPtrs &d, const KParams &k, int lo, int hi, int vin, int update_v,
                                          bool fused) {
    if constexpr (FP32) {
        auto out = [&](int i, const Sums32 &f, int, bool active, bool) {
            if (!active) return;
            if (fused) node_epilogue32<PERSIST>(d, k, i, __ldg(&d.grain[i]), vin, update_v, f,
                                                load_update32<PERSIST>(d, i, vin, update_v));
            else store_sums<true>(d, k, i, f);
        };
        tile_nodes32<PERSIST, BLOCK, true>(d, k, lo, hi, vin, false, *reinterpret_cast<Tile32<BLOCK> *>(tile_smem), out);
    } else {
        run_nodes64<PERSIST, BLOCK, true, true>(d, k, lo, hi, vin, [&](int i, const Sums64 &f, bool active, bool) {
            if (!active) return;
            if (fused) node_epilogue64<PERSIST>(d, k, i, vin, update_v, f);
            else store_sums<false>(d, k, i, f);
        });
    }
}

// The same for the persistent kernel's fused force phase: plain nodes are
// updated at once, special ones (see list_special) put on list `which`.
template <bool FP32, int BLOCK, bool TILES>
__device__ __forceinline__ void run_plain_nodes(const DevPtrs &d, const KParams &k, int lo, int hi, int vin, int which) {
    static_assert(TILES || !FP32, "FP32 split without tiles: no list of special nodes");
    if constexpr (FP32) {
        Tile32<BLOCK> &sm = *reinterpret_cast<Tile32<BLOCK> *>(tile_smem);
        tile_nodes32<true, BLOCK, false>(d, k, lo, hi, vin, true, sm,
                                         [&](int i, const Sums32 &f, int at, bool active, bool contact) {
            bool special = false;
            if (active) {
                const Update32 n{sm.v[at], sm.u[at], sm.xs[at], sm.sref[at], sm.a[at], sm.cell[at]};
                const int gi = __ldg(&d.grain[i]);
                special = contact || k.store || !cells_far_from_walls(n.cell, ldm<true>(&cur_wall<true>(d)[__ldg(&d.g_agg[gi])]));
                if (special) reinterpret_cast<float2 *>(d.fsum)[i] = make_float2(f.bx, f.by);
                else finish_node32_total<true>(d, k, i, vin, 1, n, f.bx, f.by, false, 0.0, 0.0, __ldg(&d.g_invmf[gi]));
            }
            list_special(d, which, i, special);
        });
    } else {
        run_nodes64<true, BLOCK, TILES, false>(d, k, lo, hi, vin, [&](int i, const Sums64 &f, bool active, bool contact) {
            bool special = false;
            if (active) {
                const int gi = __ldg(&d.grain[i]);
                const double2 v = ldm<true>(&d.v[vin][i]), a = ldm<true>(&d.a[i]);
                special = contact || k.store ||
                          !cells_far_from_walls(ldm<true>(&d.cell[i]), ldm<true>(&cur_wall<true>(d)[__ldg(&d.g_agg[gi])]));
                if (special) reinterpret_cast<double2 *>(d.fsum)[i] = make_double2(f.bx, f.by);
                else finish_node64_total<true>(d, k, i, vin, 1, v, a, f.bx, f.by, false, 0.0, 0.0, __ldg(&d.g_invm[gi]));
            }
            list_special(d, which, i, special);
        });
    }
}

// The special nodes of list `which`, dealt to the warps of all blocks in turn
// (one each before any takes a second into its other groups of threads).
template <bool FP32, int BLOCK>
__device__ __forceinline__ void run_special_nodes(const DevPtrs &d, const KParams &k, int vin, int which) {
    const int n = __ldcg(&d.spec_n[which]);
    constexpr int kGroups = 32 / kSpecialLanes;
    const int warps = gridDim.x * (BLOCK / 32), warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int group = (threadIdx.x & 31) / kSpecialLanes;
    for (int g = 0; g + warp < n; g += warps * kGroups) {
        const int q = g + group * warps + warp;
        const bool node = q < n;
        const int i = node ? __ldcg(&d.spec[q]) : 0;
        if constexpr (FP32) special_node32<true>(d, k, i, node, vin);
        else special_node64<true>(d, k, i, node, vin);
    }
}
template <bool FP32, int BLOCK>
constexpr int run_smem() {
    return FP32 ? (int)sizeof(Tile32<BLOCK>) : PairTile<float4, BLOCK>::kBytes;
}
// Blocks of BLOCK threads per SM of the kernels with tiles: 512 threads of up to
// 128 registers.  (FP32 split: three blocks of 256 at 80 registers spilled in
// the tile loop, 211 us against 183 us on 2.28M nodes.)
constexpr int run_blocks(int block) { return 512 / block; }

// Multi-kernel path, bond tiles: k.run nodes a block (see kRunNodes).
template <bool FP32>
__global__ void __launch_bounds__(kRunBlock, run_blocks(kRunBlock))
    k_force_run(DevPtrs d, KParams k, int vin, int update_v, int fused) {
    clear_rebuild(d);
    const int lo = blockIdx.x * k.run;
    run_tiles<FP32, false, kRunBlock>(d, k, lo, min(lo + k.run, k.N), vin, update_v, fused != 0);
}

// Multi-kernel path without tiles: one block per BLOCK / LANES nodes.
template <bool FP32, int LANES>
__global__ void __launch_bounds__(kBlock, FP32 ? (LANES == 1 ? 8 : 5) : 4) k_force(DevPtrs d, KParams k, int vin, int update_v) {
    clear_rebuild(d);
    force_block<FP32, false, LANES, kBlock>(d, k, blockIdx.x * (kBlock / LANES), vin, update_v);
}

// Split variant: the lane sums of node i go to global memory and a second pass
// adds walls and integrates.
template <bool FP32, bool PERSIST, int LANES>
__device__ __forceinline__ void sums_node(const DevPtrs &d, const KParams &k, int i, int lane, int vin) {
    const bool active = i < k.N;
    typename std::conditional<FP32, Sums32, Sums64>::type f;
    [[maybe_unused]] bool contact;
    if constexpr (FP32) force_node32<PERSIST, LANES>(d, k, i, lane, active, vin, f);
    else force_node64<PERSIST, LANES, 0>(d, k, i, lane, active, vin, f, nullptr, false, contact);
    if (active && lane == 0) store_sums<FP32>(d, k, i, f);
}

template <bool FP32, bool PERSIST>
__device__ __forceinline__ void epilogue_node(const DevPtrs &d, const KParams &k, int i, int vin, int update_v) {
    const size_t N = (size_t)k.N;
    // per-part sums (k.store) or the total of the parts
    if constexpr (FP32) {
        const float *o = static_cast<const float *>(d.fsum);
        const Update32 n = load_update32<PERSIST>(d, i, vin, update_v);
        if (k.store) {
            const Sums32 f{ldm<PERSIST>(o + i), ldm<PERSIST>(o + N + i), ldm<PERSIST>(o + 2 * N + i),
                           ldm<PERSIST>(o + 3 * N + i), ldm<PERSIST>(o + 4 * N + i), ldm<PERSIST>(o + 5 * N + i)};
            node_epilogue32<PERSIST>(d, k, i, __ldg(&d.grain[i]), vin, update_v, f, n);
        } else {
            const float2 t = ldm<PERSIST>(reinterpret_cast<const float2 *>(o) + i);
            node_epilogue32<PERSIST>(d, k, i, __ldg(&d.grain[i]), vin, update_v,
                                     Sums32{t.x, t.y, 0.f, 0.f, 0.f, 0.f}, n, true);
        }
    } else {
        const double *o = static_cast<const double *>(d.fsum);
        if (k.store) {
            const Sums64 f{ldm<PERSIST>(o + i), ldm<PERSIST>(o + N + i), ldm<PERSIST>(o + 2 * N + i),
                           ldm<PERSIST>(o + 3 * N + i), ldm<PERSIST>(o + 4 * N + i), ldm<PERSIST>(o + 5 * N + i)};
            node_epilogue64<PERSIST>(d, k, i, vin, update_v, f);
        } else {
            const double2 t = ldm<PERSIST>(reinterpret_cast<const double2 *>(o) + i);
            node_epilogue64<PERSIST>(d, k, i, vin, update_v, Sums64{t.x, t.y, 0.0, 0.0, 0.0, 0.0}, true);
        }
    }
}

template <bool FP32, int LANES>
__global__ void __launch_bounds__(kBlock, FP32 ? 8 : 4) k_sums(DevPtrs d, KParams k, int vin) {
    clear_rebuild(d);
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    sums_node<FP32, false, LANES>(d, k, tid / LANES, tid % LANES, vin);
}

// (Registers for the wall terms: at 40 a thread their chain went through 1.3 to
// 1.5 KB of spills; a step near the walls, 49907 nodes FP32 split: 12 us.)
// (kManyNodes, FP32 split: with ten waves of blocks the pass is bound by memory,
// and the warps that 40 registers allow are worth more.  Step with 80 and with 40:
// 2.04M nodes, two threads each, 251 and 239 us, on the surrogate 232 and 207;
// 1.24M 159 and 155, 801k 109 and 107, 521k 74 and 75.)
constexpr int kManyNodes = 1 << 20;
template <bool FP32, int PERSM = FP32 ? 3 : 2>
__global__ void __launch_bounds__(256, PERSM) k_epilogue(DevPtrs d, KParams k, int vin, int update_v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < k.N) epilogue_node<FP32, false>(d, k, i, vin, update_v);
}

template <bool FP32>
cudaError_t launch_force_run(const DevPtrs &d, const KParams &k, int vin, int update_v, cudaStream_t s, int fused) {
    k_force_run<FP32><<<(k.N + k.run - 1) / k.run, kRunBlock, run_smem<FP32, kRunBlock>(), s>>>(d, k, vin,
                                                                                                     update_v, fused);
    return cudaGetLastError();
}
template <bool FP32>
cudaError_t init_force_run() {
    return cudaFuncSetAttribute(k_force_run<FP32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                run_smem<FP32, kRunBlock>());
}

// phase (split force phase only): 0 both passes, 1 the lane sums, 2 the epilogue.
template <bool FP32>
cudaError_t launch_force_impl(const DevPtrs &d, const KParams &k, int vin, int update_v, cudaStream_t s, int phase) {
    const long long threads = (long long)k.lanes * k.N;
    const unsigned grid = (unsigned)((threads + kBlock - 1) / kBlock);
    if (k.split) {
        if (phase != 2) {
            if (k.lanes == 8) k_sums<FP32, 8><<<grid, kBlock, 0, s>>>(d, k, vin);
            else if (k.lanes == 4) k_sums<FP32, 4><<<grid, kBlock, 0, s>>>(d, k, vin);
            else if (k.lanes == 2) k_sums<FP32, 2><<<grid, kBlock, 0, s>>>(d, k, vin);
            else if (!k.pair || (FP32 && k.sur))
                // (grains on the surrogate have no bonds to share: more warps instead of
                // tiles; 2000 grains, 2.03M nodes: 232 us a step, in tiles 250)
                k_sums<FP32, 1><<<grid, kBlock, 0, s>>>(d, k, vin);
            else if (const cudaError_t e = launch_force_run<FP32>(d, k, vin, 0, s, 0)) return e;
        }
        const unsigned nb = (unsigned)((k.N + 255) / 256);
        if (phase == 1) return cudaGetLastError();
        if constexpr (FP32) {
            if (k.N > kManyNodes) {
                k_epilogue<FP32, 6><<<nb, 256, 0, s>>>(d, k, vin, update_v);
                return cudaGetLastError();
            }
        }
        k_epilogue<FP32><<<nb, 256, 0, s>>>(d, k, vin, update_v);
        return cudaGetLastError();
    }
    if (phase != 0) return cudaErrorInvalidValue;
    if (k.lanes == 8) k_force<FP32, 8><<<grid, kBlock, 0, s>>>(d, k, vin, update_v);
    else if (k.lanes == 4) k_force<FP32, 4><<<grid, kBlock, 0, s>>>(d, k, vin, update_v);
    else if (k.lanes == 2) k_force<FP32, 2><<<grid, kBlock, 0, s>>>(d, k, vin, update_v);
    else if (!k.pair) k_force<FP32, 1><<<grid, kBlock, 0, s>>>(d, k, vin, update_v);
    else return launch_force_run<FP32>(d, k, vin, update_v, s, 1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// persistent step kernel

// One time step of the persistent kernel, all phases:
//   A  displacement update, positions, rebuild test       (Algorithm 1)
//      (FP32 split: taken by the previous step's velocity update instead,
//      except in the first step of a launch that finds no valid prediction)
//   R  the candidate lists, when some node moved kSkinTrigger * skin since the
//      last rebuild (rebuild_lists)
//   E  forces, acceleration and velocity update (bond tiles, and in FP64 one
//      thread per node, with the fused force phase: plain nodes, then special ones)
// The barrier after A is left out where A was taken by the step before (FP32
// split, after the first step): what it published is then known already.
//   * The time of the step follows from the step counter at the launch.
//   * The wall cells of step st lie in half st & 1 of wall_cell, written during
//     the step before.
//   * The rebuild flag of step st is word st % 3 of rebuild3, raised by the
//     velocity updates of step st - 1 and cleared during step st - 2 (every
//     block has read the word in step st - 3, and none raises it before
//     st - 1).
// s_cur_* hold this step's displacement, positions, time, wall cells and the
// word its rebuild test raises.  False when a grid barrier gave up (the kernel then returns).
template <bool FP32, int LANES, int BLOCK, bool TILES>
__device__ __forceinline__ bool persistent_step(const DevPtrs &d, const KParams &k, int vin, int st, int nsteps,
                                                bool predicted, long long step0, unsigned &epoch, int *sm) {
    const int nthreads = gridDim.x * BLOCK;
    const int gtid = blockIdx.x * BLOCK + threadIdx.x;
    const bool known = FP32 && st > 0;
    if (!known) {
        // A
        if (st == 0) prefetch_force_inputs(d, k, gtid, nthreads);
        if (!predicted) {
            bool need = false;
            for (int i = gtid; i < k.N; i += nthreads) need |= predict_node<true>(d, k, i, vin, 1);
            if (__any_sync(0xffffffffu, need) && (threadIdx.x & 31) == 0) *(volatile int *)d.rebuild = 1;
        }
        if (blockIdx.x == 0) {
            if (st == 0 && threadIdx.x == 0) {
                d.bar[2] = 0u;
                d.spec_n[0] = d.spec_n[1] = 0;
                if constexpr (FP32) {
                    // the last launch's rebuild test becomes this step's flag (no
                    // block reads the flag before the barrier below)
                    if (predicted && *(volatile int *)d.rebuild_next) *(volatile int *)d.rebuild = 1;
                    *(volatile int *)d.rebuild_next = 0;
                    d.rebuild3[0] = d.rebuild3[1] = d.rebuild3[2] = 0;
                }
            }
            wall_cells(d, k, (double)(step0 + st + 1) * k.dt, d.wall_cell + (st & 1) * k.n_agg);
        }
        if (st == 0 ? !grid_barrier_first(d, k.bar_spins) : !grid_barrier(d, k.bar_spins, epoch)) return false;
    }
    const bool rebuild = __ldcg(known ? &d.rebuild3[st % 3] : d.rebuild) != 0;
    if (gtid == 0) {
        if (FP32) d.rebuild3[(st + 2) % 3] = 0;
        if (st + 1 == nsteps) {
            *d.step = step0 + nsteps;
            *d.t_now = (double)(step0 + nsteps) * k.dt;
        }
    }
    // the next step's wall cells, by the block with the shortest run of nodes
    if (FP32 && st + 1 < nsteps && blockIdx.x == gridDim.x - 1)
        wall_cells(d, k, (double)(step0 + st + 2) * k.dt, d.wall_cell + ((st + 1) & 1) * k.n_agg);
    if (rebuild && !rebuild_lists<true, BLOCK>(d, k, blockIdx.x, gridDim.x, sm,
                                               [&] { return grid_barrier(d, k.bar_spins, epoch); }))
        return false;
    // E
    const int len = run_length(k.N, gridDim.x);
    const int lo0 = (int)min((long long)k.N, (long long)blockIdx.x * len), hi0 = min(lo0 + len, k.N);
    if (k.split) {
        if constexpr (TILES) {
            run_tiles<FP32, true, BLOCK>(d, k, lo0, hi0, vin, 1, false);
        } else {
            const long long total = (((long long)LANES * k.N + 31) / 32) * 32;
            for (long long t = gtid; t < total; t += nthreads)
                sums_node<FP32, true, LANES>(d, k, (int)(t / LANES), (int)(t % LANES), vin);
        }
        if (!grid_barrier(d, k.bar_spins, epoch)) return false;
        for (int i = gtid; i < k.N; i += nthreads) epilogue_node<FP32, true>(d, k, i, vin, 1);
    } else if constexpr (TILES || (LANES == 1 && !FP32)) {
        run_plain_nodes<FP32, BLOCK, TILES>(d, k, lo0, hi0, vin, st & 1);
        if (!grid_barrier(d, k.bar_spins, epoch)) return false;
        if (gtid == 0) d.spec_n[(st + 1) & 1] = 0;
        run_special_nodes<FP32, BLOCK>(d, k, vin, st & 1);
    } else {
        for (int node0 = blockIdx.x * (BLOCK / LANES); node0 < k.N; node0 += gridDim.x * (BLOCK / LANES))
            force_block<FP32, true, LANES, BLOCK>(d, k, node0, vin, 1);
    }
    // the end of the launch orders the last step before whatever follows
    return st + 1 >= nsteps || grid_barrier(d, k.bar_spins, epoch);
}

// nsteps time steps in one cooperative launch, phases separated by bounded
// grid barriers.  Every step reads its current displacement and positions
// through s_cur_u / s_cur_pq, the buffers of its parity (the FP32 split keeps
// two of each; the FP64 path one).
// (Capped at 128 registers, four blocks of 128 threads per SM.  What one thread
// per node without tiles needs beside them is the L1 that tiles would take from
// its gathers: horizon 4 h, 306907 nodes, blocks of 256, with the tiles' shared
// memory FP32 split 75.7 us a step and FP64 284, without 62.5 and 240.  Twice
// the threads at 64 registers: FP32 split 60.4, but 157138 nodes of it 38 us
// for 43, 49438 nodes 17.9 for 16.4, 10010 nodes 8.8 for 8.1.)
template <bool FP32, int LANES, int BLOCK, bool TILES>
__global__ void __launch_bounds__(BLOCK, run_blocks(BLOCK))
    k_persistent(DevPtrs d, KParams k, int vin, int nsteps) {
    __shared__ int sm[33];
    // wait test: the withheld block never arrives, so the others' barrier waits run out
    if ((int)blockIdx.x == k.withhold_block) return;
    // read by every thread before the first grid barrier; written only after it
    const bool pred0 = FP32 && *(volatile int *)d.pred_ok != 0;
    const long long step0 = __ldcg(d.step);
    unsigned epoch = 0;
    for (int st = 0; st < nsteps; ++st) {
        if (threadIdx.x == 0) {
            s_cur_u = d.ub[vin ^ 1];
            s_cur_pq = d.pqb[vin ^ 1];
            s_cur_t = (double)(step0 + st + 1) * k.dt;
            s_cur_wall = d.wall_cell + (st & 1) * k.n_agg;
            s_raise = st + 1 < nsteps ? &d.rebuild3[(st + 1) % 3] : d.rebuild_next;
        }
        __syncthreads();
        const bool predicted = FP32 && (st > 0 || pred0);
        if (!persistent_step<FP32, LANES, BLOCK, TILES>(d, k, vin, st, nsteps, predicted, step0, epoch, sm)) return;
        vin ^= 1;
    }
    // the next launch may skip its first update phase (the end of this launch
    // orders every node's prediction before it)
    if (FP32 && blockIdx.x == 0 && threadIdx.x == 0) *(volatile int *)d.pred_ok = 1;
}

template <bool FP32, int LANES, int BLOCK, bool TILES>
cudaError_t launch_persistent_cfg(const DevPtrs &d, const KParams &k, int vin, int nsteps, cudaStream_t s) {
    auto kern = k_persistent<FP32, LANES, BLOCK, TILES>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t smem = TILES ? run_smem<FP32, BLOCK>() : 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BLOCK, smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const long long need = ((long long)LANES * k.N + BLOCK - 1) / BLOCK;
    const int grid = (int)std::max(1LL, std::min<long long>((long long)per_sm * sms, need));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(BLOCK);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, d, k, vin, nsteps);
}

// The persistent kernels of one precision and one thread count per node, with
// or without tiles (both block sizes), each instantiated in a translation unit
// of its own (pd_persist.cu, compiled once per combination) so that they build
// in parallel.
template <bool FP32, int LANES, bool TILES>
cudaError_t launch_persistent_lanes(const DevPtrs &d, const KParams &k, int vin, int nsteps, int block,
                                    cudaStream_t s);

// Shared-memory limits of the kernels with bond tiles (once, outside captures).
template <bool FP32>
cudaError_t init_persistent_tiles();

template <bool FP32>
cudaError_t launch_persistent_impl(const DevPtrs &d, const KParams &k, int vin, int nsteps, int block, cudaStream_t s) {
    if (k.lanes == 8) return launch_persistent_lanes<FP32, 8, false>(d, k, vin, nsteps, block, s);
    if (k.lanes == 4) return launch_persistent_lanes<FP32, 4, false>(d, k, vin, nsteps, block, s);
    if (k.lanes == 2) return launch_persistent_lanes<FP32, 2, false>(d, k, vin, nsteps, block, s);
    if (!k.pair) return launch_persistent_lanes<FP32, 1, false>(d, k, vin, nsteps, block, s);
    return launch_persistent_lanes<FP32, 1, true>(d, k, vin, nsteps, block, s);
}

}  // namespace pd
