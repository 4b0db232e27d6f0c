// Small columns in one launch of one thread-block cluster.
//
// The three launches of fp_warp.cuh are a chain of launches and global round
// trips that a column of a few hundred warp tiles cannot hide.  Here one
// cluster decodes the whole column: every warp takes consecutive tiles, the
// warps' scan elements meet in shared memory, the blocks' totals through
// distributed shared memory, and the codes of a warp's first tile stay in its
// registers from the length pass to the assembly.
//
//   1  index pass (first string of every tile, all threads) and, per warp, the
//      scan element of its tiles, last tile first;
//   2  scan of the warps' elements in the block, of the blocks' in the cluster
//      (one cluster barrier);
//   3  every warp assembles its tiles, each tile's total giving the next one
//      its offset.
//
// No wait on anything but the hardware barrier, no look-back words.  What
// bounds it is latency: at 36 tiles about 8 us, a chain of launch, extent,
// codes, two barriers, boundaries and assembly.
#pragma once
#include "fp_warp.cuh"

namespace fp {
namespace {

__device__ __forceinline__ u32 cluster_rank() {
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ u32 cluster_size() {
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Cluster barrier: writes before the arrival (shared or global) are visible
// after the wait to every thread of the cluster.
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
// (.aligned: the warp's lanes meet first, whatever branches they come from)
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A word of the same shared variable in block `rank` of the cluster.
__device__ __forceinline__ u64 ld_cluster(const u64* a, u32 rank) {
    u32 addr;
    u64 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(a)), "r"(rank));
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}

template <int CODEC, int K, bool DSMEM, int NW, int W>
__global__ void __launch_bounds__(NW * 32, 1) cluster_decode_kernel(const DecodeParams pp) {
    typedef WarpCore<CODEC, K, DSMEM, W> C;
    constexpr bool FSST = C::FSST;
    static_assert(!C::BULK_CODES, "codes in registers");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) u64 s_bar;
    __shared__ Elem s_elem[NW], s_excl[NW];
    __shared__ __align__(8) u64 s_total[3];   // the block's element
    __shared__ u64 s_base;                    // bytes before the block | entering state << 63
    uint4* s_dict = reinterpret_cast<uint4*>(smem_raw);
    uint8_t* s_lens = smem_raw + C::DICT_BYTES;
    typename C::Area& area = reinterpret_cast<typename C::Area*>(smem_raw + C::STAGED_BYTES)[threadIdx.x >> 5];
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const u32 rank = cluster_rank(), blocks = cluster_size();
    u32 err = 0;
    if (C::BULK_STAGE) {
        err = C::stage_dict_bulk(pp, s_dict, s_lens, &s_bar, NW * 32);
    } else if (DSMEM) {
        C::stage_dict(pp, s_dict, s_lens, NW * 32);
        __syncthreads();
    }
    // the launch before (the dictionary staged above is older than any launch this one may overlap)
    grid_wait();
    grid_release();
    DecodeParams p = pp;
    p.codes = after_wait(pp.codes);
    const Extent x = column_extent(p, C::TILE);
    const u32 n = (u32)x.n_tiles;
    // the block's tiles [b0, b1), the warp's [t0, t1)
    const u32 b0 = (u32)((u64)n * rank / blocks), b1 = (u32)((u64)n * (rank + 1) / blocks);
    const u32 t0 = b0 + (u32)((u64)(b1 - b0) * warp / NW), t1 = b0 + (u32)((u64)(b1 - b0) * (warp + 1) / NW);
    u32 wv[C::LANE_WORDS];
    bool in = false;
    if (t0 < t1) in = C::load_fast(p, C::lane_q0(x, t1 - 1), wv);
    const uint8_t* lens = DSMEM ? s_lens : p.dict.lens;
    index_groups(p, x, (u32)(__ffs(C::TILE) - 1), 0, (u64)p.n_strings + 1, (u64)rank * blockDim.x + threadIdx.x,
                 (u64)blocks * blockDim.x, const_cast<u32*>(p.first));
    typename C::R r;
    {
        Elem e = elem_identity();
        for (u32 t = t1; t > t0;) {
            --t;
            C::finish_load(p, x, C::lane_q0(x, t), wv, in, lens, r);
            if (t > t0) in = C::load_fast(p, C::lane_q0(x, t - 1), wv);
            const TElem te = C::tile_element(r, lane, err);
            e = then<FSST>(Elem{te.b0, te.b1, te.n}, e);
        }
        if (lane == 0) s_elem[warp] = e;
    }
    __syncthreads();
    if (warp == 0) {
        const Elem e = lane < (u32)NW ? s_elem[lane] : elem_identity();
        const Elem inc = warp_scan_incl<FSST>(e, lane, elem_identity());
        Elem lex = shfl_up_e<FSST>(inc, 1);
        if (lane == 0) lex = elem_identity();
        if (lane < (u32)NW) s_excl[lane] = lex;
        if (lane == 31) {
            s_total[0] = inc.b0;
            s_total[1] = inc.b1;
            s_total[2] = inc.n;
        }
    }
    cluster_arrive();
    cluster_wait();
    if (warp == 0) {
        Elem e = elem_identity();
        if (lane < blocks) e = Elem{ld_cluster(&s_total[0], lane), ld_cluster(&s_total[1], lane),
                                    (u32)ld_cluster(&s_total[2], lane)};
        const Elem inc = warp_scan_incl<FSST>(e, lane, elem_identity());
        Elem lex = shfl_up_e<FSST>(inc, 1);
        if (lane == 0) lex = elem_identity();
        // the column is entered on a code: state 0
        if (lane == rank) s_base = lex.b0 | ((u64)(FSST ? (lex.n & 1u) : 0u) << 63);
        if (rank == 0 && lane == 31) {
            WsHeader* ws = p.ws;
            *p.total_out = inc.b0;
            u32 bits = 0;
            if (inc.b0 > p.capacity && !p.size_only) bits |= ERRB_CAPACITY;
            if (inc.b0 > 0x7fffffffull) bits |= ERRB_OVERFLOW;
            if (*(volatile u32*)&ws->spin_limit) {   // the stall hook: nothing here waits, so report at once
                bits |= ERRB_TIMEOUT;
                ws->tile_counter = 0;
                ws->spin_limit = 0;
                ws->bar_count = 0;
            }
            if (bits) atomicOr(p.err_word, bits);
        }
    }
    cluster_arrive();   // the totals have been read: a block may end once all have arrived
    __syncthreads();
    if (t0 < t1) {
        const Elem we = s_excl[warp];
        const u32 s = (u32)(s_base >> 63);
        u64 ex = (s_base & 0x7fffffffffffffffull) + ((FSST && s) ? we.b1 : we.b0);
        ex |= (u64)(FSST ? ((we.n >> s) & 1u) : 0u) << 63;
        for (u32 t = t0; t < t1; ++t) {
            typename C::Strings sb;
            C::strings_begin(p, in_order_l2(p.first + t), in_order_l2(p.first + t + 1), sb);
            if (t > t0) C::finish_load(p, x, C::lane_q0(x, t), wv, in, lens, r);
            if (t + 1 < t1) in = C::load_fast(p, C::lane_q0(x, t + 1), wv);
            ex = C::assemble_tile(p, x, t, r, ex, sb, s_dict, area, err);
        }
        C::stage_free(lane);
    }
    if (err) atomicOr(p.err_word, err);
    cluster_wait();
}

}  // namespace
}  // namespace fp
