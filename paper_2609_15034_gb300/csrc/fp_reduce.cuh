// Pass 1 of the warp-tile decoder for large FSST-8 and OnPair-16 columns: the
// scan element of every warp tile, the code stream read once.
//
// One block per SM, some of its warps for the index pass first, its lengths
// in a shared-memory table laid out for the gather.  What bounded the general
// reduce_kernel there was the gather (OnPair-16: about 10 L1 wavefronts per 32
// codes, FSST-8: bank conflicts of 32 lanes on a 256-byte table) and the work
// around it (FSST-8: 17 instructions per slot).
//
//   FSST-8   a 256-byte row per code, lane l's copy of the entry in word l:
//            no conflicts, and one byte permutation of a code word gives the
//            address.  Literal slots are turned into 0xFF codes first (no
//            bytes) and counted; the element's second entry state differs
//            from the first by one slot's length.
//   OnPair-16  the 64 KiB of lengths once (about 3 wavefronts).
//
// A code without a token is stored with length 255 (OnPair-16): a lane's sum
// above its largest possible one gives it away, without a test per code.
//
// The 12-bit codecs stay with reduce_kernel: a 128 KiB table without
// conflicts was no faster there (36M codes: 22 us against 23, both bound by
// the integer work).
#pragma once
#include "fp_warp.cuh"

namespace fp {
namespace {

// Warps of a block that run the index pass before they join the reduce: a chunk of 256 boundaries takes a memory round trip and few
// instructions, so many warps share it, about four chunks each.
inline uint32_t reduce_index_warps(uint64_t boundaries, uint64_t blocks) {
    const uint64_t w = boundaries / (1024 * blocks) + 1;
    return w > 8 ? 8u : (uint32_t)w;
}

// Code slots from which on a codec's reduce is this one (0: never), and its
// threads per block.  Below, filling the table costs more than it saves.
// Whole calls, general reduce -> this one: OnPair-16 2.0M slots 20.6 -> 22.5
// us, 4.0M 33.4 -> 32.6, 8.0M 52 -> 49, 40M 203 -> 184 (512 threads; 1,024:
// 188); FSST-8 26.7M slots 90.0 -> 91.4, 53M 158 -> 155, 211M 553 -> 534 (640
// threads, 102 registers; 1,024 threads spill: 538).
template <int CODEC, int K>
struct LargeReduce {
    static constexpr uint64_t slots = CODEC == FP_FSST8 && K == 32 ? 40ull << 20 : CODEC == FP_ONPAIR16 ? 4ull << 20 : 0;
    static constexpr int threads = CODEC == FP_FSST8 ? 640 : 512;
};

// Every byte filled with its own sign bit.
__device__ __forceinline__ u32 spread_signs(u32 w) {
    u32 r;
    asm("prmt.b32 %0, %1, %1, 0xba98;" : "=r"(r) : "r"(w));
    return r;
}

template <int CODEC, int K>
struct LengthTable {
    typedef WarpCore<CODEC, K, false, (CODEC == FP_ONPAIR16 || CODEC == FP_ONPAIR12) ? 16 : 8, false, true> C;
    static_assert(CODEC == FP_ONPAIR16 || CODEC == FP_FSST8, "codecs with a table here");
    static constexpr int BYTES = 65536;
    static constexpr u32 MAX_SUM = 16 * K;

    // Every thread of the block; the caller synchronises.
    static __device__ __forceinline__ void fill(const DecodeParams& p, unsigned char* tab) {
        if (C::FSST) {
            for (u32 i = threadIdx.x; i < 256u * 8u; i += blockDim.x) {
                const u32 code = i >> 3;
                const u32 v = (u32)__ldg(p.dict.lens + code);   // 0 for the escape
                // a warp writes four rows; the rotation spreads their pieces over the banks
                reinterpret_cast<uint4*>(tab)[code * 16u + ((i + code) & 7u)] = make_uint4(v, v, v, v);
            }
        } else {
            const uint4* src = reinterpret_cast<const uint4*>(p.dict.lens);
            for (u32 i = threadIdx.x; i < 4096u; i += blockDim.x) {
                uint4 v = __ldg(src + i);
                v.x |= __vcmpeq4(v.x, 0u); v.y |= __vcmpeq4(v.y, 0u);
                v.z |= __vcmpeq4(v.z, 0u); v.w |= __vcmpeq4(v.w, 0u);
                reinterpret_cast<uint4*>(tab)[i] = v;
            }
        }
    }

    // Length of code k of the lane (its words wv, all inside the column), as stored.
    static __device__ __forceinline__ u32 at(const u32 (&wv)[C::LANE_WORDS], int k, const unsigned char* tab, u32 lane4) {
        if (C::FSST) {
            // address: byte 0 = 4 lane, byte 1 = the code
            const u32 a = __byte_perm(wv[k >> 2], lane4, 0x5504u | ((u32)(k & 3) << 4));
            return *reinterpret_cast<const u32*>(tab + a);
        }
        return tab[(wv[k >> 1] >> ((k & 1) * 16)) & 0xffffu];
    }

    // Byte count of the lane, its codes all inside the column.
    static __device__ __forceinline__ u32 lane_sum(const u32 (&wv)[C::LANE_WORDS], const unsigned char* tab, u32 lane4,
                                                   u32& err) {
        u32 sum = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) sum += at(wv, k, tab, lane4);
        if (!C::FSST && sum > MAX_SUM) {
            err |= ERRB_CORRUPT;
            sum = 0;
#pragma unroll 1
            for (int k = 0; k < K; ++k) {
                u32 L = 0;
#pragma unroll
                for (int j = 0; j < K; ++j)
                    if (j == k) L = at(wv, j, tab, lane4);
                sum += L == 255u ? 0u : L;
            }
        }
        return sum;
    }

    // 0xFF slots of the lane.
    static __device__ __forceinline__ u32 ff_slots(const u32 (&wv)[C::LANE_WORDS]) {
        u32 E = 0;
#pragma unroll
        for (int j = C::LANE_WORDS - 1; j >= 0; --j) {
            const u32 n = ~wv[j];
            const u32 z = ~(((n & 0x7f7f7f7fu) + 0x7f7f7f7fu) | n | 0x7f7f7f7fu);   // 0x80 in every 0xFF byte
            E = __funnelshift_l(z * 0x00204081u, E, 4);   // the four marks meet in the top four bits
        }
        return E;
    }

    // Scan elements of G consecutive tiles whose slots all lie inside the
    // column (every lane of the warp; lane 31 holds the results).
    template <int G>
    static __device__ __forceinline__ void elements(u32 (&wv)[G][C::LANE_WORDS], const unsigned char* tab, u32 lane,
                                                    u32& err, u64 (&e)[G]) {
        const u32 lane4 = lane * 4u;
        if constexpr (!C::FSST) {
            // a tile has at most 8,192 bytes: two sums in one warp reduction
            static_assert(G == 1 || G == 2, "tiles of a round");
            u32 s = lane_sum(wv[0], tab, lane4, err);
            if (G == 2) s |= lane_sum(wv[G - 1], tab, lane4, err) << 16;
            s = __reduce_add_sync(0xffffffffu, s);
            e[0] = s & 0xffffu;
            if (G == 2) e[G - 1] = s >> 16;
        } else {
            static_assert(G == 1, "one tile at a time");
            // the state entering each lane when the tile is entered on a code
            // (WarpCore::enter_state); its literals become 0xFF codes
            const u32 E = ff_slots(wv[0]);
            u32 lit, esc;
            fsst_escapes<K>(E, 0u, lit, esc);
            const u32 x0 = (esc >> (K - 1)) & 1u;
            const bool ident = E == C::full_mask();
            const u32 fixed = __ballot_sync(0xffffffffu, !ident);
            const u32 below = fixed & ((1u << lane) - 1u);
            const u32 xk = __shfl_sync(0xffffffffu, x0, below ? 31u - (u32)__clz(below) : 0u);
            const u32 s0 = below ? xk : 0u;
            fsst_escapes<K>(E, s0, lit, esc);
            u32 w[C::LANE_WORDS];
#pragma unroll
            for (int j = 0; j < C::LANE_WORDS; ++j)   // marks at the bytes' sign bits, spread over the bytes
                w[j] = wv[0][j] | spread_signs(((lit >> (4 * j)) & 0xfu) * 0x10204080u);
            const u32 b0 = __reduce_add_sync(0xffffffffu, lane_sum(w, tab, lane4, err) + __popc(lit));
            // Entered on a literal instead, the tile differs up to its first
            // slot that is not 0xFF, m slots into the first lane that has
            // one: after an even number of 0xFF slots that slot turns from a
            // code into a literal, after an odd number from a literal into a
            // code (of the run itself every other slot is a byte both times).
            const u32 first = fixed ? (u32)__ffs(fixed) - 1u : 0u;
            const u32 m = (u32)__ffs(~E & C::full_mask()) - 1u;
            u32 c = wv[0][0];
#pragma unroll
            for (int j = 1; j < C::LANE_WORDS; ++j)
                if ((m >> 2) == (u32)j) c = wv[0][j];
            const u32 L = *reinterpret_cast<const u32*>(tab + (((c >> ((m & 3u) * 8u)) & 0xffu) << 8 | lane4));
            const u32 d = __shfl_sync(0xffffffffu, (m & 1u) ? L : 1u - L, first);
            const u32 b1 = fixed ? b0 + d : b0;
            const u32 x = __shfl_sync(0xffffffffu, ident ? s0 : x0, 31);
            e[0] = wt_pack<true>(TElem{b0, b1, fixed ? x * 3u : 2u});
        }
    }
};

// A warp takes G consecutive tiles at a time, the next ones in flight.
template <int CODEC, int K>
__global__ void __launch_bounds__(LargeReduce<CODEC, K>::threads, 1) length_reduce_kernel(const DecodeParams pp, u64* agg, u32 index_warps) {
    typedef LengthTable<CODEC, K> T;
    typedef typename T::C C;
    constexpr int G = C::FSST ? 1 : 2;
    extern __shared__ __align__(128) unsigned char tab[];
    T::fill(pp, tab);   // the dictionary is older than any launch this one may overlap
    grid_wait();        // the launch before: the column may be its output, the workspace its scratch
    DecodeParams p = pp;
    p.codes = after_wait(pp.codes);
    grid_release();
    const Extent x = column_extent(p, C::TILE);
    __shared__ u32 s_unit;   // next of the block's units of G tiles
    if (threadIdx.x == 0) s_unit = 0u;
    __syncthreads();
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (warp < index_warps)
        index_by_warps(p, x, (u32)(__ffs(C::TILE) - 1), blockIdx.x * index_warps + warp, gridDim.x * index_warps,
                       const_cast<u32*>(p.first));
    // Tiles [t_lo, t_hi) lie wholly inside the column and the code buffer:
    // their lanes load their code words at a fixed stride (32-bit tile
    // indices: fewer than 2^32 tiles).  Edge tiles take the general path.
    constexpr u32 TB = C::TILE * C::WBITS / 8;   // code bytes of a tile
    const u32 nt = (u32)x.n_tiles;
    const u64 buf_slots = p.codes_bytes * 8 / C::WBITS;
    const u64 end = x.c_end < buf_slots ? x.c_end : buf_slots;
    const u64 lo64 = (x.c_begin + C::TILE - 1) / C::TILE, hi64 = end / C::TILE;
    const u32 t_lo = (u32)(lo64 - x.first_tile);
    const u32 t_hi = hi64 > lo64 ? (u32)(hi64 - x.first_tile) : t_lo;
    const uint8_t* base = p.codes + x.first_tile * (u64)TB + (u64)lane * C::LANE_BYTES;
    auto load = [&](u32 t, u32 (&w)[G][C::LANE_WORDS]) {
        const uint8_t* a = base + (u64)t * TB;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (C::LANE_BYTES % 16 == 0) {
                const uint4* src = reinterpret_cast<const uint4*>(a + g * TB);
#pragma unroll
                for (int v = 0; v < C::LANE_WORDS / 4; ++v) {
                    const uint4 q = __ldcs(src + v);
                    w[g][4 * v] = q.x; w[g][4 * v + 1] = q.y; w[g][4 * v + 2] = q.z; w[g][4 * v + 3] = q.w;
                }
            } else {
                const uint2* src = reinterpret_cast<const uint2*>(a + g * TB);
#pragma unroll
                for (int v = 0; v < C::LANE_WORDS / 2; ++v) {
                    const uint2 q = __ldcs(src + v);
                    w[g][2 * v] = q.x; w[g][2 * v + 1] = q.y;
                }
            }
        }
    };
    // units blockIdx.x, blockIdx.x + gridDim.x, ... by whichever warp is free
    auto take = [&] {
        u32 k = 0;
        if (lane == 0u) k = atomicAdd(&s_unit, 1u);
        return (__shfl_sync(0xffffffffu, k, 0) * gridDim.x + blockIdx.x) * G;
    };
    u32 err = 0;
    u32 t = take();
    u32 nv[G][C::LANE_WORDS];
    bool in = t >= t_lo && t + G <= t_hi;
    if (in) load(t, nv);
    while (t < nt) {
        u32 wv[G][C::LANE_WORDS];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < C::LANE_WORDS; ++i) wv[g][i] = nv[g][i];
        const bool now = in;
        const u32 tn = take();
        in = tn >= t_lo && tn + G <= t_hi;
        if (in) load(tn, nv);
        if (now) {
            u64 e[G];
            T::template elements<G>(wv, tab, lane, err, e);
            if (lane == 31) {
#pragma unroll
                for (int g = 0; g < G; ++g) agg[t + g] = e[g];
            }
        } else {
            typedef WarpCore<CODEC, K, false> E;   // lengths through L1
            for (u32 q = t; q < t + G && q < nt; ++q) {
                u32 gw[C::LANE_WORDS];
                const bool fast = C::load_fast(p, C::lane_q0(x, q), gw);
                typename E::R r;
                E::finish_load(p, x, E::lane_q0(x, q), gw, fast, p.dict.lens, r);
                const TElem e = E::tile_element(r, lane, err);
                if (lane == 31) agg[q] = wt_pack<C::FSST>(e);
            }
        }
        t = tn;
    }
    if (err) atomicOr(p.err_word, err);
}

}  // namespace
}  // namespace fp
