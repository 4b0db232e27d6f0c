// Selective decode (paper Sec. 1 and Sec. 2.1: the strings of an FSST-family
// column decode independently, so a subset of rows can be decoded alone).
//
// The selected rows' code slots are laid out one after another in a virtual
// slot space: row k occupies virtual slots [v[k], v[k+1]), v being the
// exclusive scan of the rows' slot counts.  Two launches build v and, for every
// 32 groups of virtual slots, the row they begin in (per-block sums of the row
// lengths, then the offsets, each block adding up the sums before it; a
// selection of more than 8 M rows has the sums scanned by a launch between
// them); the next gathers the selected codes into one contiguous stored
// stream (each thread writes whole aligned words of it), and fp_decode's
// kernels then decode that stream with v as its code_offsets.
#include <cstddef>

#include "fp_decoder.cuh"

namespace fp {
namespace {

constexpr int kRowBlock = 256;
constexpr int kRowItems = 2048;   // rows per scan block (8 per thread)
constexpr int kRowPer = kRowItems / kRowBlock;
constexpr u32 kRowDirect = 4096;  // blocks up to which every block adds up the sums before it
// Virtual slots of a gather thread, and of a warp (a chunk).
constexpr int row_group(int codec) { return codec == FP_FSST8 ? 16 : 8; }
constexpr int row_chunk(int codec) { return 32 * row_group(codec); }

// Pass 1: each block sums the slot counts of its kRowItems rows and stores
// the counts in v[] (the next pass turns them into offsets in place) and
// each row's first slot in src[].  A bad row (its id, or its offsets) counts 0
// slots and sets ERRB_CORRUPT.  The offsets are read from random places: a
// thread's eight row ids, then its sixteen offsets are in flight together,
// with no branch between them (500k rows: 14 us with one).
__global__ void __launch_bounds__(kRowBlock) rows_sums_kernel(const RowsArgs a, u32* v, u32* src, u64* block_sums,
                                                            unsigned* err_word) {
    __shared__ u64 red[kRowBlock / 32];
    grid_release();
    const u64 base = (u64)blockIdx.x * kRowItems + threadIdx.x;
    u32 err = 0;
    u64 s = 0;
    u32 id[kRowPer], b[kRowPer], e[kRowPer];
#pragma unroll
    for (int k = 0; k < kRowPer; ++k) {
        const u64 r = base + k * kRowBlock;
        id[k] = r < a.n_rows ? __ldg(a.row_ids + r) : 0u;
    }
#pragma unroll
    for (int k = 0; k < kRowPer; ++k) {
        const u32 i = id[k] < a.n_strings ? id[k] : 0u;
        b[k] = __ldg(a.code_offsets + i);
        e[k] = __ldg(a.code_offsets + i + (a.n_strings ? 1u : 0u));
    }
#pragma unroll
    for (int k = 0; k < kRowPer; ++k) {
        const u64 r = base + k * kRowBlock;
        const bool bad = id[k] >= a.n_strings || e[k] < b[k] || (u64)e[k] > a.max_slots;
        const u32 L = bad ? 0u : e[k] - b[k];
        if (r < a.n_rows) {
            if (bad) err |= ERRB_CORRUPT;
            v[r] = L;
            src[r] = b[k];
            s += L;
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31u) == 0u) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        u64 t = 0;
        for (int w = 0; w < kRowBlock / 32; ++w) t += red[w];
        block_sums[blockIdx.x] = t;
    }
    if (err) atomicOr(err_word, err);
}

// Between the passes, for many rows (one block): exclusive scan of the block sums.
__global__ void __launch_bounds__(kRowBlock) rows_scan_sums_kernel(u64* block_sums, u32 nb) {
    __shared__ u64 wsum[kRowBlock / 32];
    __shared__ u64 carry_s;
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    grid_wait();
    grid_release();
    __syncthreads();
    for (u32 base = 0; base < nb; base += kRowBlock) {
        const u32 i = base + threadIdx.x;
        const u64 x = i < nb ? block_sums[i] : 0;
        u64 inc = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (u32)d) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        u64 before = 0, tot = 0;
        for (u32 w = 0; w < kRowBlock / 32; ++w) {
            if (w < warp) before += wsum[w];
            tot += wsum[w];
        }
        const u64 carry = carry_s;
        if (i < nb) block_sums[i] = carry + before + inc - x;
        __syncthreads();
        if (threadIdx.x == 0) carry_s = carry + tot;
        __syncthreads();
    }
}

// Pass 2: v[k] = slots of the rows before k (in place), v[n_rows] = total,
// and row_of[c] = the row that holds virtual slot c * chunk.  The last block
// checks the total against the bound (and 32-bit offsets).  `scanned`: the
// block sums are offsets already.
__global__ void __launch_bounds__(kRowBlock) rows_offsets_kernel(const RowsArgs a, u32* v, const u64* block_sums,
                                                               u32 scanned, u32* row_of, u32 chunk_log2, u64 bound,
                                                               WsHeader* ws) {
    __shared__ u64 wsum[kRowBlock / 32], wbefore[kRowBlock / 32];
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const u64 base = (u64)blockIdx.x * kRowItems + (u64)threadIdx.x * kRowPer;
    grid_wait();
    grid_release();
    u32 len[kRowPer];
    u64 s = 0;
#pragma unroll
    for (int k = 0; k < kRowPer; ++k) {
        const u64 r = base + k;
        len[k] = r < a.n_rows ? v[r] : 0u;
        s += len[k];
    }
    u64 prior = 0;   // this thread's share of the blocks before
    if (!scanned)
        for (u32 i = threadIdx.x; i < blockIdx.x; i += kRowBlock) prior += block_sums[i];
    u64 inc = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const u64 y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (u32)d) inc += y;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) prior += __shfl_down_sync(0xffffffffu, prior, d);
    if (lane == 31) wsum[warp] = inc;
    if (lane == 0) wbefore[warp] = prior;
    __syncthreads();
    u64 o = scanned ? block_sums[blockIdx.x] : 0;
#pragma unroll
    for (u32 w = 0; w < kRowBlock / 32; ++w) {
        o += scanned ? 0 : wbefore[w];
        if (w < warp) o += wsum[w];
    }
    o += inc - s;
#pragma unroll
    for (int k = 0; k < kRowPer; ++k) {
        const u64 r = base + k;
        if (r <= a.n_rows) v[r] = (u32)o;   // r == n_rows: the total (32 bits; larger totals are flagged)
        if (r == a.n_rows) {
            ws->rows_slots = o;
            if (o > bound || o > 0xffffffffull) atomicOr(&ws->status, ERRB_CAPACITY);
        }
        const u64 end = o + len[k] < bound ? o + len[k] : bound;
        if (row_of)
            for (u64 c = (o + (1u << chunk_log2) - 1) >> chunk_log2; (c << chunk_log2) < end; ++c) row_of[c] = (u32)r;
        o += len[k];
    }
}

// Bits below b of a word (b may lie outside 0 .. 32).
__device__ __forceinline__ u32 bits_below(int b) { return b <= 0 ? 0u : (b >= 32 ? 0xffffffffu : (1u << b) - 1u); }

// Pass 3: gather.  A warp writes a chunk of 32 groups of G virtual slots of
// the compacted stream, a lane one group as whole words: 8 slots of 16 or 12
// bits (4 or 3 words), 16 slots of 8 bits (4 words).  The chunk's rows (about
// 14 of 18 codes, as many as slots of one code) pass through a window in
// shared memory, and a row's part of a group is one window of aligned words of
// the stored stream shifted into place, where a byte or two per slot took up
// to 16 loads and a search over all rows 20 more.
//
// The window holds a chunk of one-code rows (half of one of FSST-8's), so that
// nearly every lane finds its rows in the first one; with one of 64 rows the
// lanes past it searched global memory row by row.  500k of 5M rows, a whole
// call, a byte or two per slot -> window of 64 -> this: OnPair-12, 1 code a row
// 62.1 -> 74.0 -> 45.1 us, 2 codes 58.0 -> 59.6 -> 37.4, 18 codes 123.4 -> 88.8 ->
// 89.4; FSST-8 65.0 -> 121.8 -> 60.8, 64.2 -> 85.2 -> 47.2, 141.2 -> 81.4 -> 80.6.
// (FSST-8 with 512 rows: 1 code 57.0, but 20M selected slots of 13 codes a row
// 136 against 129: the window takes the L1 that the words need.)  A chunk of
// more rows than kRowWindows windows hold (almost all of them empty) has the
// rest searched in global memory.  Slots past the selected total (or the
// bound) are not written and never decoded.
constexpr u32 kRowWindow = 256, kRowWindows = 8;
// Blocks per SM that the registers allow without spilling (48 for FSST-8's
// groups of 16 slots, else 40; 8 blocks of 32 registers spill and are 2-8 %
// slower per call).
__host__ __device__ constexpr int row_gather_blocks(int codec) { return codec == FP_FSST8 ? 5 : 6; }

template <int CODEC>
__global__ void __launch_bounds__(kRowBlock, row_gather_blocks(CODEC)) rows_gather_kernel(const RowsArgs a, const u32* v, const u32* src,
                                                              const u32* row_of, uint8_t* out, u64 bound,
                                                              const WsHeader* ws) {
    constexpr int BITS = CODEC == FP_ONPAIR16 ? 16 : (CODEC == FP_FSST8 ? 8 : 12);
    constexpr int G = CODEC == FP_FSST8 ? 16 : 8, CH = 32 * G, NW = G * BITS / 32;
    constexpr u32 WIN = kRowWindow;
    __shared__ u32 s_v[kRowBlock / 32][WIN + 1], s_src[kRowBlock / 32][WIN];
    grid_wait();
    grid_release();
    const u64 total_raw = *(const volatile u64*)&ws->rows_slots;
    // a total past 32 bits left v[] wrapped (and flagged): gather nothing
    const u64 total64 = total_raw > 0xffffffffull ? 0 : (total_raw < bound ? total_raw : bound);
    const u32 total = (u32)total64;
    const u32 n_chunks = (u32)((total64 + CH - 1) / CH);
    const u32 m = a.n_rows, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    u32* const wv = s_v[warp];
    u32* const wsrc = s_src[warp];
    // the stored stream as words, zero outside it; its last bytes make a word
    // of their own.  The buffer may be larger than slots can name: 2^32 codes
    // of 16 bits lie in the first 2^31 words, so more are not counted.
    const u32* const words = reinterpret_cast<const u32*>(a.codes);
    const u64 all_words = a.codes_bytes / 4;
    const u32 n_words = all_words < (1ull << 31) ? (u32)all_words : 1u << 31;
    u32 tail = 0;
    for (u32 q = 0; q < (u32)(a.codes_bytes & 3u); ++q) tail |= (u32)__ldg(a.codes + 4 * all_words + q) << (8 * q);
    auto word = [&](u32 i) { return i < n_words ? __ldg(words + i) : (i == n_words ? tail : 0u); };
    for (u32 c = blockIdx.x * (kRowBlock / 32) + warp; c < n_chunks; c += gridDim.x * (kRowBlock / 32)) {
        // the chunk's rows lie in [k0, k_end)
        const u32 k0 = row_of[c], k_end = c + 1u < n_chunks ? row_of[c + 1u] + 1u : m;
        const u32 v0 = c * (u32)CH + lane * G;
        u32 acc[NW] = {};
        const u32 left = v0 < total ? min(total - v0, (u32)G) : 0u;
        u32 j = 0;   // slots of the group done
        // slots j .. of the group from the row of slot v0 + j (non-empty, so
        // its id passed the checks): its first virtual slot, its end, its
        // first stored slot
        auto take = [&](u32 vs, u32 ve, u32 sb) {
            const u32 end = min(left, ve - v0);
            // the words from the stored bit of the group's slot 0 on, as if
            // the row began early enough (only those that slots j .. end - 1
            // touch are loaded: 2 of 5 for a row of one code)
            const long long bit = (long long)BITS * ((long long)sb + v0 - vs);
            const u32 w0 = (u32)(bit >> 5);
            const u32 q_lo = j * BITS / 32u, q_hi = (end * BITS - 1u) / 32u + 1u;
            // one check for all of them: a check per word cost 3 % of a call
            u32 x[NW + 1];
            if (bit >= 0 && (u64)w0 + NW < n_words) {
#pragma unroll
                for (int q = 0; q <= NW; ++q) x[q] = (u32)q >= q_lo && (u32)q <= q_hi ? __ldg(words + w0 + q) : 0u;
            } else {
#pragma unroll
                for (int q = 0; q <= NW; ++q) x[q] = word(w0 + q);
            }
#pragma unroll
            for (int q = 0; q < NW; ++q) {
                const u32 keep = j ? bits_below((int)j * BITS - 32 * q) : 0u;
                acc[q] = (acc[q] & keep) | (__funnelshift_r(x[q], x[q + 1], (u32)bit) & ~keep);
            }
            j = end;
        };
        u32 base = k0;
        for (u32 w = 0; w < kRowWindows; ++w) {
            const u32 n_in = min(k_end - base, WIN);
            for (u32 i = lane; i <= n_in; i += 32u) {
                wv[i] = v[base + i];
                if (i < n_in) wsrc[i] = src[base + i];
            }
            __syncwarp();
            const u32 covered = wv[n_in], step = n_in > 1u ? 1u << (31 - __clz(n_in - 1u)) : 0u;
            u32 i = n_in;   // the row in the window
            while (j < left && v0 + j < covered) {
                const u32 pos = v0 + j;
                if (i == n_in) {
                    i = 0u;
                    for (u32 d = step; d > 0u; d >>= 1)
                        if (i + d < n_in && wv[i + d] <= pos) i += d;
                } else {
                    do ++i;
                    while (wv[i + 1] <= pos);
                }
                take(wv[i], wv[i + 1], wsrc[i]);
            }
            base += n_in;
            const bool done = __all_sync(0xffffffffu, j >= left) || base >= k_end;
            __syncwarp();   // the window is refilled
            if (done) break;
        }
        while (j < left && base < k_end) {
            const u32 pos = v0 + j;
            u32 hi = k_end;   // v[base] <= pos < v[hi]
            while (hi - base > 1u) {
                const u32 mid = base + (hi - base) / 2u;
                if (v[mid] <= pos) base = mid;
                else hi = mid;
            }
            take(v[base], v[base + 1], src[base]);
        }
        if (left < (u32)G)
#pragma unroll
            for (int q = 0; q < NW; ++q) acc[q] &= bits_below((int)left * BITS - 32 * q);
        if (left) {
            const u64 g = (u64)c * 32u + lane;
            if (NW == 4) {
                reinterpret_cast<uint4*>(out)[g] = make_uint4(acc[0], acc[1], acc[2], acc[NW - 1]);
            } else {
                u32* w = reinterpret_cast<u32*>(out) + 3 * g;
                w[0] = acc[0];
                w[1] = acc[1];
                w[2] = acc[2];
            }
        }
    }
}

// Launch that may start while the launch before it finishes (it waits in the kernel).
template <class... A, class... B>
cudaError_t launch_early(void (*kernel)(A...), u32 grid, cudaStream_t stream, B... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kRowBlock);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, (A)args...);
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

RowsLayout rows_layout(int codec, uint32_t n_rows, uint64_t selected_slots) {
    RowsLayout L{};
    const uint64_t nb = ((uint64_t)n_rows + kRowItems - 1) / kRowItems + 1;
    L.o_v = 0;
    L.o_src = al256(((size_t)n_rows + 1) * sizeof(u32));
    L.o_sums = L.o_src + al256(((size_t)n_rows + 1) * sizeof(u32));
    L.o_row_of = L.o_sums + al256(nb * sizeof(u64));
    L.o_codes = L.o_row_of + al256((selected_slots / row_chunk(codec) + 1) * sizeof(u32));
    const uint64_t G = row_group(codec), group_bytes = G * code_bits(codec) / 8;
    const uint64_t groups = (selected_slots + G - 1) / G;
    L.codes_bytes = (selected_slots * code_bits(codec) + 7) / 8;
    L.bytes = L.o_codes + al256(groups * group_bytes + 16);
    return L;
}

cudaError_t launch_rows_gather(int codec, const RowsArgs& a, uint64_t selected_slots, bool gather, void* scratch,
                               const RowsLayout& L, WsHeader* ws, int sms, cudaStream_t stream) {
    char* base = static_cast<char*>(scratch);
    u32* v = reinterpret_cast<u32*>(base + L.o_v);
    u32* src = reinterpret_cast<u32*>(base + L.o_src);
    u64* sums = reinterpret_cast<u64*>(base + L.o_sums);
    u32* row_of = reinterpret_cast<u32*>(base + L.o_row_of);
    uint8_t* codes = reinterpret_cast<uint8_t*>(base + L.o_codes);
    const u32 nb = (u32)((uint64_t)a.n_rows / kRowItems) + 1;   // the blocks of v[0 .. n_rows]
    rows_sums_kernel<<<nb, kRowBlock, 0, stream>>>(a, v, src, sums, &ws->status);
    cudaError_t e = cudaGetLastError();
    const u32 scanned = nb > kRowDirect ? 1u : 0u;
    if (e == cudaSuccess && scanned) e = launch_early(rows_scan_sums_kernel, 1, stream, sums, nb);
    const u32 chunk_log2 = codec == FP_FSST8 ? 9 : 8;
    if (e == cudaSuccess)
        e = launch_early(rows_offsets_kernel, nb, stream, a, v, sums, scanned, gather ? row_of : nullptr, chunk_log2,
                         selected_slots, ws);
    if (e != cudaSuccess || !gather) return e;
    const uint64_t per_block = (uint64_t)row_chunk(codec) * (kRowBlock / 32);
    uint64_t grid = (selected_slots + per_block - 1) / per_block;
    const uint64_t grid_max = (uint64_t)sms * row_gather_blocks(codec);
    if (grid > grid_max) grid = grid_max;
    if (grid < 1) grid = 1;
    const u32 g = (u32)grid;
    switch (codec) {
        case FP_ONPAIR16: return launch_early(rows_gather_kernel<FP_ONPAIR16>, g, stream, a, v, src, row_of, codes, selected_slots, ws);
        case FP_ONPAIR12: return launch_early(rows_gather_kernel<FP_ONPAIR12>, g, stream, a, v, src, row_of, codes, selected_slots, ws);
        case FP_FSST8: return launch_early(rows_gather_kernel<FP_FSST8>, g, stream, a, v, src, row_of, codes, selected_slots, ws);
        default: return launch_early(rows_gather_kernel<FP_FSST12>, g, stream, a, v, src, row_of, codes, selected_slots, ws);
    }
}

}  // namespace fp
