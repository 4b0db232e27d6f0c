// Warp-tile decoder: the column is cut into warp tiles of 32*K code slots,
// and a decode runs in three launches:
//
//   reduce_kernel (or length_reduce_kernel, fp_reduce.cuh)  its first blocks
//                   run the index pass (the first string boundary of every
//                   warp tile); in the others each warp computes the scan
//                   element of a warp tile (its decoded bytes; for FSST-8
//                   the two-state element of the escape parity) and stores
//                   it: fully parallel, the code stream is read once;
//   tiles_scan_kernel  single-pass exclusive scan of the warp-tile elements
//                   (blocks of 2,048 elements, decoupled look-back across
//                   blocks): every warp tile's output offset and entering
//                   escape state;
//   warp_decode_kernel  every warp decodes whole warp tiles on its own: code
//                   unpack, lengths, a warp scan inside the tile, assembly in
//                   a per-warp staging area in shared memory, one bulk copy
//                   of its whole 16-byte chunks, string offsets.  No block
//                   barrier and no wait on other warps, so the SM hides the
//                   latency of one warp's loads with the others' work.
//
// Reading the code stream twice costs its bytes (about a fifth of the
// traffic at 6 decoded bytes per 12-bit code) but removes the serial
// look-back from the decode itself; this is the paper's sidecar (Sec. 3.1)
// regenerated on the device by the first two passes.
#pragma once
#include <type_traits>

#include "fp_decoder.cuh"

namespace fp {
namespace {

// Warp-tile element <-> 64-bit word (bytes of a warp tile stay below 2^20).
template <bool FSST>
__device__ __forceinline__ u64 wt_pack(const TElem& e) {
    if (!FSST) return e.b0;
    return (u64)e.b0 | ((u64)e.b1 << 24) | ((u64)(e.n & 3u) << 48);
}
template <bool FSST>
__device__ __forceinline__ Elem wt_unpack(u64 w) {
    if (!FSST) return Elem{w, 0, 0};
    return Elem{w & 0xffffffull, (w >> 24) & 0xffffffull, (u32)((w >> 48) & 3u)};
}

// A lane's run of tokens appended to the warp's staging area as aligned
// 64-bit words: `m` bytes of the current word (at `at`) are in c0, c1.
//
// Words in shared memory instead of 16-byte chunks in registers: moving a
// token into a 16-byte window took about 12 selects, 8 funnel shifts and a
// scattered 16-byte store, and that integer work bound the decode (ALU pipe
// 64-72 % active).  Of the word sizes, 32 bits take the fewest instructions
// (five shifts, four selects) but up to four stores a token, 64 bits two more
// selects per word and at most two stores, one for FSST symbols.  The decode
// kernel, 16-byte window -> 32-bit -> 64-bit words: OnPair-12, 36M codes 149 ->
// 118 -> 110 us; FSST-8, 38M slots 134 -> 93 -> 92; FSST-12, 33M codes 110 -> 72
// -> 70.  What bounds it now is the shared-memory pipe (77 % of its wavefronts
// on OnPair-12: about 10 per 32 codes for the table reads, 8 for these
// stores, 3 for the lengths), with the ALU pipe at 66 %.
struct StageWriter {
    u64* at;
    u32 m, c0, c1;

    // Continue at staging byte `pos`; a word begun by the lanes before is
    // completed here with their bytes zero, and they add theirs by
    // finish().
    __device__ __forceinline__ void begin(u32* stage, u32 pos) {
        at = reinterpret_cast<u64*>(stage) + (pos >> 3);
        m = pos & 7u;
        c0 = c1 = 0u;
    }
    // Append a token of up to 16 bytes (zero past its length).
    __device__ __forceinline__ void put(const uint4 t, u32 len) {
        const u32 sh = m * 8u;
        const bool q = (m & 4u) != 0u;
        const u32 y0 = __funnelshift_l(0u, t.x, sh), y1 = __funnelshift_l(t.x, t.y, sh),
                  y2 = __funnelshift_l(t.y, t.z, sh), y3 = __funnelshift_l(t.z, t.w, sh),
                  y4 = __funnelshift_l(t.w, 0u, sh);
        const u32 z0 = c0 | (q ? 0u : y0), z1 = c1 | (q ? y0 : y1), z2 = q ? y1 : y2, z3 = q ? y2 : y3,
                  z4 = q ? y3 : y4, z5 = q ? y4 : 0u;
        const u32 e = m + len;
        if (e >= 8u) *reinterpret_cast<uint2*>(at) = make_uint2(z0, z1);
        if (e >= 16u) *reinterpret_cast<uint2*>(at + 1) = make_uint2(z2, z3);
        c0 = e >= 8u ? z2 : z0;
        c1 = e >= 8u ? z3 : z1;
        c0 = e >= 16u ? z4 : c0;
        c1 = e >= 16u ? z5 : c1;
        at += e >> 3;
        m = e & 7u;
    }
    // Append a token of up to 8 bytes (zero past its length).
    __device__ __forceinline__ void put8(const uint2 t, u32 len) {
        const u32 sh = m * 8u;
        const bool q = (m & 4u) != 0u;
        const u32 y0 = __funnelshift_l(0u, t.x, sh), y1 = __funnelshift_l(t.x, t.y, sh),
                  y2 = __funnelshift_l(t.y, 0u, sh);
        const u32 z0 = c0 | (q ? 0u : y0), z1 = c1 | (q ? y0 : y1), z2 = q ? y1 : y2, z3 = q ? y2 : 0u;
        const u32 e = m + len;
        if (e >= 8u) *reinterpret_cast<uint2*>(at) = make_uint2(z0, z1);
        c0 = e >= 8u ? z2 : z0;
        c1 = e >= 8u ? z3 : z1;
        at += e >> 3;
        m = e & 7u;
    }
    // The lane's bytes of a word that a following lane completed (every lane
    // of the warp has stored its words).
    __device__ __forceinline__ void finish() {
        u32* a = reinterpret_cast<u32*>(at);
        if (c0) atomicOr(a, c0);
        if (c1) atomicOr(a + 1, c1);
    }
};

// Per-warp shared-memory area of the decode kernel.  `stage` holds up to CAP
// decoded bytes, at the alignment they have in the output, so that the whole
// 16-byte chunks leave by one bulk copy per tile (no store instructions, and
// no scattered lines in L1).
template <int K, int CAP, int CODE_BYTES>
struct WarpArea {
    uint4 stage[CAP / 16 + 1];
    // code bytes of the tile to decode next (bulk copy)
    uint4 codes[CODE_BYTES ? CODE_BYTES / 16 : 1];
    u32 pre[K / 4][32];     // tile-relative output offset of slot 4m of each lane
    u32 contrib[K / 4][32]; // bytes each slot produced, one byte per slot
    u32 lit_mask[32];       // FSST-8: bit k = slot k holds a literal byte
};

// W: dictionary read width of the OnPair codecs (paper Sec. 3.2 and 4.3):
// 16 reads whole 16-byte entries, 8 reads the low plane (bytes 0-7) for
// every token and the high plane (bytes 8-15) only for longer tokens.  The
// FSST codecs have 8-byte entries (W = 8).
// PACKED: the codes are stored bit-packed at p.packed_bits bits per code
// (LSB-first, 1..16) instead of the codec's own layout -- the cascade layer
// the paper removes on the host (Sec. 5), unpacked here inside the kernels.
// LSMEM: the length table is staged in shared memory (with DSMEM the
// dictionary too).  OnPair-16 stages its 64 KiB of lengths: a gather of 32
// bytes takes about 3 wavefronts there against 10 through L1, whose lines
// then serve the tokens (40M codes: 250 -> 210 us per call).
template <int CODEC, int K, bool DSMEM, int W = (CODEC == FP_ONPAIR16 || CODEC == FP_ONPAIR12) ? 16 : 8,
          bool PACKED = false, bool LSMEM = DSMEM>
struct WarpCore {
    static constexpr bool FSST = (CODEC == FP_FSST8);   // escape codec: two-state scan elements
    static constexpr bool TOK8 = (CODEC == FP_FSST8 || CODEC == FP_FSST12);   // 8-byte table entries
    static constexpr bool W12 = (CODEC == FP_ONPAIR12 || CODEC == FP_FSST12);  // 12-bit codes
    static constexpr int TILE = 32 * K;
    static constexpr int WBITS = (CODEC == FP_ONPAIR16) ? 16 : (W12 ? 12 : 8);
    static constexpr int LANE_BYTES = K * WBITS / 8;   // code bytes of one lane
    // words a lane loads: its code bytes, or (packed codes) at most as many
    static constexpr int LANE_WORDS = LANE_BYTES / 4;
    // entries of the table (a staged table, or the global planes)
    static constexpr int kTable = (CODEC == FP_FSST8) ? 256 : (CODEC == FP_ONPAIR16 ? 65536 : 4096);
    // FSST-8 with a staged table: the symbols, then the 256 literal bytes as
    // tokens of their own, so a slot reads entry code + 256 * literal.
    static constexpr bool LITTAB = FSST && DSMEM;
    static constexpr int DICT_BYTES = DSMEM ? (kTable + (LITTAB ? 256 : 0)) * (TOK8 ? 8 : 16) : 0;
    // Staged output bytes of a warp: an ordinary tile in one round (512
    // tokens of 7.5 bytes: 3.8 KB; 1,024 FSST symbols: 4.6 KB); less where
    // the dictionary is read through L1, which shares the SM's memory.
    static constexpr int CAP = DSMEM ? 6144 : 4096;
    static constexpr int TILE_BYTES = TILE * WBITS / 8;   // code bytes of a tile, at most
    static __device__ __forceinline__ u32 tile_bytes(const DecodeParams& p) {
        return PACKED ? TILE / 8 * p.packed_bits : (u32)TILE_BYTES;   // a multiple of 16
    }
    // The next tile's codes come by a bulk copy into the warp's area (32-slot
    // lanes), or into registers.  The copy frees 8 to 12 registers and
    // writes each line once where lanes 32 or 48 bytes apart touch it several
    // times; 32-slot lanes are short of registers (FSST-8 16M strings 601 ->
    // 576 us per call, FSST-12 documents 114 -> 105), 16-slot lanes are not
    // and only pay the wait (OnPair-12 10M 648 -> 659).
    static constexpr bool BULK_CODES = K == 32;
    typedef WarpArea<K, CAP, BULK_CODES ? TILE_BYTES : 0> Area;
    static constexpr int LENS_BYTES = LSMEM ? kTable : 0;
    static constexpr int STAGED_BYTES = DICT_BYTES + LENS_BYTES;   // tables in front of the warp areas
    typedef TileRegs<CODEC, K> R;
    static_assert(K == 8 || K == 16 || K == 32, "slots per lane");
    static_assert(!FSST || K >= 16, "FSST-8 handles 16 slots at a time");
    static_assert(!DSMEM || CODEC != FP_ONPAIR16, "OnPair-16 tables do not fit in shared memory");
    static_assert(LANE_BYTES % 8 == 0, "lane code bytes are read in 8-byte words");
    static_assert(W == 16 || W == 8, "read width");
    static_assert(!TOK8 || W == 8, "FSST entries are 8 bytes");
    static_assert(!PACKED || (!FSST && K >= 16), "packed codes: escape-free codecs, 16 or 32 slots per lane");

    static __device__ __forceinline__ u32 full_mask() { return K == 32 ? 0xffffffffu : ((1u << K) - 1u); }

    // ---- codes of slots [q0, q0 + K) ---------------------------------------
    static __device__ __forceinline__ void unpack_words(const u32* wv, R& r) {
        if (W12) {
#pragma unroll
            for (int g = 0; g < K / 8; ++g) {
                const u32 a = wv[3 * g], bb = wv[3 * g + 1], c = wv[3 * g + 2];
                r.c[4 * g + 0] = (a & 0xfffu) | (((a >> 12) & 0xfffu) << 16);
                r.c[4 * g + 1] = (__funnelshift_r(a, bb, 24) & 0xfffu) | (((bb >> 4) & 0xfffu) << 16);
                r.c[4 * g + 2] = ((bb >> 16) & 0xfffu) | ((__funnelshift_r(bb, c, 28) & 0xfffu) << 16);
                r.c[4 * g + 3] = ((c >> 8) & 0xfffu) | ((c >> 20) << 16);
            }
        } else {
#pragma unroll
            for (int m = 0; m < R::CW; ++m) r.c[m] = wv[m];
        }
    }

    // Raw code words of the lane (LANE_WORDS words); false if they run past
    // the buffer (then load_guarded() is used).  AHEAD: read before the
    // kernel's wait (past L1).
    template <bool AHEAD = false>
    static __device__ __forceinline__ bool load_fast(const DecodeParams& p, u64 q0, u32 (&wv)[LANE_WORDS]) {
        if (PACKED) {
            const u64 w0 = (q0 * p.packed_bits) >> 5;   // the word holding the lane's first bit
            const u32 n = packed_words(p.packed_bits);
            if ((w0 + n) * 4 > p.codes_bytes) return false;
            load_packed<AHEAD>(reinterpret_cast<const u32*>(p.codes) + w0, n, wv);
            return true;
        }
        const u64 b0 = q0 * WBITS / 8;   // q0 is a multiple of K, K a multiple of 8
        if (b0 + LANE_BYTES > p.codes_bytes) return false;
        if (LANE_BYTES % 16 == 0) {
            const uint4* src = reinterpret_cast<const uint4*>(p.codes + b0);
#pragma unroll
            for (int v = 0; v < LANE_BYTES / 16; ++v) {
                const uint4 a = AHEAD ? __ldcg(src + v) : __ldcs(src + v);
                wv[4 * v] = a.x; wv[4 * v + 1] = a.y; wv[4 * v + 2] = a.z; wv[4 * v + 3] = a.w;
            }
        } else {
            const uint2* src = reinterpret_cast<const uint2*>(p.codes + b0);
#pragma unroll
            for (int v = 0; v < LANE_BYTES / 8; ++v) {
                const uint2 a = AHEAD ? __ldcg(src + v) : __ldcs(src + v);
                wv[2 * v] = a.x; wv[2 * v + 1] = a.y;
            }
        }
        return true;
    }

    // The same words from the tile's bulk-copied code bytes.
    static __device__ __forceinline__ void load_staged(const DecodeParams& p, const uint4* codes, u32 lane,
                                                       u32 (&wv)[LANE_WORDS]) {
        if (PACKED) {
            // words b apart over the lanes: at most 8 lanes of a load share a bank (b = 8), 2 at 10 bits
            const u32* src = reinterpret_cast<const u32*>(codes) + lane * p.packed_bits;
#pragma unroll
            for (int i = 0; i < LANE_WORDS; ++i) wv[i] = (u32)i < p.packed_bits ? src[i] : 0u;
            return;
        }
#pragma unroll
        for (int v = 0; v < LANE_BYTES / 16; ++v) {
            const uint4 a = codes[lane * (LANE_BYTES / 16) + v];
            wv[4 * v] = a.x; wv[4 * v + 1] = a.y; wv[4 * v + 2] = a.z; wv[4 * v + 3] = a.w;
        }
    }

    static __device__ void load_guarded(const DecodeParams& p, u64 q0, R& r) {
        if (PACKED) {
            // bit-packed codes near the end of the buffer: byte by byte
            const u32 b = p.packed_bits, mask = (1u << b) - 1u;
#pragma unroll
            for (int m = 0; m < K / 2; ++m) {
                u32 v = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const u64 q = q0 + 2 * m + h;
                    if (q < p.max_slots) {
                        const u64 P = q * b, by = P >> 3;
                        u32 x = 0;
#pragma unroll
                        for (int e = 0; e < 3; ++e)
                            if (by + e < p.codes_bytes) x |= (u32)p.codes[by + e] << (8 * e);
                        v |= ((x >> (P & 7u)) & mask) << (16 * h);
                    }
                }
                r.c[m] = v;
            }
            return;
        }
        if (CODEC == FP_ONPAIR16) {
#pragma unroll
            for (int m = 0; m < K / 2; ++m) {
                u32 v = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const u64 q = q0 + 2 * m + h;
                    if (q < p.max_slots) v |= ((u32)p.codes[2 * q] | ((u32)p.codes[2 * q + 1] << 8)) << (16 * h);
                }
                r.c[m] = v;
            }
        } else if (W12) {
#pragma unroll
            for (int m = 0; m < K / 2; ++m) {
                u32 v = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const u64 q = q0 + 2 * m + h;
                    if (q < p.max_slots) {
                        const u64 by = q * 3 / 2;
                        const u32 lo8 = p.codes[by], hi8 = p.codes[by + 1];
                        const u32 c = (q & 1) ? ((lo8 >> 4) | (hi8 << 4)) : (lo8 | ((hi8 & 0xfu) << 8));
                        v |= c << (16 * h);
                    }
                }
                r.c[m] = v;
            }
        } else {
#pragma unroll
            for (int m = 0; m < K / 4; ++m) {
                u32 v = 0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const u64 q = q0 + 4 * m + h;
                    if (q < p.max_slots) v |= (u32)p.codes[q] << (8 * h);
                }
                r.c[m] = v;
            }
        }
    }

    // Packed codes of b bits: 32 of them are b words.  A lane's 16 are 16 b bits
    // from a multiple of 16 bits on, so they begin at a word, or (odd b, odd
    // lanes) in the middle of one, and lie in these words either way.
    static __device__ __forceinline__ u32 packed_words(u32 b) { return K == 32 ? b : (b + 1u) >> 1; }
    template <bool AHEAD = false>
    static __device__ __forceinline__ void load_packed(const u32* src, u32 n, u32* wv) {
#pragma unroll
        for (int i = 0; i < LANE_WORDS; ++i) wv[i] = (u32)i < n ? (AHEAD ? __ldcg(src + i) : __ldcs(src + i)) : 0u;
    }
    // `o`: the bit the codes begin at in wv[0], 0 or 16.
    template <int B>
    static __device__ __forceinline__ void unpack_bits(const u32 (&wv)[LANE_WORDS], u32 o, R& r) {
        constexpr int N = (K * B + 31) / 32;
        constexpr u32 MASK = (1u << B) - 1u;
        u32 w[N + 1];
#pragma unroll
        for (int i = 0; i < N; ++i) w[i] = (K == 16 && (B & 1)) ? __funnelshift_r(wv[i], i + 1 < N ? wv[i + 1] : 0u, o) : wv[i];
        w[N] = 0u;
#pragma unroll
        for (int m = 0; m < K / 2; ++m) {
            const int bit = 2 * m * B, i = bit >> 5, sh = bit & 31;
            const u32 two = sh + 2 * B <= 32 ? w[i] >> sh : __funnelshift_r(w[i], w[i + 1], sh);
            r.c[m] = B == 16 ? two : (two & MASK) | ((two << (16 - B)) & (MASK << 16));
        }
    }
    // (a width above the codec's own is refused by the host)
    template <int B>
    static __device__ __forceinline__ void unpack_width(const u32 (&wv)[LANE_WORDS], u32 o, R& r) {
        unpack_bits<B <= WBITS ? B : WBITS>(wv, o, r);
    }
    // Every width has a body of its own, taken by one branch that is the same
    // for the whole grid: constant bit positions cost two instructions a
    // code, positions computed from a run-time width about seven and two
    // wavefronts of the shared-memory pipe a code (the words have to be
    // indexed there).  FSST-12 at 10 bits, 16M strings: 562 -> 492 us a call,
    // with the reduce summing lengths as for the codec's own layout.
    static __device__ __forceinline__ void unpack_packed(const u32 (&wv)[LANE_WORDS], u32 o, u32 b, R& r) {
        switch (b) {
            case 1: unpack_width<1>(wv, o, r); break;
            case 2: unpack_width<2>(wv, o, r); break;
            case 3: unpack_width<3>(wv, o, r); break;
            case 4: unpack_width<4>(wv, o, r); break;
            case 5: unpack_width<5>(wv, o, r); break;
            case 6: unpack_width<6>(wv, o, r); break;
            case 7: unpack_width<7>(wv, o, r); break;
            case 8: unpack_width<8>(wv, o, r); break;
            case 9: unpack_width<9>(wv, o, r); break;
            case 10: unpack_width<10>(wv, o, r); break;
            case 11: unpack_width<11>(wv, o, r); break;
            case 12: unpack_width<12>(wv, o, r); break;
            case 13: unpack_width<13>(wv, o, r); break;
            case 14: unpack_width<14>(wv, o, r); break;
            case 15: unpack_width<15>(wv, o, r); break;
            default: unpack_width<16>(wv, o, r); break;
        }
    }

    // Codes, from words load_fast() or load_staged() fetched or by guarded
    // loads.
    static __device__ __forceinline__ void unpack(const DecodeParams& p, u64 q0, const u32 (&wv)[LANE_WORDS], bool fast,
                                                  R& r) {
        if (fast) {
            if constexpr (PACKED) unpack_packed(wv, (u32)((q0 * p.packed_bits) & 31u), p.packed_bits, r);
            else unpack_words(wv, r);
        } else {
            load_guarded(p, q0, r);
        }
    }

    // The slots of the lane inside the column.
    static __device__ __forceinline__ void mark_valid(const Extent& x, u64 q0, R& r) {
        if (q0 >= x.c_begin && q0 + K <= x.c_end) {
            r.valid = full_mask();
        } else {
            u32 v = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const u64 q = q0 + k;
                v |= ((q >= x.c_begin && q < x.c_end) ? 1u : 0u) << k;
            }
            r.valid = v;
        }
    }

    // The codes, the slots inside the column and their token lengths.
    static __device__ __forceinline__ void finish_load(const DecodeParams& p, const Extent& x, u64 q0,
                                                       const u32 (&wv)[LANE_WORDS], bool fast, const uint8_t* lens,
                                                       R& r) {
        unpack(p, q0, wv, fast, r);
        mark_valid(x, q0, r);
#pragma unroll
        for (int j = 0; j < K / 4; ++j) {
            u32 w = 0;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const u32 code = code_at<CODEC, K>(r, 4 * j + h);
                const u32 L = LSMEM ? (u32)lens[code] : (u32)__ldg(lens + code);
                w |= L << (8 * h);
            }
            r.L[j] = w;
        }
    }

    // FSST-8 helpers on the lane's registers.
    static __device__ __forceinline__ u32 ff_mask(const R& r) {
        u32 E = 0;
#pragma unroll
        for (int j = 0; j < K / 4; ++j) E |= ff_bits4(r.c[j]) << (4 * j);
        return E;
    }
    static __device__ __forceinline__ u32 fsst_bytes(const R& r, u32 codes, u32 lits) {
        u32 n = __popc(lits);
#pragma unroll
        for (int j = 0; j < K / 4; ++j) n = masked_byte_sum(r.L[j], ones_of4(codes >> (4 * j)), n);
        return n;
    }

    // FSST-8 escape state across lanes.  A lane maps the state entering it
    // (1: its first slot is a literal) to the state after it.  For a lane
    // whose K slots are all 0xFF that map is the identity (codes and
    // literals alternate, K is even); for any other lane it is constant: a
    // slot that is not 0xFF (or lies outside the column, which resets the
    // state) fixes the parity of every later slot.  x0 is the state after
    // the lane entered with 0; `ident` marks the identity lanes.
    static __device__ __forceinline__ void lane_state(const R& r, bool allv, u32 E, u32& x0, bool& ident) {
        if (allv) {
            u32 lit, esc;
            fsst_escapes<K>(E, 0u, lit, esc);
            x0 = (esc >> (K - 1)) & 1u;
            ident = (E == full_mask());
            return;
        }
        u32 st = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool v = (r.valid >> k) & 1u;
            st = v ? (st ? 0u : (code_at<CODEC, K>(r, k) == 255u ? 1u : 0u)) : 0u;
        }
        x0 = st;
        ident = false;
    }
    // The state entering this lane when s_tile enters the tile: the exit of
    // the nearest lower lane whose map is constant, else s_tile (only
    // identity lanes before it).  One ballot and one shuffle; every lane of
    // the warp calls it.
    static __device__ __forceinline__ u32 enter_state(u32 cmask, u32 x0, u32 s_tile, u32 lane) {
        const u32 below = cmask & ((1u << lane) - 1u);
        const u32 src = below ? 31u - (u32)__clz(below) : 0u;
        const u32 xk = __shfl_sync(0xffffffffu, x0, src);
        return below ? xk : s_tile;
    }
    // Bytes of an all-inside lane entered in state s (lit/esc: its literal
    // and escape-code slots).
    static __device__ __forceinline__ u32 fsst_lane_bytes(const R& r, u32 E, u32 s) {
        u32 lit, esc;
        fsst_escapes<K>(E, s, lit, esc);
        return fsst_bytes(r, ~(lit | esc) & full_mask(), lit);
    }
    // Bytes of an edge lane (some slots outside the column) entered in state s.
    static __device__ __forceinline__ u32 fsst_edge_bytes(const R& r, u32 s) {
        u32 n = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool v = (r.valid >> k) & 1u;
            const bool is255 = code_at<CODEC, K>(r, k) == 255u;
            n += v ? (s ? 1u : (is255 ? 0u : len_at<CODEC, K>(r, k))) : 0u;
            s = v ? (s ? 0u : (is255 ? 1u : 0u)) : 0u;
        }
        return n;
    }

    // The warp tile's scan element; every lane of the warp calls it.  OnPair:
    // the tile's byte count (the same for both entry states; corrupt codes
    // set ERRB_CORRUPT).  FSST-8: for each escape state entering the tile,
    // the bytes it produces and the state after it.
    static __device__ __forceinline__ TElem tile_element(const R& r, u32 lane, u32& err) {
        const bool allv = (r.valid == full_mask());
        if (!FSST) {
            u32 sum = 0;
            if (allv) {
                bool zero = false;
#pragma unroll
                for (int j = 0; j < K / 4; ++j) {
                    sum += byte_sum(r.L[j]);
                    zero |= has_zero_byte(r.L[j]);
                }
                if (zero) err |= ERRB_CORRUPT;
            } else {
#pragma unroll
                for (int j = 0; j < K / 4; ++j) {
                    const u32 vm = bytes_of4(r.valid >> (4 * j));
                    sum += byte_sum(r.L[j] & vm);
                    if (__vcmpeq4(r.L[j], 0u) & vm) err |= ERRB_CORRUPT;
                }
            }
            sum = __reduce_add_sync(0xffffffffu, sum);
            return TElem{sum, sum, 2u};
        }
        const u32 E = allv ? ff_mask(r) : 0u;
        u32 x0;
        bool ident;
        lane_state(r, allv, E, x0, ident);
        // states entering this lane when the tile is entered with 0 and with 1:
        // they differ only for lanes that only identity lanes precede
        const u32 below = __ballot_sync(0xffffffffu, !ident) & ((1u << lane) - 1u);
        const u32 xk = __shfl_sync(0xffffffffu, x0, below ? 31u - (u32)__clz(below) : 0u);
        const u32 s0 = below ? xk : 0u, s1 = below ? xk : 1u;
        u32 b0 = allv ? fsst_lane_bytes(r, E, s0) : fsst_edge_bytes(r, s0);
        u32 b1 = b0;
        if (__any_sync(0xffffffffu, s0 != s1) && s0 != s1) b1 = allv ? fsst_lane_bytes(r, E, s1) : fsst_edge_bytes(r, s1);
        b0 = __reduce_add_sync(0xffffffffu, b0);
        b1 = __reduce_add_sync(0xffffffffu, b1);
        const u32 e = (ident ? s0 : x0) | ((ident ? s1 : x0) << 1);
        return TElem{b0, b1, __shfl_sync(0xffffffffu, e, 31)};
    }

    // Token of `code` (zero padded to 16 bytes), from the table staged in
    // shared memory (DSMEM) or through L1.  OnPair: the whole 16-byte entry
    // (W = 16) or the low plane and, for longer tokens, the high plane
    // (W = 8).  FSST: 8-byte entries.
    static __device__ __forceinline__ uint4 token(const DecodeParams& p, const uint4* dict, u32 code, u32 len) {
        if (TOK8) {
            const uint2 d = DSMEM ? reinterpret_cast<const uint2*>(dict)[code]
                                  : __ldg(reinterpret_cast<const uint2*>(p.dict.table) + code);
            return make_uint4(d.x, d.y, 0u, 0u);
        }
        // W = 16: whole 16-byte entries, one load (staged as the table is laid out)
        if (W == 16) return DSMEM ? dict[code] : __ldg(reinterpret_cast<const uint4*>(p.dict.table) + code);
        const uint2* lo = DSMEM ? reinterpret_cast<const uint2*>(dict) : reinterpret_cast<const uint2*>(p.dict.planes);
        const uint2 a = DSMEM ? lo[code] : __ldg(lo + code);
        uint2 b = make_uint2(0u, 0u);
        // split read: the high plane only for longer tokens (W = 8), always for W = 16
        if (W == 16 || len > 8u) b = DSMEM ? lo[kTable + code] : __ldg(lo + kTable + code);
        return make_uint4(a.x, a.y, b.x, b.y);
    }

    // Token of an FSST slot, zero past its length.  FSST-8: a literal's byte,
    // else the symbol; a slot that yields no byte is an escape or a corrupt
    // code, whose table entries (255, and those past the dictionary) are all
    // zero, so in a lane whose slots are all inside the column only literals
    // need a select.
    static __device__ __forceinline__ uint2 token8(const DecodeParams& p, const uint4* dict, u32 code, bool lit) {
        const uint2* tab = DSMEM ? reinterpret_cast<const uint2*>(dict) : reinterpret_cast<const uint2*>(p.dict.table);
        if (LITTAB) return tab[code | (lit ? 256u : 0u)];
        const uint2 d = DSMEM ? tab[code] : __ldg(tab + code);
        return (FSST && lit) ? make_uint2(code, 0u) : d;
    }

    // Append the lane's K tokens (cw: the bytes of each slot, `lit` its
    // literals) in two independent runs, slots 0 .. K/2 - 1 by w0 and the
    // others by w1: an append waits for the one before it in its run, so two
    // runs hide half of that wait.  The next four tokens are read while four
    // are appended: the compiler cannot move dictionary reads over the
    // staging stores itself.
    template <bool ALLV>
    static __device__ __forceinline__ void assemble(const DecodeParams& p, const uint4* dict, const R& r,
                                                    const u32 (&cw)[K / 4], u32 lit, StageWriter& w0,
                                                    StageWriter& w1) {
        typedef typename std::conditional<TOK8, uint2, uint4>::type Tok;
        Tok tok[2][4];
        // step g: slots 2g, 2g + 1 and K/2 + 2g, K/2 + 2g + 1
        auto slot = [](int g, int h) { return 2 * g + (h & 1) + (h >> 1) * (K / 2); };
        auto bytes = [&](int k) { return (cw[k >> 2] >> (8 * (k & 3))) & 0xffu; };
        auto load = [&](int g) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int k = slot(g, h);
                const u32 code = code_at<CODEC, K>(r, k);
                Tok& t = tok[g & 1][h];
                if constexpr (TOK8) t = token8(p, dict, code, (lit >> k) & 1u);
                else t = token(p, dict, code, len_at<CODEC, K>(r, k));
                if (!ALLV && bytes(k) == 0u) t = Tok{};
            }
        };
        load(0);
#pragma unroll
        for (int g = 0; g < K / 4; ++g) {
            if (g + 1 < K / 4) load(g + 1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (TOK8) {
                    w0.put8(tok[g & 1][h], bytes(slot(g, h)));
                    w1.put8(tok[g & 1][h + 2], bytes(slot(g, h + 2)));
                } else {
                    w0.put(tok[g & 1][h], bytes(slot(g, h)));
                    w1.put(tok[g & 1][h + 2], bytes(slot(g, h + 2)));
                }
            }
        }
    }

    // Write the staged bytes [off0, nb) to the 16-byte chunks from g on:
    // the whole chunks by one bulk copy (left in flight: stage_free() before
    // the area is written again), the bytes of the two edge chunks, shared
    // with the neighbouring tiles, one per lane.  Every lane has fenced its
    // stores for the copy engine.
    static __device__ __forceinline__ void flush(const uint4* stage, uint4* g, u32 off0, u32 nb, u32 lane) {
        const u32 first = off0 ? 1u : 0u, last = nb >> 4;
        if (lane == 0u && last > first) bulk_s2g(g + first, stage + first, (last - first) * 16u);
        const u32 b = lane & 15u, e = nb & 15u;
        const bool head = lane < 16u;
        const bool w = head ? (off0 != 0u && b >= off0 && b < nb) : (b < e && !(last == 0u && off0 != 0u));
        if (w) {
            const u32 i = head ? b : last * 16u + b;
            reinterpret_cast<uint8_t*>(g)[i] = reinterpret_cast<const uint8_t*>(stage)[i];
        }
    }
    // The copy engine has read what the last flush() gave it (every lane of
    // the warp calls this).
    static __device__ __forceinline__ void stage_free(u32 lane) {
        if (lane == 0u) bulk_wait_read();
        __syncwarp();
    }

    // Stage the dictionary and the token lengths in shared memory (every
    // thread of the block; the caller synchronises).  FSST: the 8-byte
    // entries, for FSST-8 with the literals after them (LITTAB); OnPair read
    // whole (W = 16): the 16-byte entries; OnPair split read (W = 8): the two
    // planes (entry e's bytes 0..7 at low-plane word e, bytes 8..15 at
    // high-plane word e).
    static __device__ __forceinline__ void stage_dict(const DecodeParams& p, uint4* s_dict, uint8_t* s_lens,
                                                      int nthreads) {
        if (!LSMEM) return;
        if (LITTAB) {
            const uint2* tab = reinterpret_cast<const uint2*>(p.dict.table);
            for (int i = threadIdx.x; i < 512; i += nthreads)
                reinterpret_cast<uint2*>(s_dict)[i] = i < 256 ? __ldg(tab + i) : make_uint2((u32)i - 256u, 0u);
        } else if (DSMEM) {
            const uint4* src = reinterpret_cast<const uint4*>((TOK8 || W == 16) ? p.dict.table : p.dict.planes);
            for (int i = threadIdx.x; i < DICT_BYTES / 16; i += nthreads) s_dict[i] = __ldg(src + i);
        }
        const uint4* lsrc = reinterpret_cast<const uint4*>(p.dict.lens);
        for (int i = threadIdx.x; i < LENS_BYTES / 16; i += nthreads) reinterpret_cast<uint4*>(s_lens)[i] = __ldg(lsrc + i);
    }

    // The same staging by the bulk-copy engine where the staged layout is the
    // stored one (no planes, no literals): thread 0 issues the two
    // copies (cp.async.bulk, completion counted on one mbarrier) and every
    // thread waits for them, bounded.  Falls back to the loads above for tables
    // that are not 16-byte aligned, and where a wait gave up (after one more
    // for the copies in flight): then the result is ERRB_TIMEOUT, else 0.
    // Every thread of the block calls it; returns synchronised.
    static constexpr bool BULK_STAGE = LSMEM && !LITTAB && (!DSMEM || TOK8 || W == 16);
    static __device__ __forceinline__ u32 stage_dict_bulk(const DecodeParams& p, uint4* s_dict, uint8_t* s_lens,
                                                          u64* bar, int nthreads) {
        const bool aligned =
            ((reinterpret_cast<uintptr_t>(p.dict.table) | reinterpret_cast<uintptr_t>(p.dict.lens)) & 15u) == 0u;
        if (!aligned) {
            stage_dict(p, s_dict, s_lens, nthreads);
            __syncthreads();
            return 0u;
        }
        if (threadIdx.x == 0) {
            mbar_init(bar, FP_COPY_ARRIVALS);
            mbar_init_fence();
            bulk_tables(p, s_dict, s_lens, bar);
        }
        __syncthreads();   // the barrier is initialised before anyone waits on it
        return wait_tables(p, s_dict, s_lens, bar, 0u, nthreads);
    }
    static __device__ __forceinline__ u32 wait_tables(const DecodeParams& p, uint4* s_dict, uint8_t* s_lens, u64* bar,
                                                      u32 phase, int nthreads) {
        if (!__syncthreads_or(!mbar_wait(bar, phase, p.ws))) return 0u;
        mbar_wait(bar, phase, p.ws);
        stage_dict(p, s_dict, s_lens, nthreads);
        __syncthreads();
        return ERRB_TIMEOUT;
    }
    // Issue the two copies (one thread; `bar` is initialised).
    static __device__ __forceinline__ void bulk_tables(const DecodeParams& p, uint4* s_dict, uint8_t* s_lens, u64* bar) {
        mbar_expect_tx(bar, (u32)(DICT_BYTES + LENS_BYTES));
        if (DSMEM) bulk_g2s(s_dict, p.dict.table, (u32)DICT_BYTES, bar);
        bulk_g2s(s_lens, p.dict.lens, (u32)LENS_BYTES, bar);
        mbar_arrive(bar);
    }

    // Byte count of an escape-free lane whose K slots all lie inside the
    // column, straight from its code words (constant bit positions): one
    // extract, one length load and one add per code; a code without a token
    // (length 0) raises ERRB_CORRUPT.
    // Packed codes: `o` and `b` as in unpack_packed().
    static __device__ __forceinline__ u32 lane_length_sum(const u32 (&wv)[LANE_WORDS], const uint8_t* lens,
                                                          u32& err, u32 o = 0, u32 b = 0) {
        static_assert(!FSST, "escape-free codecs");
        constexpr u32 MASK = (1u << WBITS) - 1u;
        u32 sum = 0, mn = 0xffu;
        R r;
        if constexpr (PACKED) unpack_packed(wv, o, b, r);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            u32 code;
            if constexpr (PACKED) {
                code = code_at<CODEC, K>(r, k);
            } else {
                const int bit = k * WBITS, w = bit >> 5, sh = bit & 31;
                code = (sh + WBITS <= 32) ? ((wv[w] >> sh) & MASK) : (__funnelshift_r(wv[w], wv[w + 1], sh) & MASK);
            }
            const u32 L = LSMEM ? (u32)lens[code] : (u32)__ldg(lens + code);
            sum += L;
            mn = min(mn, L);
        }
        if (mn == 0u) err |= ERRB_CORRUPT;
        return sum;
    }

    static __device__ __forceinline__ u64 lane_q0(const Extent& x, u64 t) {
        return (x.first_tile + t) * (u64)TILE + (u64)(threadIdx.x & 31u) * K;
    }

    // Inputs of a warp tile fetched ahead of its decode: its codes (`in` is
    // false for a lane whose codes run past the code buffer: guarded loads
    // instead; with BULK_CODES for a whole tile), the tile's scanned offset
    // and its string boundaries [lo, hi) (as stored: clamped where they are
    // used, so that nothing waits for the loads here).
    struct Fetch {
        u32 wv[BULK_CODES ? 1 : LANE_WORDS];
        bool in;
        u64 ex;
        u32 lo, hi;
    };
    // The warp's mbarrier for those copies and the phase of the next one, 2
    // more once this lane's wait has given up: from then on it takes its codes
    // by guarded loads (and lane 0 issues no copies).  Each lane goes by its own
    // wait: a vote of the warp cost 0.3-1 % of a call.
    struct CodeBar {
        u64* bar;
        u32 phase;
        __device__ __forceinline__ bool usable() const { return phase < 2u; }
        __device__ __forceinline__ bool wait(WsHeader* ws) {
            const bool ok = mbar_wait(bar, phase, ws);
            phase = ok ? phase ^ 1u : phase | 2u;
            return ok;
        }
        // Before the area is used for something else, or the block ends: once
        // more for a copy that was given up.
        __device__ __forceinline__ void drain(WsHeader* ws) const {
            if (!usable()) mbar_wait(bar, phase & 1u, ws);
        }
        // Every lane of the warp calls it, before the first fetch().
        __device__ __forceinline__ void init(u64* b) {
            bar = b;
            phase = 0u;
            if ((threadIdx.x & 31u) == 0u) {
                mbar_init(bar, FP_COPY_ARRIVALS);
                mbar_init_fence();
            }
            __syncwarp();
        }
    };
    // Rounds of 32 boundaries whose code_offsets are in flight together.
    static constexpr int PB = K / 8;

    // Issue the loads of tile t (every lane of the warp, the tile before it
    // read from area.codes): its codes, and what the passes before the decode
    // made.  AHEAD: the codes before the kernel's wait (past L1).
    template <bool AHEAD = false>
    static __device__ __forceinline__ void fetch_codes(const DecodeParams& p, const Extent& x, u64 t, Area& area,
                                                       const CodeBar& cb, Fetch& f) {
        if constexpr (BULK_CODES) {
            const u32 tb = tile_bytes(p);
            const u64 b0 = (x.first_tile + t) * tb;   // a multiple of 16, as tb is
            f.in = b0 + tb <= p.codes_bytes && cb.usable();
            if (f.in && (threadIdx.x & 31u) == 0u) {
                mbar_expect_tx(cb.bar, tb);
                bulk_g2s(area.codes, p.codes + b0, tb, cb.bar);
                mbar_arrive(cb.bar);
            }
        } else {
            f.in = load_fast<AHEAD>(p, lane_q0(x, t), f.wv);
        }
    }
    // The launches (or phases) before this one wrote these while it was
    // already running.
    static __device__ __forceinline__ void fetch_scanned(const u64* ex, const u32* first, u64 t, Fetch& f) {
        f.ex = in_order_l2(ex + t);
        f.lo = in_order_l2(first + t);
        f.hi = in_order_l2(first + t + 1);
    }
    static __device__ __forceinline__ void fetch(const DecodeParams& p, const Extent& x, const u64* ex, u64 t,
                                                 Area& area, const CodeBar& cb, Fetch& f) {
        fetch_codes(p, x, t, area, cb, f);
        fetch_scanned(ex, p.first, t, f);
    }

    // The first boundaries of a tile: positions in flight while it is
    // assembled.
    struct Strings {
        u32 first, left;   // the lane's first boundary, boundaries from it to the tile's end
        u32 pos[PB];
    };
    // Boundaries [lo, hi), clamped to the column's; issues the loads (in
    // order: they stay ahead of the assembly that hides them, and off the
    // read-only path, since the one-cluster decode may have started before
    // the kernel that writes the column ended).
    static __device__ __forceinline__ void strings_begin(const DecodeParams& p, u32 lo, u32 hi, Strings& sb) {
        const u32 nb_col = p.n_strings + 1u;
        const u32 lane = threadIdx.x & 31u;
        lo = min(lo, nb_col);
        hi = min(hi, nb_col);
        sb.first = lo + lane;   // (may pass 2^32 where nothing is left)
        sb.left = hi > lo && hi - lo > lane ? hi - lo - lane : 0u;
#pragma unroll
        for (int j = 0; j < PB; ++j) sb.pos[j] = 32u * j < sb.left ? in_order(p.code_offsets + sb.first + 32u * j) : 0u;
    }

    // Assemble warp tile t of column (p, x) from its codes and token lengths
    // (r): the bytes, then the offsets of the strings whose boundaries it
    // owns.  `ex` is its output offset and entering escape state; returns
    // the same for the tile after it.
    static __device__ __forceinline__ u64 assemble_tile(const DecodeParams& p, const Extent& x, u64 t, R& r, u64 ex,
                                                        Strings& sb, const uint4* dict, Area& area, u32& err) {
        const u32 lane = threadIdx.x & 31u;
        const u64 tile_start = (x.first_tile + t) * (u64)TILE;
        const bool allv = (r.valid == full_mask());
        const u64 tile_excl = ex & 0x7fffffffffffffffull;
        const u32 s_tile = FSST ? (u32)(ex >> 63) : 0u;

        // bytes of each slot (cw, one byte per slot) and of the lane; FSST-8:
        // the lane's entering escape state first, then its literals
        u32 cw[K / 4];
        u32 produced = 0;
        u32 lit = 0, exit_state = 0;
        if (!FSST) {
#pragma unroll
            for (int j = 0; j < K / 4; ++j) {
                // a code without a token (length 0) is corrupt input
                if (allv) {
                    cw[j] = r.L[j];
                    if (has_zero_byte(cw[j])) err |= ERRB_CORRUPT;
                } else {
                    const u32 vm = bytes_of4(r.valid >> (4 * j));
                    cw[j] = r.L[j] & vm;
                    if (__vcmpeq4(r.L[j], 0u) & vm) err |= ERRB_CORRUPT;
                }
                produced += byte_sum(cw[j]);
            }
        } else {
            const u32 E = allv ? ff_mask(r) : 0u;
            u32 x0;
            bool ident;
            lane_state(r, allv, E, x0, ident);
            const u32 s_in = enter_state(__ballot_sync(0xffffffffu, !ident), x0, s_tile, lane);
            exit_state = ident ? s_in : x0;
            if (allv) {
                u32 esc;
                fsst_escapes<K>(E, s_in, lit, esc);
                const u32 code_slots = ~(lit | esc) & full_mask();
#pragma unroll
                for (int j = 0; j < K / 4; ++j) {
                    const u32 code_ff = bytes_of4(code_slots >> (4 * j));
                    cw[j] = (r.L[j] & code_ff) | ones_of4(lit >> (4 * j));
                    if (has_zero_byte(r.L[j] | ~code_ff)) err |= ERRB_CORRUPT;
                    produced += byte_sum(cw[j]);
                }
            } else {
                u32 st = s_in;
#pragma unroll
                for (int j = 0; j < K / 4; ++j) cw[j] = 0u;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const bool v = (r.valid >> k) & 1u;
                    const u32 bt = code_at<CODEC, K>(r, k);
                    lit |= (st & 1u) << k;
                    u32 a = 0;
                    if (v) {
                        if (st) { a = 1u; st = 0u; }
                        else if (bt == 255u) { st = 1u; }
                        else {
                            a = len_at<CODEC, K>(r, k);
                            if (a == 0u) err |= ERRB_CORRUPT;
                        }
                    } else {
                        st = 0u;
                    }
                    cw[k >> 2] |= a << ((k & 3) * 8);
                    produced += a;
                }
            }
            area.lit_mask[lane] = lit;
        }

        // the lane's output offset in the tile: one warp scan of byte counts
        u32 inc = produced;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (u32)d) inc += y;
        }
        const u32 thr = inc - produced;
        const u32 tot = __shfl_sync(0xffffffffu, inc, 31);
        const u64 tile_incl = tile_excl + tot;
        const u32 tile_out_state = FSST ? __shfl_sync(0xffffffffu, exit_state, 31) : 0u;
        const bool last_tile = (t == x.n_tiles - 1);
        const bool skip = p.size_only || tile_incl > p.capacity;

        // per-slot bytes and the offsets of every fourth slot, for the string offsets
        u32 half = 0;   // bytes of the lane's first K/2 slots
        {
            u32 o = thr;
#pragma unroll
            for (int j = 0; j < K / 4; ++j) {
                if (j == K / 8) half = o - thr;
                area.contrib[j][lane] = cw[j];
                area.pre[j][lane] = o;
                o += byte_sum(cw[j]);
            }
        }
        // Assembly in the warp's staging area, then whole-chunk stores.  A tile
        // of more than CAP bytes takes rounds over consecutive lanes (a lane
        // has at most 256 bytes).
        u32* const stage = reinterpret_cast<u32*>(area.stage);
        u32 rb = 0;
        while (!skip && rb < tot) {
            u32 end = tot;
            if (tot - rb > (u32)(CAP - 16)) end = __reduce_max_sync(0xffffffffu, inc <= rb + (u32)(CAP - 16) ? inc : rb);
            const bool in = thr >= rb && inc <= end;
            const u64 G = tile_excl + rb;
            const u32 off0 = (u32)(G & 15u), nb = off0 + (end - rb);
            stage_free(lane);
            StageWriter w0, w1;
            w0.begin(stage, in ? off0 + (thr - rb) : 0u);
            w1.begin(stage, in ? off0 + (thr + half - rb) : 0u);
            if (in) {
                if (allv) assemble<true>(p, dict, r, cw, lit, w0, w1);
                else assemble<false>(p, dict, r, cw, lit, w0, w1);
            }
            // the round's last word is completed by no lane: its bytes are only added
            if (lane == 0u && (nb & 7u)) reinterpret_cast<u64*>(stage)[nb >> 3] = 0ull;
            __syncwarp();
            if (in) {
                w0.finish();
                w1.finish();
            }
            async_fence();
            __syncwarp();
            flush(area.stage, reinterpret_cast<uint4*>(p.out) + (G >> 4), off0, nb, lane);
            rb = end;
        }
        __syncwarp();

        u32 first = sb.first, left = sb.left;
        // offsets of the strings whose boundaries the tile owns
        while (left) {
#pragma unroll
            for (int j = 0; j < PB; ++j) {
                if (32u * j >= left) break;
                const u32 i = first + 32u * j;
                u32 rel = 0;
                u32 st = 0;
                const u64 at = (u64)sb.pos[j] - tile_start;   // wraps for positions before the tile
                if (at < (u64)TILE) {
                    const u32 sidx = (u32)at, sl = sidx / K, k = sidx % K;
                    // offset of slot k's group of four, then the group's slots before k
                    rel = area.pre[k >> 2][sl] + byte_sum(area.contrib[k >> 2][sl] & ((1u << (8u * (k & 3u))) - 1u));
                    if (FSST) st = (area.lit_mask[sl] >> k) & 1u;
                } else if (at == (u64)TILE) {
                    rel = tot;
                    st = tile_out_state;
                    if (!last_tile) err |= ERRB_CORRUPT;
                } else {
                    err |= ERRB_CORRUPT;
                }
                if (st) err |= ERRB_CORRUPT;   // a string would start on a literal
                if (!p.size_only) __stcs(p.out_offsets + i, (u32)tile_excl + rel);
            }
            if (left <= 32u * PB) break;
            first += 32u * PB;
            left -= 32u * PB;
#pragma unroll
            for (int j = 0; j < PB; ++j) sb.pos[j] = 32u * j < left ? in_order(p.code_offsets + first + 32u * j) : 0u;
        }
        __syncwarp();   // the areas are reused by the next tile
        return tile_incl | ((u64)tile_out_state << 63);
    }

    // Decode warp tile t of column (p, x) from its fetched inputs: offset
    // and entering escape state (from the tile scan), code words, string
    // boundaries.  `area` is the warp's scratch.  `ex_tiles` holds the
    // column's scanned tile offsets (f.ex = ex_tiles[t]): the tile's own
    // byte total, recomputed here, must bring it to ex_tiles[t + 1], else
    // ERRB_MISMATCH is raised (a self-check of the two passes, one load
    // per tile).
    // `next` issues the fetch of the warp's next tile (it is called once
    // area.codes is free).
    template <class Next>
    static __device__ __forceinline__ void decode_tile(const DecodeParams& p, const Extent& x, u64 t, const Fetch& f,
                                                       const u64* ex_tiles, const uint4* dict, const uint8_t* lens,
                                                       Area& area, CodeBar& cb, u32& err, Next&& next) {
        const u32 lane = threadIdx.x & 31u;
        const u64 q0 = lane_q0(x, t);
        const u64 ex = f.ex;
        // low word of the next tile's offset (lane 0 checks), in flight during the tile
        const bool chk = lane == 0u && t + 1 < x.n_tiles;
        const u32 ex_next = chk ? in_order_l2(reinterpret_cast<const u32*>(ex_tiles + t + 1)) : 0u;
        Strings sb;
        strings_begin(p, f.lo, f.hi, sb);
        R r;
        if constexpr (BULK_CODES) {
            u32 wv[LANE_WORDS];
            bool in = f.in;
            if (in) {
                in = cb.wait(p.ws);
                if (in) load_staged(p, area.codes, lane, wv);
                else err |= ERRB_TIMEOUT;
            }
            __syncwarp();   // the codes have left the area
            next();
            finish_load(p, x, q0, wv, in, lens, r);
        } else {
            next();
            finish_load(p, x, q0, f.wv, f.in, lens, r);
        }
        const u64 next_ex = assemble_tile(p, x, t, r, ex, sb, dict, area, err);
        if (chk && ex_next != (u32)next_ex) err |= ERRB_MISMATCH;
    }

    // Decode the tiles t0, t0 + step, ... of the column (every lane of the
    // warp).  Software pipeline: while tile t decodes, the inputs of
    // t + step are in flight.
    static __device__ __forceinline__ void decode_tiles(const DecodeParams& p, const Extent& x, const u64* ex, u64 t,
                                                        u64 step, const uint4* dict, const uint8_t* lens,
                                                        Area& area, u64* bar, u32& err) {
        if (t >= x.n_tiles) {
            grid_wait();
            return;
        }
        CodeBar cb;
        cb.init(bar);
        Fetch cur;
        fetch_codes<true>(p, x, t, area, cb, cur);
        grid_wait();   // the launch before (none before a cooperative launch's phases)
        fetch_scanned(ex, p.first, t, cur);
        for (; t < x.n_tiles; t += step) {
            Fetch nxt;
            decode_tile(p, x, t, cur, ex, dict, lens, area, cb, err, [&] {
                if (t + step >= x.n_tiles) return;
                fetch_codes(p, x, t + step, area, cb, nxt);
                fetch_scanned(ex, p.first, t + step, nxt);
            });
            cur = nxt;
        }
        stage_free(threadIdx.x & 31u);   // shared memory outlives the copies from it
        cb.drain(p.ws);                  // and the copies to it
    }
};

// ---------------------------------------------------------------------------
// Index pass by warps: warp w of nw takes chunks of 256 boundaries, eight
// consecutive ones to a lane (two 16-byte loads), the next chunk's loads in
// flight.  Results and checks as index_groups(), which takes what is out of
// the ordinary here: the first and last chunk, boundaries that decrease or
// reach the column's ends.  About 15 instructions per 32 boundaries against
// 60 with a boundary to a lane.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void index_by_warps(const DecodeParams& p, const Extent& x, u32 tile_log2, u32 w, u32 nw,
                                               u32* first) {
    constexpr u32 CH = 32 * kIdxGroup;
    static_assert(kIdxGroup == 8, "two 16-byte loads");
    const u32 lane = threadIdx.x & 31u;
    const u32* a = p.code_offsets;
    const u32 n = p.n_strings;             // the last boundary
    const u32 chunks = n / CH + 1u;        // boundaries 0 .. n
    const bool aligned = (reinterpret_cast<uintptr_t>(a) & 15u) == 0u;
    const u32 cb = (u32)x.c_begin, ce = (u32)x.c_end;
    u32* const f = first - x.first_tile;   // indexed by slot position >> tile_log2
    u32 err = x.bad ? ERRB_CORRUPT : 0u;
    u32 v[kIdxGroup], before = 0u;
    auto load = [&](u32 c) {
        const u32 i0 = c * CH + lane * kIdxGroup;
        if (aligned && c + 1u < chunks) {
            const uint4 lo = in_order4(a + i0), hi = in_order4(a + i0 + 4);
            v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w;
            v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
        } else {
#pragma unroll
            for (u32 k = 0; k < kIdxGroup; ++k) v[k] = in_order(a + (n - i0 >= k && i0 <= n ? i0 + k : n));
        }
        before = c > 0u ? in_order(a + c * CH - 1u) : 0u;
    };
    if (w < chunks) load(w);
    for (u32 c = w; c < chunks; c += nw) {
        u32 cur[kIdxGroup];
#pragma unroll
        for (int k = 0; k < kIdxGroup; ++k) cur[k] = v[k];
        u32 prev = __shfl_up_sync(0xffffffffu, cur[kIdxGroup - 1], 1);
        if (lane == 0u) prev = before;
        if (chunks - c > nw) load(c + nw);
        const u32 i0 = c * CH + lane * kIdxGroup;
        bool plain = prev >= cb && cur[kIdxGroup - 1] < ce && prev <= cur[0];
#pragma unroll
        for (int k = 1; k < kIdxGroup; ++k) plain &= cur[k - 1] <= cur[k];
        if (c > 0u && c + 1u < chunks && __all_sync(0xffffffffu, plain)) {
            u32 t = prev >> tile_log2;
#pragma unroll
            for (int k = 0; k < kIdxGroup; ++k) {
                const u32 u = cur[k] >> tile_log2;
                for (; t < u; ++t) f[t + 1u] = i0 + k;   // tiles that begin between the two boundaries
            }
        } else {
#pragma unroll
            for (u32 k = 0; k < kIdxGroup; ++k) {
                if (i0 <= n && n - i0 >= k) index_one(x, tile_log2, (u64)n + 1, (u64)i0 + k, cur[k], prev, first, err);
                prev = cur[k];
            }
        }
    }
    if (err) atomicOr(p.err_word, err);
}

// The index pass alone (a stored table replaces the other passes).
__global__ void __launch_bounds__(256) index_only_kernel(const DecodeParams p, u32 tile) {
    index_by_warps(p, column_extent(p, tile), (u32)(__ffs((int)tile) - 1), blockIdx.x * 8u + (threadIdx.x >> 5),
                   gridDim.x * 8u, const_cast<u32*>(p.first));
}

// ---------------------------------------------------------------------------
// Pass 1: warp-tile elements.
// ---------------------------------------------------------------------------
// Blocks [0, index_blocks) run the index pass (first string of every warp
// tile), the others the reduce: the two overlap in one launch.  Large FSST-8
// and OnPair-16 columns take length_reduce_kernel (fp_reduce.cuh) instead.
// Reduce shape per codec, from an A/B on GB300 (10M-16M strings): rounds of
// U tiles in flight, MINB blocks of 256 threads per SM.  Per call of that
// A/B, OnPair-12: 2 x 4 725 us, 2 x 3 733; FSST-8, whose 32-slot lanes spill
// at fewer than 128 registers: 2 x 2 1.2 % faster; FSST-12: 1 x 4 1.5 %.
template <int CODEC, int K>
struct ReduceShape {
    static constexpr int U = CODEC == FP_FSST12 ? 1 : 2;
    static constexpr int MINB = (CODEC == FP_FSST8 && K == 32) ? 2 : 4;
};

template <int CODEC, int K, bool DSMEM, bool PACKED = false>
__global__ void __launch_bounds__(256, ReduceShape<CODEC, K>::MINB) reduce_kernel(const DecodeParams pp,
                                                                                  u64* agg, u32 index_blocks) {
    typedef WarpCore<CODEC, K, DSMEM, WarpCore<CODEC, K, DSMEM>::TOK8 ? 8 : 16, PACKED> C;
    __shared__ __align__(16) uint8_t s_lens[DSMEM ? C::LENS_BYTES : 16];
    if (DSMEM && blockIdx.x >= index_blocks) {
        // the dictionary is older than any launch this one may overlap
        const uint4* src = reinterpret_cast<const uint4*>(pp.dict.lens);
        for (int i = threadIdx.x; i < C::LENS_BYTES / 16; i += blockDim.x) reinterpret_cast<uint4*>(s_lens)[i] = __ldg(src + i);
    }
    grid_wait();      // the launch before: the column may be its output, the workspace its scratch
    DecodeParams p = pp;
    p.codes = after_wait(pp.codes);
    grid_release();   // the next launch may be scheduled as these blocks retire (it waits for their results)
    if (blockIdx.x < index_blocks) {
        index_by_warps(p, column_extent(p, C::TILE), (u32)(__ffs(C::TILE) - 1), blockIdx.x * 8u + (threadIdx.x >> 5),
                       index_blocks * 8u, const_cast<u32*>(p.first));
        return;
    }
    if (DSMEM) __syncthreads();
    const Extent x = column_extent(p, C::TILE);
    const uint8_t* lens = DSMEM ? s_lens : p.dict.lens;
    const u32 lane = threadIdx.x & 31u;
    const u32 rblock = blockIdx.x - index_blocks;
    const u64 warps = (u64)(gridDim.x - index_blocks) * (blockDim.x / 32);
    u32 err = 0;
    // rounds of U tiles; the next round's loads are in flight while this one computes
    constexpr int U = ReduceShape<CODEC, K>::U;
    if constexpr (!C::FSST) {
        // Escape-free codes: tiles [t_lo, t_hi) lie wholly
        // inside the column and the code buffer; their lanes load their code
        // words at a fixed stride and sum their lengths straight from them
        // (32-bit tile indices: fewer than 2^32 tiles).  Edge tiles take the
        // general path.
        const u32 bits = PACKED ? p.packed_bits : (u32)C::WBITS;
        const u32 TB = C::tile_bytes(p);   // the words of its lanes lie within them
        const u32 nt = (u32)x.n_tiles, W = (u32)warps;
        const u64 buf_slots = p.codes_bytes * 8 / bits;
        const u64 end = x.c_end < buf_slots ? x.c_end : buf_slots;
        const u64 lo64 = (x.c_begin + C::TILE - 1) / C::TILE, hi64 = end / C::TILE;
        const u32 t_lo = (u32)(lo64 - x.first_tile);
        const u32 t_hi = hi64 > lo64 ? (u32)(hi64 - x.first_tile) : t_lo;
        // Packed codes are summed 16 to a lane, a tile of 32-slot lanes as two
        // halves: a lane's words are loaded one by one, and 16 codes a lane lie
        // half as far apart, in half the lines a load (FSST-12 at 10 bits, 16M
        // strings: 435 -> 427 us a call).
        typedef WarpCore<CODEC, PACKED ? 16 : K, DSMEM, C::TOK8 ? 8 : 16, PACKED> H;
        constexpr int HALVES = PACKED ? K / 16 : 1;
        static_assert(HALVES * H::LANE_WORDS == C::LANE_WORDS, "the halves' words are the lane's");
        const u32 lane_bit = lane * (PACKED ? 16u : (u32)K) * bits, o = PACKED ? lane_bit & 31u : 0u;
        const uint8_t* base = p.codes + x.first_tile * (u64)TB + (lane_bit - o) / 8;
        auto load = [&](u32 t, u32 (&w)[C::LANE_WORDS]) {
            if constexpr (PACKED) {
#pragma unroll
                for (int h = 0; h < HALVES; ++h)
                    H::load_packed(reinterpret_cast<const u32*>(base + (u64)t * TB + h * (TB / HALVES)),
                                   H::packed_words(bits), w + h * H::LANE_WORDS);
            } else if (C::LANE_BYTES % 16 == 0) {
                const uint4* src = reinterpret_cast<const uint4*>(base + (u64)t * TB);
#pragma unroll
                for (int v = 0; v < C::LANE_WORDS / 4; ++v) {
                    const uint4 a = __ldcs(src + v);
                    w[4 * v] = a.x; w[4 * v + 1] = a.y; w[4 * v + 2] = a.z; w[4 * v + 3] = a.w;
                }
            } else {
                const uint2* src = reinterpret_cast<const uint2*>(base + (u64)t * TB);
#pragma unroll
                for (int v = 0; v < C::LANE_WORDS / 2; ++v) {
                    const uint2 a = __ldcs(src + v);
                    w[2 * v] = a.x;
                    w[2 * v + 1] = a.y;
                }
            }
        };
        u32 t = (u32)rblock * (blockDim.x / 32) + (threadIdx.x >> 5);
        u32 wv[U][C::LANE_WORDS];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u32 tt = t + u * W;
            if (tt >= t_lo && tt < t_hi) load(tt, wv[u]);
        }
        for (; t < nt; t += U * W) {
            u32 nv[U][C::LANE_WORDS];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const u32 tt = t + (U + u) * W;
                if (tt >= t_lo && tt < t_hi) load(tt, nv[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const u32 tt = t + u * W;
                if (tt >= nt) continue;
                if (tt >= t_lo && tt < t_hi) {
                    u32 sum = 0;
#pragma unroll
                    for (int h = 0; h < HALVES; ++h) {
                        u32 hw[H::LANE_WORDS];
#pragma unroll
                        for (int i = 0; i < H::LANE_WORDS; ++i) hw[i] = wv[u][h * H::LANE_WORDS + i];
                        sum += H::lane_length_sum(hw, lens, err, o, bits);
                    }
                    const u32 tot = __reduce_add_sync(0xffffffffu, sum);
                    if (lane == 31) agg[tt] = tot;
                } else {
                    u32 gw[C::LANE_WORDS];
                    const bool fast = C::load_fast(p, C::lane_q0(x, tt), gw);
                    typename C::R r;
                    C::finish_load(p, x, C::lane_q0(x, tt), gw, fast, lens, r);
                    const TElem e = C::tile_element(r, lane, err);
                    if (lane == 31) agg[tt] = wt_pack<false>(e);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < C::LANE_WORDS; ++i) wv[u][i] = nv[u][i];
        }
        if (err) atomicOr(p.err_word, err);
        return;
    }
    u64 t0 = (u64)rblock * (blockDim.x / 32) + (threadIdx.x >> 5);
    u32 wv[U][C::LANE_WORDS];
    bool fast[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const u64 t = t0 + u * warps;
        fast[u] = t < x.n_tiles && C::load_fast(p, C::lane_q0(x, t), wv[u]);
    }
    for (; t0 < x.n_tiles; t0 += U * warps) {
        u32 nv[U][C::LANE_WORDS];
        bool nfast[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u64 t = t0 + (U + u) * warps;
            nfast[u] = t < x.n_tiles && C::load_fast(p, C::lane_q0(x, t), nv[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u64 t = t0 + u * warps;
            if (t < x.n_tiles) {
                typename C::R r;
                C::finish_load(p, x, C::lane_q0(x, t), wv[u], fast[u], lens, r);
                const TElem e = C::tile_element(r, lane, err);
                if (lane == 31) agg[t] = wt_pack<C::FSST>(e);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int i = 0; i < C::LANE_WORDS; ++i) wv[u][i] = nv[u][i];
            fast[u] = nfast[u];
        }
    }
    if (err) atomicOr(p.err_word, err);
}

// ---------------------------------------------------------------------------
// Pass 2: exclusive scan of the warp-tile elements.  Blocks of 256 threads
// take 2,048 consecutive elements by ticket; decoupled look-back across
// blocks.  Writes ex[t] = bytes before warp tile t | entering state << 63.
// ---------------------------------------------------------------------------
constexpr int kScanPerThread = 8;
constexpr int kScanTile = 256 * kScanPerThread;

// Shared state of a tile-scan block.
struct ScanShared {
    Elem wsum[8];
    u64 excl_b;
    u32 excl_s;
    u32 ticket;
};

// Scan block b (of n_blocks) over elements agg[0, n) of one column: writes
// ex[] for its 2,048 elements, publishes its look-back word in status[b]
// (status words of this column only), and at the column's last block its
// decoded size and size errors.  Every thread of the block calls this.
template <bool FSST>
__device__ __forceinline__ void scan_block(const DecodeParams& p, const u64* agg, u64* ex, u64 n, u64 b, u64 n_blocks,
                                           unsigned long long* status, u32 epoch, WsHeader* ws, ScanShared& sh) {
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const u64 pad = FSST ? wt_pack<true>(telem_identity()) : 0ull;
    const u64 i0 = b * kScanTile + (u64)threadIdx.x * kScanPerThread;
    u64 w[kScanPerThread];
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) w[k] = (i0 + k < n) ? agg[i0 + k] : pad;
    // this thread's elements composed, then a block scan of 64-bit elements
    Elem e = elem_identity();
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) e = then<FSST>(e, wt_unpack<FSST>(w[k]));
    Elem inc = e;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        Elem y = shfl_up_e<FSST>(inc, d);
        if (lane < (u32)d) y = elem_identity();
        inc = then<FSST>(y, inc);
    }
    if (lane == 31) sh.wsum[warp] = inc;
    __syncthreads();
    Elem wex = elem_identity(), tot = elem_identity();
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const Elem sv = sh.wsum[v];
        if ((u32)v < warp) wex = then<FSST>(wex, sv);
        tot = then<FSST>(tot, sv);
    }
    Elem lex = shfl_up_e<FSST>(inc, 1);
    if (lane == 0) lex = elem_identity();
    lex = then<FSST>(wex, lex);   // the block's elements before this thread's
    if (warp == 0) {
        // publish the aggregate first, so later blocks need not wait for this look-back
        if (b > 0 && lane == 0) st_volatile(status + b, status_word(kFlagAgg, epoch, agg_payload_wide<FSST>(tot)));
        u64 eb = 0;
        u32 es = 0;
        if (b > 0) lookback<FSST, true>(status, (long long)b, epoch, ws, eb, es);
        if (lane == 0) {
            const u64 ib = eb + ((FSST && es) ? tot.b1 : tot.b0);
            const u32 is = FSST ? ((tot.n >> es) & 1u) : 0u;
            st_volatile(status + b, status_word(kFlagInc, epoch, inc_payload<FSST>(ib, is)));
            sh.excl_b = eb;
            sh.excl_s = es;
            if (b == n_blocks - 1) {
                *p.total_out = ib;
                if (ib > p.capacity && !p.size_only) atomicOr(p.err_word, ERRB_CAPACITY);
                if (ib > 0x7fffffffull) atomicOr(p.err_word, ERRB_OVERFLOW);
            }
        }
    }
    __syncthreads();
    const u64 eb = sh.excl_b;
    const u32 es = sh.excl_s;
    // each element's exclusive offset and entering state
    u64 ob = eb + ((FSST && es) ? lex.b1 : lex.b0);
    u32 os = FSST ? ((lex.n >> es) & 1u) : 0u;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) {
        if (i0 + k < n) ex[i0 + k] = ob | ((u64)os << 63);
        const Elem ek = wt_unpack<FSST>(w[k]);
        ob += (FSST && os) ? ek.b1 : ek.b0;
        os = FSST ? ((ek.n >> os) & 1u) : 0u;
    }
    __syncthreads();   // shared words are rewritten for the next ticket
}

// The launch state the tile scan leaves behind (its tickets, the launch tag of
// the look-back words, the stall settings), renewed by one thread of the
// decode after it: the scan's blocks need not count themselves out.
__device__ __forceinline__ void renew_launch(WsHeader* ws) {
    ws->tile_counter = 0;
    ws->abort = 0;
    ws->spin_limit = 0;
    ws->bar_count = 0;
    const u32 ne = (ws->epoch + 1u) & kEpochMask;
    ws->epoch = ne ? ne : 1u;
}

// Everything that does not depend on the reduce (the first ticket and the
// launch tag, which the call before left, the caller's extent) is fetched,
// past L1, while the reduce still runs: on a small column the scan is a chain
// of global round trips (FSST-8, 30k strings, with all of it and the decode's
// first codes after the wait: 13.2 us a call against 12.3).
template <bool FSST>
__global__ void __launch_bounds__(256, 4) tiles_scan_kernel(const DecodeParams p, u32 tile, const u64* agg, u64* ex,
                                                            unsigned long long* status) {
    __shared__ ScanShared sh;
    WsHeader* ws = p.ws;
    grid_release();   // the decode may start launching (its blocks stage the dictionary, then wait)
    if (p.own_column) grid_wait();
    if (threadIdx.x == 0) sh.ticket = atomicAdd(&ws->tile_counter, 1u);
    const u32 epoch = *(volatile u32*)&ws->epoch;
    const u64 n = column_extent<true>(p, tile).n_tiles;
    const u64 n_blocks = (n + kScanTile - 1) / kScanTile;
    grid_wait();      // the reduce's elements
    for (;;) {
        __syncthreads();
        const u64 b = sh.ticket;
        if (b >= n_blocks) break;
        scan_block<FSST>(p, agg, ex, n, b, n_blocks, status, epoch, ws, sh);
        // with a block per scan block the first tickets cover them all: no
        // second ticket (one atomic round trip less at the end of the scan)
        if ((u64)gridDim.x >= n_blocks) break;
        if (threadIdx.x == 0) sh.ticket = atomicAdd(&ws->tile_counter, 1u);
    }
}

// ---------------------------------------------------------------------------
// Pass 3: every warp decodes warp tiles on its own (grid-stride order).
// ---------------------------------------------------------------------------
template <int CODEC, int K, bool DSMEM, int NW, int MINB, int W = WarpCore<CODEC, K, DSMEM>::TOK8 ? 8 : 16,
          bool PACKED = false, bool LSMEM = DSMEM, bool RENEW = true>
__global__ void __launch_bounds__(NW * 32, MINB) warp_decode_kernel(const DecodeParams p, const u64* ex) {
    typedef WarpCore<CODEC, K, DSMEM, W, PACKED, LSMEM> C;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint4* s_dict = reinterpret_cast<uint4*>(smem_raw);
    uint8_t* s_lens = smem_raw + C::DICT_BYTES;
    typename C::Area* areas = reinterpret_cast<typename C::Area*>(smem_raw + C::STAGED_BYTES);
    __shared__ __align__(8) u64 s_bar;
    __shared__ __align__(8) u64 s_code_bar[NW];
    u32 err = 0;
    if (C::BULK_STAGE) {
        err = C::stage_dict_bulk(p, s_dict, s_lens, &s_bar, NW * 32);
    } else if (LSMEM) {
        C::stage_dict(p, s_dict, s_lens, NW * 32);
        __syncthreads();
    }
    if (p.own_column) grid_wait();
    const Extent x = column_extent<true>(p, C::TILE);
    const uint8_t* lens = LSMEM ? s_lens : p.dict.lens;
    // decode_tiles() fetches the first tile's codes, then waits for the tile
    // scan's offsets: staging and fetch overlap the scan
    C::decode_tiles(p, x, ex, (u64)blockIdx.x * NW + (threadIdx.x >> 5), (u64)gridDim.x * NW, s_dict, lens,
                    areas[threadIdx.x >> 5], s_code_bar + (threadIdx.x >> 5), err);
    if (RENEW && blockIdx.x == 0 && threadIdx.x == 0) renew_launch(p.ws);
    if (err) atomicOr(p.err_word, err);
}


// ---------------------------------------------------------------------------
// Small columns in one cooperative launch: the three passes above as phases
// of one kernel, separated by grid barriers (bounded waits), so a column of
// a few thousand warp tiles pays one launch instead of three.
//   phase 1  index pass (every thread) and tile elements (every warp);
//   phase 2  block 0 scans the tile elements (one block is enough for the
//            sizes this path takes) and checks the decoded size;
//   phase 3  every warp decodes tiles, as warp_decode_kernel.
// Data written by earlier phases is read through L2 (ld.global.cg).
// ---------------------------------------------------------------------------
// Exclusive scan of n tile elements by one block of NT threads: ex[t] =
// bytes before tile t | entering state << 63; the decoded size and its
// checks as the tile scan's last block.
template <bool FSST, int NT>
__device__ __forceinline__ void block_scan_tiles(const DecodeParams& p, const u64* agg, u64* ex, u64 n, Elem* s_w) {
    const u32 lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const u64 per = (n + NT - 1) / NT;
    const u64 i0 = (u64)threadIdx.x * per, i1 = i0 + per < n ? i0 + per : n;
    Elem e = elem_identity();
    for (u64 i = i0; i < i1; ++i) e = then<FSST>(e, wt_unpack<FSST>(__ldcg(agg + i)));
    Elem inc = e;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        Elem y = shfl_up_e<FSST>(inc, d);
        if (lane < (u32)d) y = elem_identity();
        inc = then<FSST>(y, inc);
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    Elem before = elem_identity(), tot = elem_identity();
    for (int w = 0; w < NT / 32; ++w) {
        if ((u32)w < warp) before = then<FSST>(before, s_w[w]);
        tot = then<FSST>(tot, s_w[w]);
    }
    Elem lex = shfl_up_e<FSST>(inc, 1);
    if (lane == 0) lex = elem_identity();
    lex = then<FSST>(before, lex);
    u64 ob = lex.b0;   // the column is entered on a code: state 0
    u32 os = FSST ? (lex.n & 1u) : 0u;
    for (u64 i = i0; i < i1; ++i) {
        ex[i] = ob | ((u64)os << 63);
        const Elem ek = wt_unpack<FSST>(__ldcg(agg + i));
        ob += (FSST && os) ? ek.b1 : ek.b0;
        os = FSST ? ((ek.n >> os) & 1u) : 0u;
    }
    if (threadIdx.x == 0) {
        const u64 total = tot.b0;
        *p.total_out = total;
        if (total > p.capacity && !p.size_only) atomicOr(p.err_word, ERRB_CAPACITY);
        if (total > 0x7fffffffull) atomicOr(p.err_word, ERRB_OVERFLOW);
    }
}

template <int CODEC, int K, bool DSMEM, int NW, int W = WarpCore<CODEC, K, DSMEM>::TOK8 ? 8 : 16>
__global__ void __launch_bounds__(NW * 32, 1) fused_decode_kernel(const DecodeParams p, Extent* xp, u64* agg,
                                                                   u64* ex) {
    typedef WarpCore<CODEC, K, DSMEM, W> C;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ Elem s_w[NW];
    __shared__ __align__(8) u64 s_code_bar[NW];
    uint4* s_dict = reinterpret_cast<uint4*>(smem_raw);
    uint8_t* s_lens = smem_raw + C::DICT_BYTES;
    typename C::Area* areas = reinterpret_cast<typename C::Area*>(smem_raw + C::STAGED_BYTES);
    if (DSMEM) {
        C::stage_dict(p, s_dict, s_lens, NW * 32);
        __syncthreads();
    }
    const uint8_t* lens = DSMEM ? s_lens : p.dict.lens;
    const u32 epoch = *(volatile u32*)&p.ws->epoch;
    const Extent x = column_extent(p, C::TILE);
    if (blockIdx.x == 0 && threadIdx.x == 0) *xp = x;
    const u32 lane = threadIdx.x & 31u;
    const u64 gwarp = (u64)blockIdx.x * NW + (threadIdx.x >> 5), gwarps = (u64)gridDim.x * NW;
    u32 err = 0;
    // phase 1
    index_groups(p, x, (u32)(__ffs(C::TILE) - 1), 0, (u64)p.n_strings + 1, (u64)blockIdx.x * blockDim.x + threadIdx.x,
                 (u64)gridDim.x * blockDim.x, const_cast<u32*>(p.first));
    for (u64 t = gwarp; t < x.n_tiles; t += gwarps) {
        u32 wv[C::LANE_WORDS];
        const u64 q0 = C::lane_q0(x, t);
        const bool fast = C::load_fast(p, q0, wv);
        typename C::R r;
        C::finish_load(p, x, q0, wv, fast, lens, r);
        const TElem e = C::tile_element(r, lane, err);
        if (lane == 31) agg[t] = wt_pack<C::FSST>(e);
    }
    grid_barrier(p.ws);
    // phase 2
    if (blockIdx.x == 0) block_scan_tiles<C::FSST, NW * 32>(p, agg, ex, x.n_tiles, s_w);
    grid_barrier(p.ws);
    // phase 3
    C::decode_tiles(p, x, ex, gwarp, gwarps, s_dict, lens, areas[threadIdx.x >> 5],
                                   s_code_bar + (threadIdx.x >> 5), err);
    if (err) atomicOr(p.err_word, err);
    __syncthreads();
    finish_launch(p.ws, epoch);   // the last block out clears the abort flag and the stall settings
}

}  // namespace
}  // namespace fp
