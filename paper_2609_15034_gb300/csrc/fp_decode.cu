// Single-column decoder for sm_103a: the variant tables (their kernel
// instantiations are in fp_var*.cu) with their size- and width-dependent
// defaults, and the launches of one decode call (index pass + block-pipeline
// decode, or index pass and reduce in one grid + tile scan + warp-tile
// decode).
#include "fp_decoder.cuh"
#include "fp_reduce.cuh"
#include "fp_warp.cuh"

namespace fp {
namespace {

// Index pass of the block pipeline over one column (grid-stride over its
// string boundaries).
__global__ void __launch_bounds__(256) index_kernel(const DecodeParams p, u32 tile, u32* first) {
    const Extent x = column_extent(p, tile);
    index_groups(p, x, (u32)(__ffsll((long long)tile) - 1), 0, (u64)p.n_strings + 1,
                 (u64)blockIdx.x * blockDim.x + threadIdx.x, (u64)gridDim.x * blockDim.x, first);
}

}  // namespace

// Variant tables (one translation unit per codec).
const Variant* variants_onpair16(int* n);
const Variant* variants_onpair12(int* n);
const Variant* variants_fsst8(int* n);
const Variant* variants_fsst12(int* n);

static const Variant* table_for(int codec, int* n) {
    switch (codec) {
        case FP_ONPAIR16: return variants_onpair16(n);
        case FP_ONPAIR12: return variants_onpair12(n);
        case FP_FSST8: return variants_fsst8(n);
        case FP_FSST12: return variants_fsst12(n);
        default: *n = 0; return nullptr;
    }
}

int variant_count(int codec) {
    int n;
    table_for(codec, &n);
    return n;
}

const Variant* variant_get(int codec, int v) {
    int n;
    const Variant* t = table_for(codec, &n);
    return (t && v >= 0 && v < n) ? &t[v] : nullptr;
}

// Defaults chosen by measurement on GB300 (synthetic columns, every variant
// timed at 30k..10M strings): warp tiles for every codec, one block of 16
// warps per SM for large columns, with the dictionary (OnPair-16: its
// lengths) in shared memory: OnPair-12, 10M strings, 583 us a call against 797
// with the table read through L1; OnPair-16, 2M strings, 174 against 198 for
// blocks of 8 warps; FSST-8, 16M strings, 529 with 32-slot lanes against 562
// for blocks of 8 warps and 698 with 16-slot lanes; FSST-12, 20k documents, 99
// with 32-slot lanes, 106 with 16, 130 through L1.  This is the rule where no
// tuned shape is loaded.  OnPair-12 stages its table at every size (calls of
// 2^17 .. 2^23 slots, staged against through L1: 11.9 : 14.0, 12.0 : 14.5, 12.0 :
// 15.7, 17.0 : 17.2, 22.5 : 25.4, 30.9 : 39.4, 52.3 : 67.6 us; split reads 11.9 :
// 14.9 .. 51.9 : 73.6); FSST-8 and FSST-12 take 16-slot lanes below 2^22 and 2^23
// slots.  The OnPair codecs come in both read widths (split read W = 8, whole
// entries W = 16); the dictionary's width picks between them.
//
// Below 2^17 slots (256 tiles of 512: one to a warp of 16 blocks) the whole
// column goes to one cluster in one launch: 9.0-10.0 us a call back to back
// against 13.0-14.6 for three launches, alone 23.8-27.7 against 26.7-29.1, from
// 9k to 125k slots (OnPair-16, whose tiles have half the slots, 12.8-14.0
// against 13.2-13.7 from 80k on, alone 29.6-30.4 against 29.1); at 146k-177k
// slots the cluster's 16 SMs are the slower side (13.3-17.6 us against
// 12.8-13.4).  Four host-launched streams: 4.8 us a call, one launch's host time,
// against 8.1; four streams of graphs, 18k slots: 1.8-2.1 against 2.4-3.0.  What
// it costs is throughput with the GPU full of small columns: 16 streams of
// graphs, 1.0-1.1 us against 0.73-0.86 at 18k slots, 1.2-1.8 against 0.8-1.05
// at 100k.  Split-read dictionaries keep the three launches.
//
// A cluster's 256 warps also write every string's offset: with 2^17 strings
// or more the three launches are the faster side (100k slots: 100k strings
// 13.6-18.7 us against 14.5-15.7, 300k strings 22.6-30.6 against 18.9-26.2, 4M
// strings 189-299 against 119-239).
uint64_t cluster_strings_limit() { return 1ull << 17; }

int variant_default(int codec, uint64_t max_slots, int width) {
    const bool split = width != 16;
    if (max_slots < (1ull << 17)) {
        switch (codec) {
            case FP_ONPAIR12: if (!split) return 12; break;
            case FP_ONPAIR16: if (!split) return 7; break;
            case FP_FSST8: return 6;
            case FP_FSST12: return 4;
            default: break;
        }
    }
    switch (codec) {
        case FP_ONPAIR12:
            return split ? 6 : 8;
        case FP_ONPAIR16: return split ? 5 : 4;
        case FP_FSST8: return max_slots >= (1ull << 22) ? 4 : 2;
        case FP_FSST12: return max_slots >= (1ull << 23) ? 2 : 0;
        default: return 0;
    }
}

int noalloc_default(int codec) {
    switch (codec) {
        case FP_FSST8: return 1;    // block pipeline, 32 slots per thread
        case FP_FSST12: return 0;   // no block pipeline: warp tiles
        default: return 0;          // block pipeline
    }
}

uint64_t variant_tile(const Variant& v) {
    return (uint64_t)(v.warp_tiles ? 32 : kWork) * (uint64_t)v.slots_per_thread;
}

namespace {

// Launch with programmatic stream serialization: the kernel may begin while
// the previous kernel on the stream finishes; it calls grid_wait() before it
// reads that kernel's results.
cudaError_t launch_after(const void* func, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, func, args);
}

constexpr size_t kExtentBytes = 64;
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch layout of a variant for a buffer of max_slots slots.
struct ScratchLayout {
    uint64_t n_tiles;        // tiles (block tiles or warp tiles) covering the buffer, plus slack
    size_t o_status, o_first, o_agg, o_ex, o_extent, bytes;
};

ScratchLayout scratch_layout(const Variant& v, uint64_t max_slots) {
    ScratchLayout L{};
    L.n_tiles = max_slots / variant_tile(v) + 2;
    if (!v.warp_tiles) {
        L.o_status = 0;
        L.o_first = al256(L.n_tiles * sizeof(unsigned long long));
        L.bytes = al256(L.o_first + (L.n_tiles + 1) * sizeof(uint32_t));
        return L;
    }
    const uint64_t n_scan = L.n_tiles / kScanTile + 2;
    L.o_status = 0;
    L.o_extent = al256(n_scan * sizeof(unsigned long long));
    L.o_agg = L.o_extent + al256(kExtentBytes);
    L.o_ex = L.o_agg + al256(L.n_tiles * sizeof(u64));
    L.o_first = L.o_ex + al256(L.n_tiles * sizeof(u64));
    L.bytes = al256(L.o_first + (L.n_tiles + 1) * sizeof(uint32_t));
    return L;
}

}  // namespace

size_t variant_scratch_bytes(const Variant& v, uint64_t max_slots) { return scratch_layout(v, max_slots).bytes; }

cudaError_t launch_decode(int codec, const Variant& var, const DecodeParams& p_in, void* scratch, uint64_t max_slots,
                          int grid, int sms, cudaStream_t stream) {
    (void)codec;
    const ScratchLayout L = scratch_layout(var, max_slots);
    char* base = static_cast<char*>(scratch);
    DecodeParams p = p_in;
    p.err_word = &p.ws->status;
    p.total_out = &p.ws->total;
    p.tile_status = reinterpret_cast<unsigned long long*>(base + L.o_status);
    uint32_t* first = reinterpret_cast<uint32_t*>(base + L.o_first);
    p.first = first;
    const uint64_t tile = variant_tile(var);
    const uint64_t nb = (uint64_t)p.n_strings + 1;
    uint64_t ib = (nb + 256 * kIdxGroup - 1) / (256 * kIdxGroup);
    if (ib > (uint64_t)sms * 2) ib = (uint64_t)sms * 2;   // two index blocks per SM
    cudaError_t e;
    void* args[] = {(void*)&p};
    if (!var.warp_tiles) {
        index_kernel<<<(unsigned)ib, 256, 0, stream>>>(p, (u32)tile, first);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return cudaLaunchKernel(var.kernel, dim3(grid), dim3(var.threads), args, var.smem_bytes, stream);
    }

    Extent* xp = reinterpret_cast<Extent*>(base + L.o_extent);
    u64* agg = reinterpret_cast<u64*>(base + L.o_agg);
    u64* ex = reinterpret_cast<u64*>(base + L.o_ex);
    if (var.warp_tiles == 2) {
        // one cooperative launch: every block resident, phases split by grid barriers
        const int nw = var.threads / 32;
        uint64_t dg = (L.n_tiles + nw - 1) / nw;
        if (dg > (uint64_t)grid) dg = (uint64_t)grid;
        void* fargs[] = {(void*)&p, (void*)&xp, (void*)&agg, (void*)&ex};
        return cudaLaunchCooperativeKernel(var.kernel, dim3((unsigned)dg), dim3(var.threads), fargs, var.smem_bytes,
                                           stream);
    }

    if (var.warp_tiles == 3) {
        // one cluster of up to `grid` blocks, four tiles to a block while there
        // are blocks (OnPair-12, 36 tiles: 11.1 us a call; one tile to each
        // of a block's 16 warps, on three blocks: 12.2)
        unsigned blocks = 1;
        while (blocks < (unsigned)grid && blocks * 4ull < L.n_tiles) blocks *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(var.threads);
        cfg.dynamicSmemBytes = var.smem_bytes;
        cfg.stream = stream;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = blocks;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        return cudaLaunchKernelExC(&cfg, var.kernel, args);
    }

    // warp tiles: index pass + reduce in one launch, tile scan, decode.  Each
    // may start while the launch before it finishes and waits in the kernel
    // before it reads that launch's results.
    const uint64_t n_wt_max = L.n_tiles;   // upper bound; the kernels compute the true count
    const bool large = var.reduce_large && max_slots >= var.reduce_large_slots;
    const uint64_t rw = large ? var.reduce_large_threads / 32 : 8, rg_cap = (uint64_t)sms * (large ? 1 : 8);
    uint64_t rg = (n_wt_max + rw - 1) / rw;
    if (rg > rg_cap) rg = rg_cap;
    u32 index = large ? reduce_index_warps(nb, rg) : (u32)ib;   // warps of every block, or blocks
    void* rargs[] = {(void*)&p, (void*)&agg, (void*)&index};
    if (large) e = launch_after(var.reduce_large, dim3((unsigned)rg), dim3(var.reduce_large_threads), rargs, var.reduce_large_smem, stream);
    else e = launch_after(var.reduce, dim3((unsigned)(rg + ib)), dim3(256), rargs, 0, stream);
    if (e != cudaSuccess) return e;
    uint64_t sg = n_wt_max / kScanTile + 1;
    if (sg > (uint64_t)sms * 2) sg = (uint64_t)sms * 2;
    const u64* cagg = agg;
    unsigned long long* st = p.tile_status;
    u32 tile32 = (u32)tile;
    void* sargs[] = {(void*)&p, (void*)&tile32, (void*)&cagg, (void*)&ex, (void*)&st};
    e = launch_after(var.scan, dim3((unsigned)sg), dim3(256), sargs, 0, stream);
    if (e != cudaSuccess) return e;
    const u64* cex = ex;
    void* dargs[] = {(void*)&p, (void*)&cex};
    const int nw = var.threads / 32;
    uint64_t dg = (n_wt_max + nw - 1) / nw;
    if (dg > (uint64_t)grid) dg = (uint64_t)grid;
    e = launch_after(var.kernel, dim3((unsigned)dg), dim3(var.threads), dargs, var.smem_bytes, stream);
    if (e != cudaSuccess) {
        // the scan is enqueued and the decode, which renews the launch state
        // (renew_launch()), is not: the tickets go back to zero, the stall
        // settings too, and no look-back word keeps this launch's tag
        char* ws = reinterpret_cast<char*>(p.ws);
        cudaMemsetAsync(ws + kWsCounters, 0, kWsCounterBytes, stream);
        cudaMemsetAsync(ws + offsetof(WsHeader, spin_limit), 0, 2 * sizeof(unsigned), stream);
        cudaMemsetAsync(base + L.o_status, 0, L.o_extent - L.o_status, stream);
    }
    return e;
}

}  // namespace fp
