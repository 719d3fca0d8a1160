// Append (prefill write of the replayed suffix, Sec. 3.2) and crop
// (restore = crop, Sec. 3.4(b); Alg. 1 Restore) kernels.
//
// Both are HBM/latency-bound copies: every thread moves whole 16-byte chunks
// (8 bf16) with vector loads and stores; consecutive threads touch consecutive
// chunks of one d-row, so a warp reads 512 contiguous bytes of the caller's
// K/V and writes whole 256-byte rows (d = 128) of a page slot.
#include <algorithm>
#include <cstddef>
#include <cstring>

#include "pe_internal.h"
#include "ptx.cuh"

namespace pe {

// The finite poison written by the debug crop: bf16 2^100 (0x7180) in every lane.
constexpr uint32_t kPoisonPair = 0x71807180u;

__device__ __forceinline__ uint4 ld_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// A launch's parameter block is copied by the host, by CUDA and by the GPU's front end: 15 KB of it cost a
// launch 0.5 us more than 1 KB (2.03 against 1.60 us of host time).  A batch of few sequences and pages
// takes the kernel's form with the small block.
constexpr int kSmallSegs = 16, kSmallPages = 128;

template <typename Params>
__global__ void __launch_bounds__(256) append_kv_kernel(const __grid_constant__ Params p, int64_t chunks)
{
    // the attention launch that follows may start its set-up now; it waits for this grid's writes
    ptx::griddep_launch_dependents();
    // launched with programmatic serialization: only the launch overlaps the previous kernel; every
    // read and write here waits for it (a crop before may still be poisoning freed pages).  With
    // p.beside that kernel is a decode merge, which lets dependents in once the decode kernel, and so all
    // before it, is complete, and which reads only partials: the append runs beside it and waits at its
    // end, so that whatever waits for the append waits for the merge too (16 agents, some 120 rounds of an
    // append, a decode and a merge: 6630 -> 6404 us)
    if (!p.beside) ptx::griddep_wait();
    // 1) mirror the new page ids and lengths into the device tables
    if (blockIdx.x == 0) {
        for (int s = 0; s < p.n_segs; ++s) {
            const AppendSeg &sg = p.segs[s];
            for (int i = threadIdx.x; i < sg.n_new; i += blockDim.x)
                p.page_table[sg.table_row + sg.first_new_lp + i] = p.new_pages[sg.new0 + i];
            if (threadIdx.x == 0)
                p.seq_len[sg.seq] = static_cast<int64_t>(sg.len0) + sg.n_tokens;
        }
    }
    // 2) scatter K/V rows into their page slots
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; c < chunks; c += stride) {
        const int dv = static_cast<int>(c % p.dvec);
        int64_t r = c / p.dvec;
        const int h = static_cast<int>(r % p.hkv);
        r /= p.hkv;
        const int t = static_cast<int>(r % p.seg_tokens);  // token within this launch's segments
        const int l = static_cast<int>(r / p.seg_tokens);
        int lo = 0, hi = p.n_segs - 1;
        while (lo < hi) {  // last segment with cum0 <= t
            const int mid = (lo + hi + 1) >> 1;
            if (p.segs[mid].cum0 <= t) lo = mid; else hi = mid - 1;
        }
        const AppendSeg &sg = p.segs[lo];
        const int local = t - sg.cum0;
        const int pos = sg.len0 + local;
        const int lp = pos / p.ps;
        const int slot = pos - lp * p.ps;
        const int page = lp < sg.first_new_lp ? sg.last_page : p.new_pages[sg.new0 + (lp - sg.first_new_lp)];
        const int64_t src = ((static_cast<int64_t>(l) * p.n_total + sg.tok0 + local) * p.hkv + h) * p.dvec + dv;
        const int64_t dst =
            (((static_cast<int64_t>(l) * p.num_pages + page) * p.hkv + h) * p.ps + slot) * p.dvec + dv;
        const uint4 kv = ld_stream(p.K + src);
        const uint4 vv = ld_stream(p.V + src);
        p.k_pool[dst] = kv;
        p.v_pool[dst] = vv;
    }
    if (p.beside) ptx::griddep_wait();
}

// The fields before the segment table, which both forms of a parameter block share.
template <typename Small, typename Full>
static void copy_header(Small &q, const Full &p)
{
    static_assert(offsetof(Small, segs) == offsetof(Full, segs), "the same header");
    std::memcpy(static_cast<void *>(&q), static_cast<const void *>(&p), offsetof(Full, segs));
}

cudaError_t launch_append(const AppendParams &p, int64_t chunks, cudaStream_t st)
{
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 148;
    }
    int64_t blocks = (chunks + 255) / 256;
    const int64_t cap = static_cast<int64_t>(sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.n_segs <= kSmallSegs && p.n_new <= kSmallPages) {
        using Small = AppendParamsT<kSmallSegs, kSmallPages>;
        Small q;
        copy_header(q, p);
        std::copy(p.segs, p.segs + p.n_segs, q.segs);
        std::copy(p.new_pages, p.new_pages + p.n_new, q.new_pages);
        return cudaLaunchKernelEx(&cfg, append_kv_kernel<Small>, q, chunks);
    }
    return cudaLaunchKernelEx(&cfg, append_kv_kernel<AppendParams>, p, chunks);
}

// One block per cropped sequence.  Debug poison first overwrites the pages
// whose last reference this crop dropped (every layer, head, slot, K and V) and
// the stale tail of the last kept page when no other sequence holds it; then
// the table entries [keep, old_n) of this sequence become -1.
template <typename Params>
__global__ void __launch_bounds__(256) crop_kernel(const __grid_constant__ Params p)
{
    // launched with programmatic serialization: the launch overlaps the previous kernel (an attention
    // launch that may still read the pages this crop frees); every write here waits for it
    ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    const CropSeg &sg = p.segs[blockIdx.x];
    int32_t *row = p.page_table + sg.table_row;
    if (p.poison) {
        const uint4 poison = make_uint4(kPoisonPair, kPoisonPair, kPoisonPair, kPoisonPair);
        const int slot_chunks = p.dvec;                          // chunks per (page, head, slot)
        const int page_chunks = p.hkv * p.ps * slot_chunks;      // per (layer, page)
        for (int e = 0; e < sg.n_freed; ++e) {
            const int page = p.freed[sg.freed0 + e];
            if (page < 0 || page >= p.num_pages) continue;
            for (int l = 0; l < p.L; ++l) {
                const int64_t base = (static_cast<int64_t>(l) * p.num_pages + page) * page_chunks;
                for (int i = threadIdx.x; i < page_chunks; i += blockDim.x) {
                    p.k_pool[base + i] = poison;
                    p.v_pool[base + i] = poison;
                }
            }
        }
        const int tail = static_cast<int>(sg.new_len % p.ps);
        const int page = sg.tail_page;
        if (tail != 0 && page >= 0 && page < p.num_pages) {
            const int per_head = (p.ps - tail) * slot_chunks;
            for (int l = 0; l < p.L; ++l)
                for (int h = 0; h < p.hkv; ++h) {
                    const int64_t base =
                        (((static_cast<int64_t>(l) * p.num_pages + page) * p.hkv + h) * p.ps + tail) * slot_chunks;
                    for (int i = threadIdx.x; i < per_head; i += blockDim.x) {
                        p.k_pool[base + i] = poison;
                        p.v_pool[base + i] = poison;
                    }
                }
        }
        __syncthreads();
    }
    for (int e = sg.keep + static_cast<int>(threadIdx.x); e < sg.old_n; e += blockDim.x)
        row[e] = -1;
    if (threadIdx.x == 0)
        p.seq_len[sg.seq] = sg.new_len;
}

cudaError_t launch_crop(const CropParams &p, cudaStream_t st)
{
    if (p.n <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(p.n));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.n <= kSmallSegs && !p.poison) {  // (the freed pages are only read to poison them)
        using Small = CropParamsT<kSmallSegs, 1>;
        Small q;
        copy_header(q, p);
        std::copy(p.segs, p.segs + p.n, q.segs);
        return cudaLaunchKernelEx(&cfg, crop_kernel<Small>, q);
    }
    return cudaLaunchKernelEx(&cfg, crop_kernel<CropParams>, p);
}

__global__ void __launch_bounds__(256) table_copy_kernel(int32_t *page_table, int32_t src_row, int32_t dst_row,
                                                         int32_t n, int64_t *seq_len, int32_t dst_seq, int64_t len)
{
    ptx::griddep_wait();  // launched with programmatic serialization: only the launch overlaps the kernel before
    for (int i = threadIdx.x; i < n; i += blockDim.x) page_table[dst_row + i] = page_table[src_row + i];
    if (threadIdx.x == 0) seq_len[dst_seq] = len;
}

cudaError_t launch_table_copy(int32_t *page_table, int32_t src_row, int32_t dst_row, int32_t n, int64_t *seq_len,
                              int32_t dst_seq, int64_t len, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, table_copy_kernel, page_table, src_row, dst_row, n, seq_len, dst_seq, len);
}

// The copies of one append call, one launch before its append launch: grid (layer x kv-head, copy), each
// block `slots` rows of d (16-byte chunks).  A few KB each, so a launch's own time is what they cost: one
// launch per forked sequence (7 of 8 branches, 3.3 us each, one after another) made a replay of 8 branches
// 205 us; one launch, overlapped like the forks' table copies with the kernel before it, 153 us.
__global__ void __launch_bounds__(128) cow_copy_kernel(const __grid_constant__ CowParams p)
{
    ptx::griddep_wait();  // launched with programmatic serialization
    const CowCopy &c = p.copies[blockIdx.y];
    const int l = blockIdx.x / p.hkv;
    const int h = blockIdx.x % p.hkv;
    const int64_t s_base = ((static_cast<int64_t>(l) * p.num_pages + c.src) * p.hkv + h) * p.ps * p.dvec;
    const int64_t d_base = ((static_cast<int64_t>(l) * p.num_pages + c.dst) * p.hkv + h) * p.ps * p.dvec;
    for (int i = threadIdx.x; i < c.slots * p.dvec; i += blockDim.x) {
        p.k_pool[d_base + i] = p.k_pool[s_base + i];
        p.v_pool[d_base + i] = p.v_pool[s_base + i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) p.page_table[c.entry] = c.dst;
}

cudaError_t launch_cow_copy(const CowParams &p, cudaStream_t st)
{
    if (p.n <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(p.L * p.hkv), static_cast<unsigned>(p.n));
    cfg.blockDim = dim3(128);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cow_copy_kernel, p);
}

}  // namespace pe
