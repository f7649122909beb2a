// ts_topk.cu -- the top-k magnitude mask of Eq. 3-4 between the gate+up and
// the down launches of a pass: per token, only the `keep` neurons with the
// largest |Combined| (Combined = max(0, g) max(0, u), Eq. 2; a lower neuron
// index wins a tie) keep their c; the down projection then sums
// (Combined * Mask) W_down. Candidates are the token's both-active rows (every
// other row has Combined = 0 and adds nothing whether kept or not).
#include "ts_kernels.cuh"

namespace tsffn {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / kWarp;
constexpr int kKeyCache = 8;  // candidate keys a thread keeps in shared memory (the rest are re-read)

// Exclusive prefix of v over the block in thread order, and the block total
// (warp shuffles, then one warp over the warp sums).
__device__ __forceinline__ int block_excl_scan(int v, int* s_warp, int* s_total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == kWarp - 1) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = lane < kSelWarps ? s_warp[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += n;
        }
        if (lane < kSelWarps) s_warp[lane] = wi - w;
        if (lane == kWarp - 1) *s_total = wi;
    }
    __syncthreads();
    const int r = s_warp[warp] + incl - v;
    __syncthreads();  // s_warp is reused by the next scan
    return r;
}

// The digit (shift .. shift + 7) of the rem-th largest key, counted from the top, given the histogram of the
// keys that match the digits found so far: one warp, lane l holding digits 255 - 8l .. 248 - 8l. Digit 0 when
// none reaches rem, as a scan from the top stops at the bottom.
__device__ __forceinline__ void find_digit(const unsigned* hist, int shift, unsigned& s_prefix, unsigned& s_mask,
                                           int& s_remaining) {
    const int lane = threadIdx.x & 31;
    const unsigned prefix = s_prefix, mask = s_mask;
    const int rem0 = s_remaining;
    int c8[8], sum = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        c8[q] = (int)hist[255 - 8 * lane - q];
        sum += c8[q];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    int above = incl - sum;  // keys in higher digits
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int dg = 255 - 8 * lane - q;
        const bool reach = above + c8[q] >= rem0;
        const bool first = dg == 255 || above < rem0;
        if (first && (reach || dg == 0)) {
            s_prefix = prefix | ((unsigned)dg << shift);
            s_remaining = rem0 - above;  // how many keys equal to the final prefix are kept, at the end
        }
        above += c8[q];
    }
    if (lane == 0) s_mask = mask | (255u << shift);
}

// One CTA per token of the pass, up to kFastRows rows. c > 0 at a both-active row, so the fp32 bit pattern
// orders the candidates. A warp takes 16 words of the token's bitmap; the keys of a word's rows are one
// coalesced load, and all of them are compacted, in row order, into shared memory. An MSB-first radix select
// (four 8-bit digits, a warp adding its lanes' equal digits with one atomic: nearly all keys share the first
// digit) finds the keep-th largest key T; the rows with key > T and the first rows (ascending) with key == T
// stay. One CTA's latency is all there is to it: with each thread walking its own bitmap bytes the same
// selection took 12 us, 10 of them in the passes and their scattered key loads. With one token the union is the token's own bitmap, written here
// too (its dropped rows are then read by nobody, so their c stays).
//
// Every part is kept short where nearly all rows are candidates too: only the first digit, which nearly all keys
// share, is counted by match (it takes a step per distinct digit); a thread's candidates are consecutive, so it
// clears a bitmap word once; and the keys lie one word further every 32, which keeps those reads off one bank. The
// whole call of one token, d = 1024, m = 8000, all active (keep 400): 33.8 us with the kernel below, 31.5 with
// this one (38.8 when all digits were counted by match and every dropped row cleared by itself); 10% active: 24.5
// and 22.5. m = 16384, all active, keep 5461: 73.8 and 60.1. Never slower from 2000 to 16384 rows, 5 to 100% active.
constexpr int kFastRows = 16384;
constexpr int kWordsPerWarp = kFastRows / 32 / kSelWarps;
__host__ __device__ constexpr int cand_at(int c) { return c + (c >> 5); }  // place of candidate c
__global__ void __launch_bounds__(kSelThreads) k_topk_select_fast(const FfnLaunch a, int keep) {
    extern __shared__ unsigned s_key[];  // [cand_at(n_rows)] keys, then their rows (16 bits each)
    __shared__ unsigned s_kept[kFastRows / 32];
    __shared__ unsigned hist[256];
    __shared__ int s_warp[kSelWarps];
    __shared__ unsigned s_prefix, s_mask;
    __shared__ int s_remaining, s_total;
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.x;  // batch slot of the pass
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* cv = a.cval + (size_t)k * a.cval_tok_stride;
    unsigned* bb = reinterpret_cast<unsigned*>(a.bbits + (size_t)(a.bits_tok_base + k) * a.nbytes);
    unsigned short* s_row = reinterpret_cast<unsigned short*>(s_key + cand_at(a.n_rows));
    const int n_words = (a.n_rows + 31) / 32;
    unsigned word = 0u;
    if (lane < kWordsPerWarp) {
        const int w = warp * kWordsPerWarp + lane;
        if (w < n_words) {
            word = __ldcg(bb + w);
            const int left = a.n_rows - w * 32;  // bits past the row space may be stale
            if (left < 32) word &= (1u << left) - 1u;
            s_kept[w] = word;
        }
    }
    if (tid < 256) hist[tid] = 0u;
    if (tid == 0) {
        s_prefix = 0u;
        s_mask = 0u;
        s_remaining = keep;
    }
    int off = block_excl_scan(__popc(word), s_warp, &s_total);
    const int n = s_total;
    const bool one = a.nt == 1;
    if (keep < n) {
        float v[kWordsPerWarp];
#pragma unroll
        for (int i = 0; i < kWordsPerWarp; ++i) {
            const unsigned wi = __shfl_sync(0xffffffffu, word, i);
            v[i] = ((wi >> lane) & 1u) ? __ldcg(cv + (warp * kWordsPerWarp + i) * 32 + lane) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < kWordsPerWarp; ++i) {
            const unsigned wi = __shfl_sync(0xffffffffu, word, i);
            const int at = cand_at(__shfl_sync(0xffffffffu, off, i) + __popc(wi & ((1u << lane) - 1u)));
            if ((wi >> lane) & 1u) {
                s_key[at] = __float_as_uint(v[i]);
                s_row[at] = (unsigned short)((warp * kWordsPerWarp + i) * 32 + lane);
            }
        }
        __syncthreads();
        for (int shift = 24; shift >= 0 && keep > 0; shift -= 8) {
            const unsigned prefix = s_prefix, mask = s_mask;
            for (int b = 0; b < n; b += kSelThreads) {
                unsigned dg = 256u;
                if (b + tid < n) {
                    const unsigned key = s_key[cand_at(b + tid)];
                    if ((key & mask) == prefix) dg = (key >> shift) & 255u;
                }
                if (shift == 24) {
                    const unsigned peers = __match_any_sync(0xffffffffu, dg);
                    if (dg < 256u && lane == __ffs(peers) - 1) atomicAdd(&hist[dg], (unsigned)__popc(peers));
                } else if (dg < 256u) {
                    atomicAdd(&hist[dg], 1u);
                }
            }
            __syncthreads();
            if (warp == 0) {
                find_digit(hist, shift, s_prefix, s_mask, s_remaining);
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 8; ++q) hist[lane + 32 * q] = 0u;  // for the next digit
            }
            __syncthreads();
        }
        const unsigned T = keep > 0 ? s_prefix : 0xffffffffu;
        const int need_eq = keep > 0 ? s_remaining : 0;
        // rank of each key == T in row order: a thread's candidates are consecutive
        const int per = (n + kSelThreads - 1) / kSelThreads;
        const int c0 = min(tid * per, n), c1 = min(c0 + per, n);
        int eq = 0;
        for (int c = c0; c < c1; ++c) eq += s_key[cand_at(c)] == T;
        int rank = block_excl_scan(eq, s_warp, &s_total);
        int w = -1;  // the bitmap word of the last row dropped, and its rows dropped so far
        unsigned gone = 0u;
        for (int c = c0; c < c1; ++c) {
            const unsigned key = s_key[cand_at(c)];
            bool stays = key > T;
            if (key == T) stays = rank++ < need_eq;
            if (!stays) {
                const int row = s_row[cand_at(c)];
                if (row >> 5 != w) {
                    if (gone) atomicAnd(&s_kept[w], ~gone);
                    w = row >> 5;
                    gone = 0u;
                }
                gone |= 1u << (row & 31);
                if (!one) cv[row] = 0.0f;  // the down projection multiplies by c
            }
        }
        if (gone) atomicAnd(&s_kept[w], ~gone);
        __syncthreads();
    }
    for (int w = tid; w < n_words; w += kSelThreads) {
        const unsigned kept = s_kept[w];
        bb[w] = kept;
        if (one) reinterpret_cast<unsigned*>(a.ubits)[w] = kept;
    }
}

// The same for more than kFastRows rows: one CTA per token of the pass. c > 0 at a both-active row, so the fp32 bit
// pattern orders the candidates; an MSB-first radix select (four 8-bit
// digits) finds the keep-th largest key T, then the rows with key > T and the
// first rows (ascending) with key == T are kept. Threads own contiguous byte
// ranges of the bitmap, so a block prefix over the threads is row order; each
// thread keeps its first kKeyCache candidate keys in shared memory for the
// passes.
__global__ void __launch_bounds__(kSelThreads) k_topk_select(const FfnLaunch a, int keep) {
    __shared__ unsigned hist[256];
    __shared__ unsigned s_key[kKeyCache * kSelThreads];  // [slot][thread]: a thread's first candidates
    __shared__ int s_warp[kSelWarps];
    __shared__ unsigned s_prefix, s_mask;
    __shared__ int s_remaining, s_total;
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.x;  // batch slot of the pass
    const int tid = threadIdx.x;
    float* cv = a.cval + (size_t)k * a.cval_tok_stride;
    uint8_t* bb = a.bbits + (size_t)(a.bits_tok_base + k) * a.nbytes;
    const int n_bytes = (a.n_rows + 7) / 8;
    const int per = (n_bytes + kSelThreads - 1) / kSelThreads;
    const int b0 = min(tid * per, n_bytes), b1 = min(b0 + per, n_bytes);
    auto key_ld = [&](int p) { return __float_as_uint(cv[p]); };
    // the i-th candidate of this thread (row p): from shared memory for the
    // first kKeyCache, else from c
    auto key_of = [&](int i, int p) { return i < kKeyCache ? s_key[i * kSelThreads + tid] : key_ld(p); };

    // candidates, the first kKeyCache keys of each thread kept in shared memory
    int cnt = 0;
    for (int b = b0; b < b1; ++b)
        for (unsigned bits = bb[b]; bits; bits &= bits - 1u, ++cnt)
            if (cnt < kKeyCache) s_key[cnt * kSelThreads + tid] = key_ld(b * 8 + __ffs(bits) - 1);
    block_excl_scan(cnt, s_warp, &s_total);
    if (tid == 0) {
        s_prefix = 0u;
        s_mask = 0u;
        s_remaining = keep;
    }
    __syncthreads();
    if (keep >= s_total) return;  // every candidate is kept

    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = tid; i < 256; i += kSelThreads) hist[i] = 0u;
        __syncthreads();
        const unsigned prefix = s_prefix, mask = s_mask;
        int i = 0;
        for (int b = b0; b < b1; ++b)
            for (unsigned bits = bb[b]; bits; bits &= bits - 1u, ++i) {
                const unsigned key = key_of(i, b * 8 + __ffs(bits) - 1);
                if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
            }
        __syncthreads();
        if (tid < kWarp) find_digit(hist, shift, s_prefix, s_mask, s_remaining);
        __syncthreads();
    }
    const unsigned T = s_prefix;
    const int need_eq = s_remaining;
    // rank of each key == T in row order
    int eq = 0;
    {
        int i = 0;
        for (int b = b0; b < b1; ++b)
            for (unsigned bits = bb[b]; bits; bits &= bits - 1u, ++i) eq += key_of(i, b * 8 + __ffs(bits) - 1) == T;
    }
    int rank = block_excl_scan(eq, s_warp, &s_total);
    int i = 0;
    for (int b = b0; b < b1; ++b) {
        unsigned kept = 0u;
        for (unsigned bits = bb[b]; bits; bits &= bits - 1u, ++i) {
            const int r = __ffs(bits) - 1;
            const int p = b * 8 + r;
            const unsigned key = key_of(i, p);
            bool keep_it = key > T;
            if (key == T) keep_it = rank++ < need_eq;
            if (keep_it)
                kept |= 1u << r;
            else
                cv[p] = 0.0f;  // the down projection multiplies by c
        }
        bb[b] = (uint8_t)kept;
    }
}

// The pass's union both-active bytes from the masked per-token bytes.
__global__ void __launch_bounds__(256) k_topk_union(const FfnLaunch a) {
    pdl_wait();
    pdl_launch_dependents();
    const int n_bytes = (a.n_rows + 7) / 8;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n_bytes) return;
    unsigned u = 0u;
    for (int k = 0; k < a.nt; ++k) u |= a.bbits[(size_t)(a.bits_tok_base + k) * a.nbytes + b];
    a.ubits[b] = (uint8_t)u;
}

constexpr size_t fast_smem(int n_rows) {
    return (size_t)cand_at(n_rows) * (sizeof(unsigned) + sizeof(unsigned short)) + 16;
}

}  // namespace

cudaError_t prepare_topk() {
    return cudaFuncSetAttribute(k_topk_select_fast, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fast_smem(kFastRows));
}

cudaError_t launch_topk(const FfnLaunch& a, int keep, cudaStream_t stream) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    lc.stream = stream;
    lc.gridDim = dim3(a.nt);
    lc.blockDim = dim3(kSelThreads);
    const bool fast = a.n_rows <= kFastRows;
    if (fast) lc.dynamicSmemBytes = fast_smem(a.n_rows);
    cudaError_t e = fast ? cudaLaunchKernelEx(&lc, k_topk_select_fast, a, keep) : cudaLaunchKernelEx(&lc, k_topk_select, a, keep);
    if (e != cudaSuccess || (fast && a.nt == 1)) return e;  // one token: the select wrote the union too
    lc.dynamicSmemBytes = 0;
    const int n_bytes = (a.n_rows + 7) / 8;
    lc.gridDim = dim3((n_bytes + 255) / 256);
    lc.blockDim = dim3(256);
    return cudaLaunchKernelEx(&lc, k_topk_union, a);
}

}  // namespace tsffn
