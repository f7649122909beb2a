// ts_wide.cu -- passes of 9-64 tokens (bf16 weights, d a multiple of 256) on
// the 5th-generation tensor cores, each weight row read once per batch.
//
// At these batch sizes the union of the tokens' active sets covers most
// neurons (Eq. 2 per token, union over the batch), so the FFN of Eq. 1 is a
// dense contraction over the active rows:
//   k_wide_gate_up  one CTA per tile of rows: G = x . W_gate^T, per-token gate
//                   bitmaps and their union, then U = x . W_up^T over the same
//                   tile's union gate-active rows (the others are not read),
//                   c = g u where both are positive (Eq. 2), per-token both
//                   bitmaps, and the tile's both-active rows listed with
//                   their c as a pair of bf16 (hi + lo, |c - hi - lo| <= 2^-16 |c|);
//   k_wide_down     partial[s][t][:] = sum over the rows that the tiles of
//                   slice s listed of c_t,p W_down[row p][:] (Eq. 1);
//   k_wide_reduce   y_t = sum over slices s in order (or h_t += y_t).
// HBM bounds them (64 tokens are 64 flop per weight byte, a quarter of what the
// tensor cores could do with it), so both kernels are built to keep weight
// copies in flight on every SM: tiles of as many rows as give each SM one,
// up to kMaxStages stages of 16-byte cp.async, and no CTA-wide barrier in the
// stream. Measured at d = 4096, m = 14336, 64 tokens (10% active): 135 -> 71.6 us
// a call (16 tokens: 97.5 -> 59.5) against separate gate and up kernels of 128-row
// tiles on 112 SMs with a barrier per stage and a down kernel of 128-column tiles.
#include "ts_kernels.cuh"
#include "ts_wide.h"

namespace tsffn {
namespace {

// gate/up: K per pipeline stage, as two tiles of 128 bytes of a row. A stage costs the MMA thread about 0.3 us
// (wait, proxy fence, issue, commit) whatever its size: 64-wide stages were bound by that.
constexpr int kTileK = 128;
constexpr int kThreads = 256;    // copying (and epilogue) threads; one more warp issues the MMAs
constexpr int kCta = kThreads + kWarp;
constexpr int kTokPad = 64;      // token columns of a list row's c
constexpr int kTcRows = 128;     // the MMA's M
constexpr int kMaxStages = 12;
// Stages whose weights are pulled into L2 before the previous kernel is waited for (copied there and then, 64
// tokens took 69.8 us as well, but the kernel before might still be writing them; only after the wait: 70.6).
constexpr int kAheadOfX = 2;
constexpr int kPipe = 220 * 1024;  // pipeline bytes of a gate+up CTA

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// 16-byte copy global -> shared; bytes = 0 fills with zeros
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// byte offset of 16-byte chunk c of row r in a tile of 128-byte rows, with
// the chunk index XOR-ed by the row so that 8 rows at one chunk hit 8 banks
__device__ __forceinline__ int swz(int r, int c, int row_bytes) { return r * row_bytes + ((c ^ (r & 7)) << 4); }

// The row of the row space at position p: the list entry or p itself;
// -1 (skipped, recorded) for a list entry out of range or not ascending.
__device__ __forceinline__ int row_of(const WideLaunch& L, int p) {
    if (L.rows == nullptr) return p;
    const int j = L.rows[p];
    if ((unsigned)j >= (unsigned)L.m || (p > 0 && L.rows[p - 1] >= j)) {
        atomicOr(L.status, kStatusBadIndex);
        return -1;
    }
    return j;
}

// ---------------------------------------------------------------------------
// tcgen05 helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tc_alloc(uint32_t* dst, uint32_t ncols) {  // warp-wide
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_relinquish() {  // warp-wide
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols) {  // warp-wide
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D (tensor memory) = A B^T (+ D when `accumulate`), one thread issues it
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrive once on `bar` when every tcgen05.mma this thread issued so far has completed
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}
// 32 lanes x 16 fp32 columns: lane l of the warp gets the 16 columns of TMEM lane (taddr lane + l)
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// shared-memory descriptor of a K-major bf16 tile with 128-byte rows and the
// 128-byte swizzle (8-row atoms of 1024 bytes, atom-aligned start)
__device__ __forceinline__ uint64_t sdesc_k128(uint32_t saddr) {
    uint64_t dsc = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address, 16-byte units
    dsc |= (uint64_t)1 << 16;                            // leading byte offset (not used by this layout)
    dsc |= (uint64_t)(1024 >> 4) << 32;                  // stride byte offset: between 8-row atoms
    dsc |= (uint64_t)1 << 46;                            // descriptor version
    dsc |= (uint64_t)2 << 61;                            // 128-byte swizzle
    return dsc;
}
// instruction descriptor: bf16 A and B (both K-major), fp32 D, shape M x N
constexpr uint32_t idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// MN-major tile with the 128-byte swizzle: 64 contiguous MN elements per
// 128-byte K-row, 8 K-rows per 1024-byte atom; `lbo` bytes between 64-element
// MN blocks, 1024 bytes between 8-row K groups
__device__ __forceinline__ uint64_t sdesc_mn128(uint32_t saddr, uint32_t lbo) {
    uint64_t dsc = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    dsc |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    dsc |= (uint64_t)(1024 >> 4) << 32;
    dsc |= (uint64_t)1 << 46;
    dsc |= (uint64_t)2 << 61;
    return dsc;
}

// Pipeline between the copying threads and the thread that issues the MMAs,
// with no CTA-wide barrier in it: a stage's `full` completes when every
// thread's copies into it have landed, its `empty` when its MMAs have read it,
// `done` when every MMA of a product has completed. (With a barrier per stage
// and every thread waiting on the MMAs, a 20 KB stage took 0.6 us: 2.9 TB/s. With
// the copying threads waiting for their own copies to fence and report them,
// instead of the fence in the MMA thread, 64 tokens took 92 us against 72.)
struct TcShared {
    uint64_t full[kMaxStages], empty[kMaxStages], done;
    uint32_t tmem;  // accumulator address
    int fail;       // a bounded wait ran out
};

// tensor memory and barriers, by the whole CTA; warp 0 allocates
__device__ void tc_setup(TcShared& ts, uint32_t cols) {
    if (threadIdx.x < kWarp) {
        tc_alloc(&ts.tmem, cols);
        tc_relinquish();
    }
    if (threadIdx.x == kWarp) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&ts.full[s], kThreads);
            mbar_init(&ts.empty[s], 1);
        }
        mbar_init(&ts.done, 1);
        ts.fail = 0;
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}
__device__ void tc_teardown(TcShared& ts, uint32_t cols, unsigned* status) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && ts.fail) atomicOr(status, kStatusTimeout);
    if (threadIdx.x < kWarp) {
        tc_fence_after();
        tc_dealloc(ts.tmem, cols);
    }
}
// arrive on `bar` when this thread's cp.async so far have landed
__device__ __forceinline__ void cp_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// stage and phase of the it-th k-block of a CTA
struct StageAt {
    int st, ph;
    __device__ __forceinline__ void next(int stages) {
        if (++st == stages) {
            st = 0;
            ph ^= 1;
        }
    }
};
__device__ __forceinline__ bool tc_wait(uint64_t* bar, int ph, TcShared& ts) {
    if (mbar_wait(bar, (unsigned)ph)) return true;
    ts.fail = 1;
    return false;
}
// The MMA thread's side of a product: issue(stage) for each of nk k-blocks.
template <typename F>
__device__ bool tc_mmas(TcShared& ts, StageAt& at, int nk, int stages, F&& issue) {
    for (int kb = 0; kb < nk; ++kb) {
        if (!tc_wait(&ts.full[at.st], at.ph, ts)) return false;
        fence_proxy_async_smem();  // the landed copies before the tensor cores' reads
        tc_fence_after();
        issue(kb, at.st);
        tc_commit(&ts.empty[at.st]);
        at.next(stages);
    }
    tc_commit(&ts.done);
    return true;
}

__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
    const uint32_t a = smem_addr(p);
    return p + ((1024u - (a & 1023u)) & 1023u);
}

// ---------------------------------------------------------------------------
// gate + up: D[i][t] = W[row(i)] . x_t for a tile of `rows` weight rows (up to
// the MMA's M of 128; the MMA also reads what lies behind them in the stage,
// whose products are not used) and all tokens padded to NP = 16 MT, the gate
// and the up product in tensor-memory accumulators of their own.
//
// The copying threads fill each K stage (their shares of the weight rows and
// of the activations) as 128-byte-swizzled K-major tiles; for each stage that
// has landed one thread issues eight tcgen05.mma (K = 16 each) and a commit
// that frees it.
// A tile keeps its rows' places between the two products (rows that are not
// gate-active are zero-filled instead of copied), so gate and up values of a
// row meet in the same tensor-memory lane and need no exchange.
// ---------------------------------------------------------------------------
template <int MT>
struct GuCfg {
    static constexpr int NP = 16 * MT;
    static constexpr int kB = NP * 128;  // activations per tile of a stage
    static constexpr int kAcc = NP <= 32 ? 32 : 64;             // tensor-memory columns of an accumulator
    static constexpr uint32_t kCols = 2 * kAcc;
    static constexpr uint32_t kIdesc = idesc_bf16_f32(kTcRows, NP);
};

// The copying threads' side of k-blocks [kb, kb1) of a product: rows i < rows with bit i of mask[] set. `at`
// and `it` (k-blocks copied so far by this CTA) run on from product to product. first_x() runs once, after
// the prefetch of the first kAheadOfX stages' weights and before any copy.
template <int MT, typename F>
__device__ bool gu_copies(const WideLaunch& L, const __nv_bfloat16* w, const int* rows_j, const unsigned* mask, int rows,
                          int stages, int kb, int kb1, StageAt& at, int it, unsigned char* sm, TcShared& ts, F&& first_x) {
    using C = GuCfg<MT>;
    const int tid = threadIdx.x, d = L.d;
    const uint32_t half = (uint32_t)rows * 128, stage_bytes = 2 * (half + C::kB), sm0 = smem_addr(sm);
    const int c = tid & 7;  // this thread's 16-byte chunk of a row's 128 bytes in the stage; rows tid / 8 + 32 i
    const __nv_bfloat16* wsrc[4];
    uint32_t wbytes[4];
    bool win[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = (tid >> 3) + 32 * i;
        win[i] = r < rows;
        const int j = win[i] ? rows_j[r] : -1;
        const bool ok = j >= 0 && ((mask[r >> 5] >> (r & 31)) & 1u);
        wbytes[i] = ok ? 16u : 0u;
        wsrc[i] = w + (size_t)(ok ? debug_row(j, L.m, L.status) : 0) * d + c * 8;
    }
    constexpr int kXPer = (C::NP + 31) / 32;
    const __nv_bfloat16* xsrc[kXPer];
    uint32_t xbytes[kXPer];
#pragma unroll
    for (int i = 0; i < kXPer; ++i) {
        const int t = (tid >> 3) + 32 * i;
        xbytes[i] = t < L.batch ? 16u : 0u;
        xsrc[i] = L.x + (size_t)(t < L.batch ? t : 0) * d + c * 8;
    }
    // rows tid / 8 + 32 i of a tile lie 4096 bytes apart and share a swizzle
    const uint32_t dst = (uint32_t)swz(tid >> 3, c, 128);
    auto load_w = [&](int kb, uint32_t base) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (win[i]) {
                cp16(base + dst + 4096 * i, wsrc[i] + kb * kTileK, wbytes[i]);
                cp16(base + half + dst + 4096 * i, wsrc[i] + kb * kTileK + 64, wbytes[i]);
            }
    };
    auto load_x = [&](int kb, uint32_t base) {
#pragma unroll
        for (int i = 0; i < kXPer; ++i)
            if ((i + 1) * 32 <= C::NP || (tid >> 3) + 32 * i < C::NP) {
                cp16(base + 2 * half + dst + 4096 * i, xsrc[i] + kb * kTileK, xbytes[i]);
                cp16(base + 2 * half + C::kB + dst + 4096 * i, xsrc[i] + kb * kTileK + 64, xbytes[i]);
            }
    };
    if (it == 0) {
        if (c == 0)
            for (int k = 0; k < min(kAheadOfX, kb1); ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (wbytes[i] != 0u) {
                        prefetch_l2(wsrc[i] + k * kTileK);
                        prefetch_l2(wsrc[i] + k * kTileK + 64);
                    }
        first_x();
    }
    for (; kb < kb1; ++kb, ++it) {
        if (it >= stages && !tc_wait(&ts.empty[at.st], at.ph ^ 1, ts)) return false;
        const uint32_t base = sm0 + at.st * stage_bytes;
        load_w(kb, base);
        load_x(kb, base);
        cp_arrive(&ts.full[at.st]);
        at.next(stages);
    }
    return true;
}

template <int MT>
__global__ void __launch_bounds__(kCta, 1) k_wide_gate_up(const WideLaunch L, int rows, int stages) {
    using C = GuCfg<MT>;
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    __shared__ int rows_j[kTcRows];
    __shared__ unsigned s_all[kTcRows / 32], s_gate[kTcRows / 32], s_both[kTcRows / 32];
    __shared__ TcShared ts;
    unsigned char* sm = align1024(sm_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p0 = blockIdx.x * rows;
    const int n_in = min(rows, L.n_rows - p0);
    const bool early = L.rows == nullptr;  // the rows are known without the previous kernel
    if (!early) pdl_wait();
    if (tid < kTcRows) rows_j[tid] = tid < n_in ? row_of(L, p0 + tid) : -1;
    if (tid < kTcRows / 32) {
        s_all[tid] = 0xffffffffu;
        s_gate[tid] = 0u;
        s_both[tid] = 0u;
    }
    tc_setup(ts, C::kCols);
    pdl_launch_dependents();
    const int nk = L.d / kTileK;
    StageAt at{0, 0};
    if (warp == kThreads / kWarp) {
        if (lane == 0) {
            const uint32_t sm0 = smem_addr(sm);
            for (int p = 0; p < 2; ++p) {
                const bool ok = tc_mmas(ts, at, nk, stages, [&](int kb, int st) {
                    const uint32_t half = (uint32_t)rows * 128, a0 = sm0 + (uint32_t)st * 2 * (half + C::kB);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint64_t ad = sdesc_k128(a0 + h * half), bd = sdesc_k128(a0 + 2 * half + h * C::kB);
#pragma unroll
                        for (int kk = 0; kk < kTileK / 32; ++kk)  // 32 bytes of each row per MMA
                            tc_mma(ts.tmem + p * C::kAcc, ad + 2 * kk, bd + 2 * kk, C::kIdesc, (kb | h | kk) != 0);
                    }
                });
                if (!ok) break;
            }
        }
        __syncwarp();
        tc_teardown(ts, C::kCols, L.status);
        return;
    }
    bool ok = gu_copies<MT>(L, L.wg, rows_j, s_all, rows, stages, 0, nk, at, 0, sm, ts, [&]() {
        if (early) pdl_wait();
    });
    // The up product's first k-blocks are copied for every row, before the gate values say which are needed,
    // so that HBM does not idle meanwhile: an eighth of the bytes that the skipped rows would save at most.
    // (80.6 -> 77 us with the lists of the down kernel fetched a piece ahead.)
    const int spec = min(stages, nk / 8);
    ok = gu_copies<MT>(L, L.wu, rows_j, s_all, rows, stages, 0, spec, at, nk, sm, ts, []() {}) && ok;
    ok = __all_sync(0xffffffffu, tc_wait(&ts.done, 0, ts) && ok);
    tc_fence_after();
    // warp w holds tile rows 32 (w % 4) .. + 31 (one per lane) of token tiles w / 4, w / 4 + 2
    const int q = warp & 3, i = 32 * q + lane;
    const bool row_in = i < n_in && rows_j[i] >= 0;
    const uint32_t acc = ts.tmem + ((uint32_t)(32 * q) << 16);
    // a lane's bitmap byte: lanes 0, 8, 16, 24 store the chunks that begin at their rows
    const bool store = (lane & 7) == 0 && i < n_in;
    const size_t byte = (size_t)(p0 + i) / 8;
    unsigned uw = 0u;
    if (ok) {
        for (int mt = warp >> 2; mt < MT; mt += 2) {
            float v[16];
            tc_ld16(acc + 16 * mt, v);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int t = 16 * mt + e;
                if (t >= L.batch) break;
                const unsigned bits = __ballot_sync(0xffffffffu, row_in && v[e] > 0.0f);
                if (store) L.gbits[(size_t)t * L.nbytes + byte] = (uint8_t)(bits >> lane);
                uw |= bits;
            }
        }
        if (lane == 0 && uw) atomicOr(&s_gate[q], uw);
    }
    named_bar_sync(1, kThreads);
    ok = gu_copies<MT>(L, L.wu, rows_j, s_gate, rows, stages, spec, nk, at, nk + spec, sm, ts, []() {}) && ok;
    ok = __all_sync(0xffffffffu, tc_wait(&ts.done, 1, ts) && ok);
    tc_fence_after();
    // c = g u where both are positive (Eq. 2), for the warp's token tiles: kept for the lists below
    constexpr int kMine = (MT + 1) / 2;
    float c[kMine][16];
    uw = 0u;
    if (ok) {
#pragma unroll
        for (int k = 0; k < kMine; ++k) {
            const int mt = (warp >> 2) + 2 * k;
            float gv[16];
            if (mt < MT) {
                tc_ld16(acc + 16 * mt, gv);
                tc_ld16(acc + C::kAcc + 16 * mt, c[k]);
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int t = 16 * mt + e;
                const bool both = mt < MT && t < L.batch && row_in && gv[e] > 0.0f && c[k][e] > 0.0f;
                c[k][e] = both ? gv[e] * c[k][e] : 0.0f;
                const unsigned bits = __ballot_sync(0xffffffffu, both);
                if (store && mt < MT && t < L.batch) L.bbits[(size_t)t * L.nbytes + byte] = (uint8_t)(bits >> lane);
                uw |= bits;
            }
        }
        if (lane == 0 && uw) atomicOr(&s_both[q], uw);
    }
    named_bar_sync(1, kThreads);
    // the tile's both-active rows from entry p0 on, c split into bf16 hi + lo
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kTcRows / 32; ++w) {
        const int n = __popc(s_both[w]);
        before += w < q ? n : 0;
        total += n;
    }
    if (tid == 0) L.ent_n[blockIdx.x] = ok ? total : 0;
    if (ok && ((s_both[q] >> lane) & 1u)) {
        const size_t at = (size_t)p0 + before + __popc(s_both[q] & ((1u << lane) - 1u));
        if (warp < 4) L.ent[at] = rows_j[i];
#pragma unroll
        for (int k = 0; k < kMine; ++k) {
            const int mt = (warp >> 2) + 2 * k;
            if (mt >= MT) break;
            __align__(16) __nv_bfloat16 hi[16], lo[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                hi[e] = __float2bfloat16_rn(c[k][e]);
                lo[e] = __float2bfloat16_rn(c[k][e] - __bfloat162float(hi[e]));
            }
            uint4* dh = reinterpret_cast<uint4*>(L.c_hi + at * kTokPad + 16 * mt);
            uint4* dl = reinterpret_cast<uint4*>(L.c_lo + at * kTokPad + 16 * mt);
            dh[0] = reinterpret_cast<const uint4*>(hi)[0];
            dh[1] = reinterpret_cast<const uint4*>(hi)[1];
            dl[0] = reinterpret_cast<const uint4*>(lo)[0];
            dl[1] = reinterpret_cast<const uint4*>(lo)[1];
        }
    }
    cp_wait<0>();
    tc_teardown(ts, C::kCols, L.status);
}

// ---------------------------------------------------------------------------
// down: D[n][t] = sum over the slice's listed rows p of W_down[row p][n0 + n]
// c_t,p for 256 output columns (two MMAs of M = 128) and all tokens (N), both
// operands MN-major: a K-row of an A block is 128 contiguous bytes of a W_down
// row, a K-row of the B tile the 128 bytes of c (64 tokens) of that row. c
// enters as its bf16 hi and lo parts, each into an accumulator for even and one
// for odd stages: the tensor core truncates as it accumulates, and four short
// sums lose less than one (64 tokens, d = 4096, m = 14336: errors of 1.03e-5 -> 9.1e-6 of y).
// Stage (64 list rows): A as four 64-column blocks of 64 rows x 128 bytes
// (128-byte swizzle, 8-row atoms), then the c hi and lo tiles (64 x 128 bytes
// each): 32 KB of weights to 16 KB of c. (128-column tiles moved as much c as
// weights through each SM: 57 us, of which the bytes need 16.)
// ---------------------------------------------------------------------------
constexpr int kDownCols = 256;     // output columns per CTA
constexpr int kDownK = 64;         // list rows per stage
constexpr int kDownPiece = kThreads;  // list entries resolved at a time: one a thread
constexpr int kDownStages = 4;
constexpr int kMaxTiles = 1024;    // gate+up tiles (kWideMaxRows rows: one per SM and wave of 128 rows)

template <int MT>
struct DownCfg {
    static constexpr int NP = 16 * MT;
    static constexpr int kBlock = kDownK * 128;               // 8 KB: 64 rows x 64 columns (or tokens)
    static constexpr int kA = kDownCols / 64 * kBlock;
    static constexpr int kStage = kA + 2 * kBlock;            // 48 KB
    static constexpr int kBytes = kDownStages * kStage + 1024;  // + slack to align the tiles to 1024 bytes
    static constexpr int kAcc = NP <= 32 ? 32 : 64;
    static constexpr uint32_t kCols = 8 * kAcc;  // of half h: hi even, hi odd, lo even, lo odd
    // bf16 A and B, both MN-major (bits 15, 16), fp32 D
    static constexpr uint32_t kIdesc = idesc_bf16_f32(kTcRows, NP) | (1u << 15) | (1u << 16);
};

template <int MT>
__global__ void __launch_bounds__(kCta, 1) k_wide_down(const WideLaunch L, int tile_rows, int n_tiles_gu) {
    using C = DownCfg<MT>;
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    __shared__ int rowj[2][kDownPiece], src[2][kDownPiece];  // neuron (-1: none), place in the lists; by piece parity
    __shared__ int start[kMaxTiles + 1];  // entries listed before each tile of the slice
    __shared__ TcShared ts;
    unsigned char* sm = align1024(sm_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = L.d;
    const int n_tiles = d / kDownCols;
    const int n0 = (int)(blockIdx.x % (unsigned)n_tiles) * kDownCols;
    const int sl = (int)(blockIdx.x / (unsigned)n_tiles);
    tc_setup(ts, C::kCols);
    pdl_wait();
    pdl_launch_dependents();
    // the slice's gate+up tiles and the entries listed before each
    const int g0 = (int)((long long)n_tiles_gu * sl / L.ks), n_g = (int)((long long)n_tiles_gu * (sl + 1) / L.ks) - g0;
    if (warp == 0) {
        int run = 0;
        for (int b = 0; b < n_g; b += kWarp) {
            const int v = b + lane < n_g ? __ldcg(L.ent_n + g0 + b + lane) : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            if (b + lane < n_g) start[b + lane] = run + incl - v;
            run += __shfl_sync(0xffffffffu, incl, kWarp - 1);
        }
        if (lane == 0) start[n_g] = run;
    }
    __syncthreads();
    const int n_list = start[n_g];
    const int nk = (n_list + kDownK - 1) / kDownK;
    float* ps = L.partial + (size_t)sl * L.batch * d;
    constexpr int S = kDownStages;
    StageAt at{0, 0};
    if (warp == kThreads / kWarp) {
        if (lane == 0) {
            const uint32_t sm0 = smem_addr(sm);
            tc_mmas(ts, at, nk, S, [&](int kb, int st) {
                const uint32_t a0 = sm0 + st * C::kStage, b0 = a0 + C::kA;
#pragma unroll
                for (int kk = 0; kk < kDownK / 16; ++kk)  // 16 rows = two 8-row atoms per MMA
#pragma unroll
                    for (int h = 0; h < 2; ++h) {  // columns 128 h .. + 127
                        const uint64_t ad = sdesc_mn128(a0 + 2 * h * C::kBlock + kk * 2048, C::kBlock);
                        const uint32_t hi = ts.tmem + (4 * h + (kb & 1)) * C::kAcc, more = kb > 1 || kk != 0;
                        tc_mma(hi, ad, sdesc_mn128(b0 + kk * 2048, C::kBlock), C::kIdesc, more);
                        tc_mma(hi + 2 * C::kAcc, ad, sdesc_mn128(b0 + C::kBlock + kk * 2048, C::kBlock), C::kIdesc, more);
                    }
            });
        }
        __syncwarp();
        tc_teardown(ts, C::kCols, L.status);
        return;
    }
    // Entry e of the slice: its place in the lists. Each thread fetches its entry of the next piece while the
    // present one is copied.
    auto place = [&](int e) {
        int lo = 0, hi = n_g - 1;  // the tile that listed it
        while (lo < hi) {
            const int m = (lo + hi + 1) / 2;
            if (start[m] <= e)
                lo = m;
            else
                hi = m - 1;
        }
        return (g0 + lo) * tile_rows + e - start[lo];
    };
    int nsrc = 0, nrow = -1;
    auto fetch = [&](int piece) {
        const int e = piece * kDownPiece + tid;
        nrow = -1;
        if (e < n_list) {
            nsrc = place(e);
            nrow = __ldcg(L.ent + nsrc);
        }
    };
    auto publish = [&](int piece) {
        rowj[piece & 1][tid] = nrow < 0 ? -1 : debug_row(nrow, L.m, L.status);
        src[piece & 1][tid] = nsrc;
        named_bar_sync(1, kThreads);  // and nobody reads the piece before the previous one any more
    };
    constexpr int kPieceStages = kDownPiece / kDownK;
    fetch(0);
    // W_down: rows warp + 8 i of the stage, chunk lane of 8 columns; c hi / lo: rows tid / 8 + 32 i, chunk tid % 8 of 8 tokens
    const uint32_t sm0 = smem_addr(sm);
    const uint32_t wdst = (uint32_t)((lane >> 3) * C::kBlock + swz(warp, lane & 7, 128));  // + 1024 i: 8 rows on
    const uint32_t cdst = (uint32_t)(C::kA + swz(tid >> 3, tid & 7, 128));
    bool ok = true;
    for (int kb = 0; kb < nk; ++kb) {
        const int piece = kb / kPieceStages;
        if (kb % kPieceStages == 0) {
            publish(piece);
            fetch(piece + 1);
        }
        if (ok && kb >= S) ok = tc_wait(&ts.empty[at.st], at.ph ^ 1, ts);
        if (!ok) continue;  // nothing is copied any more, but the barrier in publish() needs every thread
        const uint32_t base = sm0 + at.st * C::kStage;
        const int l0 = kb % kPieceStages * kDownK;
        const int *pj = rowj[piece & 1] + l0, *psrc = src[piece & 1] + l0;
#pragma unroll
        for (int i = 0; i < kDownK / 8; ++i) {
            const int j = pj[warp + 8 * i];
            cp16(base + wdst + 1024 * i, L.wd + (size_t)max(j, 0) * d + n0 + lane * 8, j >= 0 ? 16u : 0u);
        }
#pragma unroll
        for (int i = 0; i < kDownK / 32; ++i) {
            const int j = pj[(tid >> 3) + 32 * i];
            const size_t off = (size_t)(j >= 0 ? psrc[(tid >> 3) + 32 * i] : 0) * kTokPad + (tid & 7) * 8;
            cp16(base + cdst + 4096 * i, L.c_hi + off, j >= 0 ? 16u : 0u);
            cp16(base + cdst + 4096 * i + C::kBlock, L.c_lo + off, j >= 0 ? 16u : 0u);
        }
        cp_arrive(&ts.full[at.st]);
        at.next(S);
    }
    ok = __all_sync(0xffffffffu, tc_wait(&ts.done, 0, ts) && ok);
    cp_wait<0>();
    tc_fence_after();
    // warp w: columns n0 + 128 h + 32 (w % 4) + lane, token tiles w / 4, w / 4 + 2; an empty slice writes zeros
    const int q = warp & 3;
    if (ok) {
        for (int mt = warp >> 2; mt < MT; mt += 2)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t acc = ts.tmem + ((uint32_t)(32 * q) << 16) + 4 * h * C::kAcc + 16 * mt;
                float v[16], w[16];
                tc_ld16(acc + 2 * C::kAcc, w);
                tc_ld16(acc, v);
                if (nk > 1) {  // else the odd accumulators were not written
                    float vo[16], wo[16];
                    tc_ld16(acc + 3 * C::kAcc, wo);
                    tc_ld16(acc + C::kAcc, vo);
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        v[e] += vo[e];
                        w[e] += wo[e];
                    }
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] += w[e];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int t = 16 * mt + e;
                    if (t < L.batch) ps[(size_t)t * d + n0 + 128 * h + 32 * q + lane] = nk > 0 ? v[e] : 0.0f;
                }
            }
    }
    tc_teardown(ts, C::kCols, L.status);
}

// y_t = sum of the slices' partials in slice order (or h_t += y_t), four columns a thread
__global__ void __launch_bounds__(kThreads) k_wide_reduce(const WideLaunch L) {
    // the next kernel may be scheduled at once (it waits before it reads h or writes scratch): 71.5 -> 71.0 us at 64 tokens
    pdl_launch_dependents();
    pdl_wait();
    const size_t n4 = (size_t)L.batch * L.d / 4;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    const float4* p = reinterpret_cast<const float4*>(L.partial) + i;
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    constexpr int kB = 10;  // slices loaded at once (9 at d = 4096)
    for (int b = 0; b < L.ks; b += kB) {
        float4 v[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u)
            v[u] = b + u < L.ks ? __ldcg(p + (size_t)(b + u) * n4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kB; ++u) {
            s.x += v[u].x;
            s.y += v[u].y;
            s.z += v[u].z;
            s.w += v[u].w;
        }
    }
    float* o = (L.residual_out ? L.h : L.y) + 4 * i;
    const float* r = L.residual_out ? o : nullptr;
    const float4 h = r ? make_float4(r[0], r[1], r[2], r[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    s = make_float4(h.x + s.x, h.y + s.y, h.z + s.z, h.w + s.w);
    if ((reinterpret_cast<uintptr_t>(o) & 15u) == 0) {
        *reinterpret_cast<float4*>(o) = s;
    } else {
        o[0] = s.x;
        o[1] = s.y;
        o[2] = s.z;
        o[3] = s.w;
    }
}

// x_t = bf16(h_t / sqrt(mean(h_t^2) + 1e-5)) with x[d-1] = 1 (the stack glue), one CTA per token; the sum
// of squares in a fixed order (per thread, warp tree, warps in order)
constexpr int kNormThreads = 512;
__global__ void __launch_bounds__(kNormThreads) k_norm(int d, const float* h, __nv_bfloat16* xout) {
    __shared__ float red[kNormThreads / kWarp];
    pdl_wait();
    pdl_launch_dependents();
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* hr = h + (size_t)t * d;
    constexpr int kKeep = 8;  // elements a thread keeps for the quotients (the rest are read again)
    float v[kKeep], ss = 0.0f;
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
        const int i = tid + k * kNormThreads;
        v[k] = i < d ? hr[i] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kKeep; ++k) ss = fmaf(v[k], v[k], ss);
    for (int i = tid + kKeep * kNormThreads; i < d; i += kNormThreads) ss = fmaf(hr[i], hr[i], ss);
    ss = warp_sum(ss);
    if (lane == 0) red[warp] = ss;
    __syncthreads();
    float tot = 0.0f;
    for (int w = 0; w < kNormThreads / kWarp; ++w) tot += red[w];
    const float rms = __fsqrt_rn(__fadd_rn(__fdiv_rn(tot, (float)d), 1e-5f));
    auto put = [&](int i, float hv) {
        xout[(size_t)t * d + i] = __float2bfloat16_rn(i == d - 1 ? 1.0f : __fdiv_rn(hv, rms));
    };
#pragma unroll
    for (int k = 0; k < kKeep; ++k)
        if (tid + k * kNormThreads < d) put(tid + k * kNormThreads, v[k]);
    for (int i = tid + kKeep * kNormThreads; i < d; i += kNormThreads) put(i, hr[i]);
}

template <typename K, typename... Args>
cudaError_t launch(K kernel, int grid, int threads, size_t smem, cudaStream_t stream, bool pdl, Args... args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&lc, kernel, args...);
}

// Rows per gate+up tile: one tile per SM, or per SM and wave when the rows
// are more than 128 per SM (a multiple of 16: whole bitmap bytes, whole 8-row
// atoms). 14336 rows on 152 SMs: 96 rows, 150 CTAs (128-row tiles left 40 SMs idle).
int tile_rows(int n_rows, int num_sms) {
    if (n_rows < 1) return 16;
    const int waves = (n_rows + kTcRows * num_sms - 1) / (kTcRows * num_sms);
    const int rows = (n_rows + waves * num_sms - 1) / (waves * num_sms);
    return rows < 16 ? 16 : (rows + 15) / 16 * 16;
}

template <int MT>
cudaError_t run_t(const WideLaunch& L, int num_sms, cudaStream_t stream, bool pdl) {
    const int rows = tile_rows(L.n_rows, num_sms);
    const int stage = 2 * (rows * 128 + GuCfg<MT>::kB);
    // the MMA reads 128 rows from a stage's start: the last stage is followed by as much again
    int stages = (kPipe - kTcRows * 128) / stage;
    if (stages > kMaxStages) stages = kMaxStages;
    const int tiles = (L.n_rows + rows - 1) / rows;
    cudaError_t e = cudaSuccess;
    if (tiles > 0)
        e = launch(k_wide_gate_up<MT>, tiles, kCta, (size_t)stages * stage + kTcRows * 128 + 1024, stream, pdl, L, rows,
                   stages);
    if (e == cudaSuccess)
        e = launch(k_wide_down<MT>, (L.d / kDownCols) * L.ks, kCta, DownCfg<MT>::kBytes, stream, true, L, rows, tiles);
    if (e == cudaSuccess)
        e = launch(k_wide_reduce, (L.batch * L.d / 4 + kThreads - 1) / kThreads, kThreads, 0, stream, true, L);
    return e;
}

template <int MT>
cudaError_t prepare_t() {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(k_wide_gate_up<MT>, at, kPipe + 1024);
    return e == cudaSuccess ? cudaFuncSetAttribute(k_wide_down<MT>, at, DownCfg<MT>::kBytes) : e;
}

}  // namespace

bool wide_supported(int wdtype, int d, int m, int batch) {
    return wdtype == 1 && batch > kMaxPass && batch <= kTokPad && d % kDownCols == 0 && m <= kWideMaxRows;
}

int wide_slices(int d, int num_sms) {
    const int n_tiles = d / kDownCols;
    return n_tiles >= num_sms ? 1 : num_sms / n_tiles;
}

int wide_tiles(int m, int num_sms) {
    // a list of n rows has tiles of tile_rows(n) rows: never more than one per 16 rows, or per SM and wave
    const int waves = (m + kTcRows * num_sms - 1) / (kTcRows * num_sms);
    const int most = waves * num_sms, small = (m + 15) / 16;
    return small < most ? small : most;
}

cudaError_t prepare_wide() {
    cudaError_t e = prepare_t<1>();
    if (e == cudaSuccess) e = prepare_t<2>();
    if (e == cudaSuccess) e = prepare_t<3>();
    if (e == cudaSuccess) e = prepare_t<4>();
    return e;
}

cudaError_t launch_wide(const WideLaunch& L, int num_sms, cudaStream_t stream, bool pdl) {
    switch ((L.batch + 15) / 16) {
        case 1: return run_t<1>(L, num_sms, stream, pdl);
        case 2: return run_t<2>(L, num_sms, stream, pdl);
        case 3: return run_t<3>(L, num_sms, stream, pdl);
        case 4: return run_t<4>(L, num_sms, stream, pdl);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_norm(int d, int batch, const float* h, __nv_bfloat16* xout, cudaStream_t stream, bool pdl) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(batch);
    lc.blockDim = dim3(kNormThreads);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&lc, k_norm, d, h, xout);
}

}  // namespace tsffn
