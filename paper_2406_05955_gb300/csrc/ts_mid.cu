// ts_mid.cu -- passes of 2-16 tokens over bf16 and INT4 rows (Eq. 1 with the
// dReLU of Eq. 2, single FFNs and the grouped experts of an MoE layer), in
// three launches:
//   k_mid_gate_up  persistent, one CTA per SM, each CTA a contiguous range of
//                  8-row chunks: gate rows, union mask, gate-active up rows,
//                  c = w_route g u, bitmaps;
//   k_mid_down     (512 output columns) x (slice of the union both-active
//                  rows) per CTA, gathered W_down rows;
//   k_mid_reduce   the slices added in order into y, or onto the residual.
// Both contractions run on mma.sync m16n8k16 with the weights as the 16-row
// operand and 8 tokens as the columns: at 2-16 tokens the products are far
// below the tensor rate (2 * tokens flop per weight byte) and HBM bounds them.
// Measured at d = 4096, m = 14336 (10% active, calls back to back), against the
// kernels before (one thread issuing a bulk copy per row, then a down kernel
// of 64-byte column slices; at 16 tokens the kernels of ts_wide.cu): 5 tokens
// 96 -> 51 us, 16 tokens 98 -> 71 us, 8 tokens over 8 experts, top-2, 20% active:
// 721-836 -> 247-292 us, by how many experts the tokens hit. INT4 rows (before: passes of two tokens, each
// reading the weights again): 6 tokens 107 -> 44 us, 16 tokens 284 -> 79 us.
#include <cuda_fp16.h>

#include "ts_kernels.cuh"

namespace tsffn {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / kWarp;
constexpr int kGroup = 16;  // weight rows per MMA
constexpr int kMidMaxGrid = 1024;  // most gate+up CTAs (one per SM)
__device__ __forceinline__ void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                    uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// d = A B + c
__device__ __forceinline__ void mma_from(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1, float c0, float c1, float c2, float c3) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

__device__ __forceinline__ void cp16(void* dst, const void* src, int bytes) {  // 16, or 0: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cp8(void* dst, const void* src, int bytes) {  // 8, or 0: zeros
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// First of n items that share i of `of` shares gets (the shares differ by at most one item).
__device__ __forceinline__ int share_start(int n, int of, int i) { return i * (n / of) + min(i, n % of); }
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// gate + up
//
// The 16 warps are K-slices of the same rows (kw slices; 16 / kw teams share
// out the 16-row groups). A warp copies its own slice of a group in stages of
// 16 rows x 64 elements (four cp.async instructions of four full 128-byte
// lines) into its own ring of kRing stages, so no warp waits on another's
// copies and 128 KB per SM stay in flight; it holds its slice of the
// activations in registers for the whole kernel. Lane (g, t) = (lane / 4,
// lane % 4) reads 16 bytes at element 32 b + 8 t of rows g and g + 8 of a
// stage: an MMA's K index may be permuted as long as both operands agree, so
// these 8 elements serve as the lane's K positions of two MMAs, and the
// activations are loaded in the same order. A stage's four MMAs start from
// zero and are added in fp32 (the tensor core truncates when it accumulates);
// the slices' sums meet in shared memory (red) once per segment and are added
// in a fixed order, so results do not depend on timing.
//
// A CTA's chunks go in rounds, and the gate rows of round r (segment G_r) and
// its gate-active up rows (U_r) are streamed in the order G0 G1 U0 G2 U1 ...,
// so the list of the next segment is always known while the present one
// streams and the ring never drains between them.
// At 5 tokens the launch takes 34 us for 195 MB: 2.3 us until the first
// copies are out, then 6.3 TB/s. A stage of INT4 rows holds four times the weights. Their
// unpacking is 7 ALU instructions a word of 8 codes, 19 cycles of a sub-core an MMA, but no
// more than 6 of 28-34 us at 6 tokens, d = 4096, m = 14336 (670 MMAs a sub-core); start-up,
// the ends of the segments and the tails take the rest. (Loading 16 rows x
// 32 elements straight into registers ran at 3.7 TB/s: loads that share the
// few scoreboards wait for one another. Pulling the both-active W_down rows
// into L2 at the end of a round changed nothing at 3-16 tokens and cost 28 us
// over 8 experts, whose rows do not fit.)
// ---------------------------------------------------------------------------
// A stage is 128 bytes of 16 rows: 64 bf16 weights a row, or 256 INT4 codes and their 8 scales (16 bytes
// a row, behind the codes).
constexpr int kStageRow = 128;
template <bool Q4>
constexpr int kStageK = Q4 ? 256 : 64;  // elements of a row per stage
template <bool Q4>
constexpr int kStageBytes = kGroup * (kStageRow + (Q4 ? 16 : 0));
constexpr int kRing = 4;                            // stages in flight per warp
template <bool Q4>
constexpr int kRegStages = Q4 ? 1 : 4;              // stages of a slice whose activations stay in registers
constexpr int kRoundChunks = 8;                     // most chunks per round
// Fewest rounds of a CTA that has the chunks. Two keep the ring busy but for the end of the gate rows; an
// end of segment costs about 1 us, so more lost: 5 tokens 51.2 / 51.0 / 55.8 us for 2 / 3 / 4 rounds, 16
// tokens 71.4 / 73.1 / 85.2, 6 tokens over INT4 rows 47.6 / 49.0 for 2 / 3.
constexpr int kMinRounds = 2;
constexpr int kRoundRows = kRoundChunks * kChunk;
constexpr int kRoundWords = kRoundRows / 32;
static_assert(kRoundWords == 2, "mask_before");

template <int NT>
struct MidShape {
    static constexpr int kTiles = NT / 8;
};

struct MidCfg {
    int nst;    // stages of a row (the last may be partly past d)
    int kw;     // K slices
    int ring;   // stages in flight per warp (kRing, fewer for long rows)
};

// what is kept of a round from its gate segment's set-up to its end
template <int NT>
struct MidRound {
    int jrow[kRoundRows];         // neuron ids (-1: none)
    float gv[NT][kRoundRows];     // gate pre-activations
    short upos[kRoundRows];       // gate-active rows, in order
    short ce[kRoundChunks];       // the chunks' experts
    int cchunk[kRoundChunks];     // and their chunks of the row space
    unsigned gmask[kRoundWords];  // rows that are gate-active for some token
    int n_chunks;
};

template <int NT>
struct MidShared {
    ExpertSets es;
    uint64_t never;                                // nothing arrives here (FfnLaunch::test_stall)
    const unsigned char* rowp[2][kRoundRows];      // rows of segments s and s + 1 (nullptr: none)
    int seg_n[2];
    MidRound<NT> round[3];
    float uv[NT][kRoundRows];
    unsigned bmask[kRoundWords];        // rows of the round that are both-active for some token
    float wt[kMaxExperts][NT];          // routing weight of token t for expert e
    signed char kidx[kMaxExperts][NT];  // its place in the expert's token list (-1: not routed there)
};

// Word w of a row mask, the rows set before row r of its 64, and all of them.
__device__ __forceinline__ int mask_before(const unsigned (&m)[2], int r) {
    const unsigned below = (1u << (r % 32)) - 1u;
    return r < 32 ? __popc(m[0] & below) : __popc(m[0]) + __popc(m[1] & below);
}

// 16-byte chunk c of row r of a stage: with the row's parity in bit 2, the 8
// lanes of a quarter warp (two rows, four chunks of one half) hit 8 bank groups
__device__ __forceinline__ int q4_off(int r, int c) { return r * kStageRow + ((c ^ (r & 7)) << 4); }  // 8 rows at one chunk
__device__ __forceinline__ int stage_off(int r, int c) { return r * 128 + ((c ^ (((r & 1) << 2) | ((r >> 1) & 3))) << 4); }

// Segment s of a CTA with n_rounds rounds: its round, and whether it is the gate segment.
__device__ __forceinline__ bool seg_gate(int s, int n_rounds) { return s == 0 || ((s & 1) && s < 2 * n_rounds - 1); }
__device__ __forceinline__ int seg_round(int s, int n_rounds) {
    if (s == 0) return 0;
    if (s == 2 * n_rounds - 1) return n_rounds - 1;
    return (s & 1) ? (s + 1) / 2 : s / 2 - 1;
}

template <int NT, bool XREG, bool Q4>
__global__ void __launch_bounds__(kThreads, 1) k_mid_gate_up(const FfnLaunch a, const MidCfg mc) {
    constexpr int TL = MidShape<NT>::kTiles;
    extern __shared__ __align__(128) unsigned char dyn[];
    MidShared<NT>& sh = *reinterpret_cast<MidShared<NT>*>(dyn);
    unsigned char* ring_all = dyn + (sizeof(MidShared<NT>) + 127) / 128 * 128;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int SB = kStageBytes<Q4>;
    unsigned char* ring = ring_all + (size_t)warp * mc.ring * SB;
    float* red = reinterpret_cast<float*>(ring_all + (size_t)kWarps * mc.ring * SB);  // [groups][kw][NT][16]
    const int d = a.d;
    constexpr int kBps = kStageK<Q4> / 32;  // 32-element blocks (INT4: scale groups) per stage
    const int nblk = mc.nst * kBps;
    float* xs = red + (size_t)kRoundRows * mc.kw * NT;  // Q4: [TL][nblk][8] -136 * the blocks' activation sums
    uint4* xf = reinterpret_cast<uint4*>(xs + (Q4 ? (size_t)TL * nblk * 8 : 0));  // !XREG: [TL][nblk][32]
    const int n_x = a.route ? a.batch : a.nt;
    const int g = lane / 4, t4 = lane & 3;

    // rows known without the previous kernel: the first copies go out before the wait
    const bool single = a.route == nullptr;
    const bool early = (a.rows == nullptr || a.rows_ready) && single;
    // (hold_weights: only pulled into L2 before it. 9 tokens, d = 1024, m = 3000: 17.1 us with copies, 17.5 so.)
    const bool hold = NT > kMaxPass && !Q4 && early && a.hold_weights;
    if (!early) pdl_wait();
    if (!single) resolve_experts(a, sh.es);

    const int n_chunks = (a.n_rows + kChunk - 1) / kChunk;
    const int n_items = (single ? 1 : sh.es.n_act) * n_chunks;
    const int i0 = share_start(n_items, (int)gridDim.x, (int)blockIdx.x);
    const int n_local = share_start(n_items, (int)gridDim.x, (int)blockIdx.x + 1) - i0;
    if (n_local == 0) {  // a list shorter than the grid
        pdl_launch_dependents();
        if (early) pdl_wait();
        if (tid == 0 && a.ent != nullptr) a.ent_n[blockIdx.x] = 0;
        return;
    }
    // several rounds where there are chunks enough, so that every list is ready ahead of its segment
    const int n_rounds = max((n_local + kRoundChunks - 1) / kRoundChunks, min(kMinRounds, n_local / 2));
    const int n_seg = 2 * n_rounds;

    // the gate rows of round r into the list of its segment s
    auto setup_gate = [&](int s, int r) {
        MidRound<NT>& R = sh.round[r % 3];
        const int base = share_start(n_local, n_rounds, r);
        const int nr = share_start(n_local, n_rounds, r + 1) - base;
        if (tid < kRoundRows) {
            const int c = tid / kChunk;
            int j = -1;
            const unsigned char* p = nullptr;
            if (c < nr) {
                const int item = i0 + base + c;
                const int ea = single ? 0 : item / n_chunks;
                const int chunk = item - ea * n_chunks;
                const int e = single ? 0 : sh.es.act[ea];
                const int pos = chunk * kChunk + tid % kChunk;
                if (pos < a.n_rows) {
                    j = pos;
                    if (a.rows != nullptr) {
                        const int jj = a.rows[pos];
                        j = (unsigned)jj < (unsigned)a.m && (pos == 0 || a.rows[pos - 1] < jj) ? jj : -1;
                        if (j < 0) atomicOr(a.status, kStatusBadIndex);
                    }
                }
                if (j >= 0)
                    p = static_cast<const unsigned char*>(a.ex[e].wg) +
                        (size_t)debug_row(j, a.m, a.status) * a.row_bytes;
                if (tid % kChunk == 0) {
                    R.ce[c] = (short)e;
                    R.cchunk[c] = chunk;
                }
            }
            R.jrow[tid] = j;
            sh.rowp[s & 1][tid] = p;
            if (tid == 0) {
                R.n_chunks = nr;
                R.gmask[0] = R.gmask[1] = 0u;
                sh.seg_n[s & 1] = nr * kChunk;
            }
        }
    };
    // the gate-active rows of round r into the list of its up segment s
    auto setup_up = [&](int s, int r) {
        MidRound<NT>& R = sh.round[r % 3];
        if (tid < kRoundRows && ((R.gmask[tid / 32] >> (tid % 32)) & 1u)) {
            const int at = mask_before(R.gmask, tid);
            R.upos[at] = (short)tid;
            sh.rowp[s & 1][at] = static_cast<const unsigned char*>(a.ex[R.ce[tid / kChunk]].wu) +
                                 (size_t)debug_row(R.jrow[tid], a.m, a.status) * a.row_bytes;
        }
        if (tid == 0) sh.seg_n[s & 1] = __popc(R.gmask[0]) + __popc(R.gmask[1]);
    };

    // this warp's slice: stages st0 .. st0 + ns - 1 of a row; its team's groups of a segment: team, team + T, ...
    const int slice = warp % mc.kw, team = warp / mc.kw, T = kWarps / mc.kw;
    const int st0 = mc.nst * slice / mc.kw, ns = mc.nst * (slice + 1) / mc.kw - st0;

    // issue cursor: the next stage to copy
    int iseg = 0, igrp = team, ist = 0, islot = 0, seg_ready = 0, in_flight = 0;
    const unsigned char* ip[4];  // rows 4 i + lane / 8 of the group, at this lane's next chunk
    int isz[4];                  // 16, or 0 where the group has no such row
    const unsigned char* isc = nullptr;  // Q4: the scales of row lane of the group (lanes below 16)
    int iscz = 0;
    auto load_ptrs = [&]() {
        const int n = sh.seg_n[iseg & 1];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = igrp * kGroup + 4 * i + lane / 8;
            const unsigned char* p = r < n ? sh.rowp[iseg & 1][r] : nullptr;
            isz[i] = p ? 16 : 0;
            ip[i] = (p ? p : static_cast<const unsigned char*>(a.ex[0].wg)) + (size_t)(st0 * kStageRow + (lane & 7) * 16);
        }
        if constexpr (Q4) {
            const int r = igrp * kGroup + (lane & 15);
            const unsigned char* p = r < n ? sh.rowp[iseg & 1][r] : nullptr;
            iscz = p ? 16 : 0;
            isc = (p ? p : static_cast<const unsigned char*>(a.ex[0].wg)) + d / 2 + st0 * 16;
        }
    };
    // this lane's place in a stage: rows 4 i + lane / 8 are 512 bytes apart, odd i with one bit of the chunk flipped
    const int doff = Q4 ? q4_off(lane / 8, lane & 7) : stage_off(lane / 8, lane & 7);
    // copy the next stage, if one is known
    auto issue = [&]() {
        if (Q4 && ns == 0) return false;
        if (ist == 0) {
            while (iseg < seg_ready && igrp * kGroup >= sh.seg_n[iseg & 1]) {
                ++iseg;
                igrp = team;
            }
            if (iseg >= seg_ready) return false;
            load_ptrs();
        }
        unsigned char* dst = ring + islot * SB;
        // a lane past the end of the rows copies nothing (the address is not read then)
        const bool in = Q4 || (st0 + ist) * kStageK<false> + (lane & 7) * 8 < d;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cp16(dst + i * 512 + ((i & 1) ? doff ^ (Q4 ? 64 : 32) : doff), ip[i], in ? isz[i] : 0);
            ip[i] += kStageRow;
        }
        if constexpr (Q4) {
            if (lane < kGroup) cp16(dst + kGroup * kStageRow + lane * 16, isc, iscz);
            isc += 16;
        }
        cp_commit();
        ++in_flight;
        islot = islot + 1 == mc.ring ? 0 : islot + 1;
        if (++ist == ns) {
            ist = 0;
            igrp += T;
        }
        return true;
    };
    auto fill = [&]() {
        while (in_flight < mc.ring && issue()) {
        }
    };

    setup_gate(0, 0);
    __syncthreads();
    seg_ready = 1;
    if (!hold) {
        fill();
    } else if (team * kGroup < sh.seg_n[0]) {  // this warp's first stages
        load_ptrs();
        const bool ends = (lane & 7) == 0 || (lane & 7) == 7;  // a stage's 128 bytes may lie in two lines
        for (int k = 0; k < min(mc.ring, ns) && (st0 + k) * kStageK<Q4> + (lane & 7) * 8 < d; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (isz[i] && ends) prefetch_l2(ip[i] + k * kStageRow);
    }
    pdl_launch_dependents();
    // the second segment's list, the token tables
    if (n_rounds > 1) setup_gate(1, 1);
    if (tid < kMaxExperts * NT) {
        const int e = tid / NT, t = tid % NT;
        int k_of = -1;
        float w = 0.0f;
        if (single) {
            if (e == 0 && t < a.nt) {
                k_of = t;
                w = 1.0f;
            }
        } else if (e < a.n_experts) {
            for (int k = 0; k < sh.es.ntok[e]; ++k)
                if (sh.es.tok[e][k] == t) {
                    k_of = k;
                    w = sh.es.w[e][k];
                }
        }
        sh.wt[e][t] = w;
        sh.kidx[e][t] = (signed char)k_of;
    }
    if (tid == 0) {
        mbar_init(&sh.never, 1);
        mbar_fence_init();
        sh.bmask[0] = sh.bmask[1] = 0u;
    }
    for (int i = tid; i < (NT - n_x) * kRoundRows; i += kThreads) sh.uv[n_x + i / kRoundRows][i % kRoundRows] = 0.0f;
    __syncthreads();
    seg_ready = min(n_rounds, 2);
    if (hold) pdl_wait();
    fill();
    if (early && !hold) pdl_wait();
    // the failure-detection test: a wait that can only run out
    if (a.test_stall && tid == 0 && !mbar_wait(&sh.never, 0u)) atomicOr(a.status, kStatusTimeout);

    // Activations in operand order; tokens past the pass and elements past d are zero. Lane (g, t) holds, of
    // token g of a tile, the elements 8 t .. 8 t + 7 of a 32-element block, or for INT4 codes 8 s + 2 t
    // and the next for s = 0 .. 3, as the codes of word t of a group lie.
    const int x_tok0 = a.route ? 0 : a.tok0;
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(a.x) + (size_t)x_tok0 * d;
    auto load_x = [&](int q, int b) {  // tile q, block b of the row (XREG: x is 16-byte aligned)
        const int t = 8 * q + g;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (t < n_x && (Q4 || b * 32 + t4 * 8 < d)) {
            const __nv_bfloat16* src = x + (size_t)t * d + b * 32 + (Q4 ? 2 * t4 : 8 * t4);
            if (XREG) {
                if constexpr (Q4) {
                    const uint32_t* w = reinterpret_cast<const uint32_t*>(src);
                    v = make_uint4(w[0], w[4], w[8], w[12]);
                } else {
                    v = *reinterpret_cast<const uint4*>(src);
                }
            } else {
                constexpr int kStep = Q4 ? 8 : 2;
                const unsigned short* u = reinterpret_cast<const unsigned short*>(src);
                v = make_uint4(u[0] | (unsigned)u[1] << 16, u[kStep] | (unsigned)u[kStep + 1] << 16,
                               u[2 * kStep] | (unsigned)u[2 * kStep + 1] << 16, u[3 * kStep] | (unsigned)u[3 * kStep + 1] << 16);
            }
        }
        return v;
    };
    auto put_sum = [&](int q, int b, const uint4& v) {  // Q4: -136 times the block's sum, token g of the tile
        float s = 0.0f;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) s += bf16lo(w[i]) + bf16hi(w[i]);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (t4 == 0) xs[((size_t)q * nblk + b) * 8 + g] = -136.0f * s;
    };
    constexpr int kXB = XREG ? kRegStages<Q4> * kBps : 1;
    uint4 xr[XREG ? TL : 1][kXB];
    if constexpr (XREG) {
#pragma unroll
        for (int q = 0; q < TL; ++q) {
#pragma unroll
            for (int b = 0; b < kXB; ++b)
                xr[q][b] = b < kBps * ns ? load_x(q, kBps * st0 + b) : make_uint4(0u, 0u, 0u, 0u);
            if constexpr (Q4) {
#pragma unroll
                for (int b = 0; b < kXB; ++b)
                    if (b < kBps * ns) put_sum(q, kBps * st0 + b, xr[q][b]);
            }
        }
        if constexpr (Q4) __syncthreads();
    } else {
        for (int i = warp; i < TL * nblk; i += kWarps) {
            const uint4 v = load_x(i / nblk, i % nblk);
            xf[(size_t)i * kWarp + lane] = v;
            if constexpr (Q4) put_sum(i / nblk, i % nblk, v);
        }
        __syncthreads();
    }

    // this lane's first place in a group's sums: token 2 t, row g (the halves of the rows swapped, see below)
    const uint32_t red0 = smem_u32(red) + (uint32_t)((slice * NT + 2 * t4) * kGroup + (g ^ ((t4 & 1) << 3))) * 4;
    const uint32_t magic = a.q4_magic;
    int cslot = 0, n_ent = 0;  // n_ent: both-active rows listed so far (threads below kRoundRows)
    const int roff0 = stage_off(g, t4), roff1 = stage_off(g, 4 + t4);  // rows g (g + 8: 1024 bytes on), both blocks
    for (int s = 0; s < n_seg; ++s) {
        const int n = sh.seg_n[s & 1];
        const int n_grp = (n + kGroup - 1) / kGroup;
        const bool gate = seg_gate(s, n_rounds);
        const int r = seg_round(s, n_rounds);
        for (int grp = team; grp < n_grp; grp += T) {
            float sum[TL][4];
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[q][i] = 0.0f;
            // one stage; xb(q, b): the activations of its block b
            auto stage = [&](int k, auto&& xb) {
                static_assert(kRing == 4, "the waits below");
                if (in_flight == 4)
                    cp_wait<3>();
                else if (in_flight == 3)
                    cp_wait<2>();
                else if (in_flight == 2)
                    cp_wait<1>();
                else
                    cp_wait<0>();
                __syncwarp();  // every lane's copies have landed
                const unsigned char* sp = ring + cslot * SB;
                cslot = cslot + 1 == mc.ring ? 0 : cslot + 1;
                --in_flight;
                if constexpr (!Q4) {
                    const uint4 w0 = lds128(sp + roff0), w1 = lds128(sp + roff0 + 1024);
                    const uint4 v0 = lds128(sp + roff1), v1 = lds128(sp + roff1 + 1024);
                    __syncwarp();  // the slot may be refilled
                    issue();
#pragma unroll
                    for (int q = 0; q < TL; ++q) {
                        const uint4 x0 = xb(q, 0), x1 = xb(q, 1);
                        float p0[4], p1[4], p2[4], p3[4];
                        mma_from(p0, w0.x, w1.x, w0.y, w1.y, x0.x, x0.y, 0.0f, 0.0f, 0.0f, 0.0f);
                        mma_from(p1, w0.z, w1.z, w0.w, w1.w, x0.z, x0.w, 0.0f, 0.0f, 0.0f, 0.0f);
                        mma_from(p2, v0.x, v1.x, v0.y, v1.y, x1.x, x1.y, 0.0f, 0.0f, 0.0f, 0.0f);
                        mma_from(p3, v0.z, v1.z, v0.w, v1.w, x1.z, x1.w, 0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                        for (int i = 0; i < 4; ++i) sum[q][i] += (p0[i] + p1[i]) + (p2[i] + p3[i]);
                    }
                } else {
                    // word t of groups 2 p and 2 p + 1, rows g and g + 8
                    uint32_t cw[kBps / 2][4];
                    const uint32_t ca = smem_u32(sp) + ((lane & 7) + (lane & 8)) * kStageRow;
#pragma unroll
                    for (int p = 0; p < kBps / 2; ++p) ldsm4(ca + (((2 * p + (lane >> 4)) ^ (lane & 7)) << 4), cw[p]);
                    const uint4 s0 = lds128(sp + kGroup * kStageRow + g * 16), s1 = lds128(sp + kGroup * kStageRow + (g + 8) * 16);
                    const uint32_t sw0[4] = {s0.x, s0.y, s0.z, s0.w}, sw1[4] = {s1.x, s1.y, s1.z, s1.w};
                    __syncwarp();  // the slot may be refilled
                    issue();
#pragma unroll
                    for (int p = 0; p < kBps / 2; ++p) {
                        const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&sw0[p]));
                        const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&sw1[p]));
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t wa = cw[p][2 * h], wb = cw[p][2 * h + 1];
                            const uint32_t a0 = q4_frag(wa, magic), a1 = q4_frag(wb, magic), a2 = q4_frag(wa >> 4, magic), a3 = q4_frag(wb >> 4, magic);
                            const uint32_t a4 = q4_frag(wa >> 8, magic), a5 = q4_frag(wb >> 8, magic), a6 = q4_frag(wa >> 12, magic),
                                           a7 = q4_frag(wb >> 12, magic);
                            const float sa = h ? f0.y : f0.x, sb = h ? f1.y : f1.x;
#pragma unroll
                            for (int q = 0; q < TL; ++q) {
                                const uint4 xv = xb(q, 2 * p + h);
                                // start from -136 times the activations' sum: sum (128 + code) x - 136 sum x
                                const float2 c =
                                    *reinterpret_cast<const float2*>(xs + ((size_t)q * nblk + kBps * (st0 + k) + 2 * p + h) * 8 + 2 * t4);
                                float acc[4];
                                mma_from(acc, a0, a1, a2, a3, xv.x, xv.y, c.x, c.y, c.x, c.y);
                                mma(acc, a4, a5, a6, a7, xv.z, xv.w);
                                sum[q][0] = fmaf(sa, acc[0], sum[q][0]);
                                sum[q][1] = fmaf(sa, acc[1], sum[q][1]);
                                sum[q][2] = fmaf(sb, acc[2], sum[q][2]);
                                sum[q][3] = fmaf(sb, acc[3], sum[q][3]);
                            }
                        }
                    }
                }
            };
            if constexpr (XREG) {
#pragma unroll
                for (int k = 0; k < kRegStages<Q4>; ++k)
                    if (k < ns) stage(k, [&](int q, int b) { return xr[q][kBps * k + b]; });
            } else {
                for (int k = 0; k < ns; ++k)
                    stage(k, [&](int q, int b) { return xf[((size_t)q * nblk + kBps * (st0 + k) + b) * kWarp + lane]; });
            }
            // rows g and g + 8, tokens 2t and 2t + 1 of each tile: [token][16 rows], the
            // halves of the rows swapped for every second pair of tokens (fewer bank conflicts)
            const uint32_t o = red0 + (uint32_t)(grp * mc.kw) * (kGroup * NT * 4);
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) sts32(((i & 2) ? o ^ 32u : o) + (8 * q + (i & 1)) * kGroup * 4, sum[q][i]);
        }
        __syncthreads();
        MidRound<NT>& R = sh.round[r % 3];
        // Warp t finishes token t of the segment: lane = row of each 32, so that the bitmaps are ballots.
        const int n_rows = R.n_chunks * kChunk;
        if (warp < n_x) {
            const int t = warp;
            // the slices' sums, in a fixed order
            auto total = [&](int i) {
                const float* p = red + (size_t)(i / kGroup) * mc.kw * (kGroup * NT) + t * kGroup +
                                 ((i % kGroup) ^ (((t >> 1) & 1) << 3));
                constexpr int kS = kGroup * NT;
                if (mc.kw < 8) {
                    float tot = 0.0f;
                    for (int k = 0; k < mc.kw; ++k) tot += p[k * kS];
                    return tot;
                }
                float v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = p[k * kS] + p[(k + 4) * kS];
                if (mc.kw == 16) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] += p[(k + 8) * kS] + p[(k + 12) * kS];
                }
                return (v[0] + v[1]) + (v[2] + v[3]);
            };
            if (!gate) {
                for (int i = lane; i < n; i += kWarp) sh.uv[t][R.upos[i]] = total(i);
                __syncwarp();
            }
            for (int row = lane; row < (n_rows + 31) / 32 * 32; row += kWarp) {
                const bool on = row < n_rows;
                const int c = on ? row / kChunk : 0;
                const int e = R.ce[c], chunk = R.cchunk[c];
                const int k = sh.kidx[e][t];
                const bool live = on && k >= 0 && R.jrow[row] >= 0;
                const float gt = !on ? 0.0f : gate ? total(row) : R.gv[t][row];
                if (gate && on) R.gv[t][row] = gt;
                const bool gk = live && gt > 0.0f;
                const float ut = !gate && gk ? sh.uv[t][row] : 0.0f;  // a gate-active row was in the up segment
                const bool bk = gk && ut > 0.0f;
                const unsigned bits = __ballot_sync(0xffffffffu, gate ? gk : bk);
                if (lane == 0 && bits) atomicOr(gate ? &R.gmask[row / 32] : &sh.bmask[row / 32], bits);
                if (on && k >= 0 && row % kChunk == 0)
                    (gate ? a.gbits : a.bbits)[(size_t)e * a.bits_expert_stride + chunk +
                                               (size_t)(a.bits_tok_base + k) * a.nbytes] = (uint8_t)(bits >> (row % 32));
                if (!gate) {
                    const float c = bk ? sh.wt[e][t] * (gt * ut) : 0.0f;
                    const int pos = chunk * kChunk + row % kChunk;
                    sh.uv[t][row] = c;
                    if (a.entc == nullptr && on && pos < a.n_rows)
                        a.cval[((size_t)e * kMaxPass + t) * a.cval_tok_stride + pos] = c;
                }
            }
        }
        __syncthreads();
        if (!gate && tid < kRoundRows) {
            // the union bytes, and the round's both-active rows onto the CTA's list
            const unsigned m[2] = {sh.bmask[0], sh.bmask[1]};
            const int e = tid < n_rows ? R.ce[tid / kChunk] : 0, chunk = tid < n_rows ? R.cchunk[tid / kChunk] : 0;
            if (tid < n_rows && tid % kChunk == 0) {
                a.ubits[(size_t)e * a.nbytes + chunk] = (uint8_t)(m[tid / 32] >> (tid % 32));
                a.ugbits[(size_t)e * a.nbytes + chunk] = (uint8_t)(R.gmask[tid / 32] >> (tid % 32));
            }
            if (((m[tid / 32] >> (tid % 32)) & 1u) && a.ent != nullptr) {
                const size_t at = (size_t)i0 * kChunk + n_ent + mask_before(m, tid);
                a.ent[at] = make_int2(R.jrow[tid], (e << 28) | (chunk * kChunk + tid % kChunk));
                if (a.entc != nullptr) {
#pragma unroll
                    for (int t = 0; t < NT; t += 4)
                        *reinterpret_cast<float4*>(a.entc + at * NT + t) =
                            make_float4(sh.uv[t][tid], sh.uv[t + 1][tid], sh.uv[t + 2][tid], sh.uv[t + 3][tid]);
                }
            }
            n_ent += __popc(m[0]) + __popc(m[1]);
        }
        // the list of the segment after the next (after the next one's, for the only round)
        const int s2 = n_rounds == 1 ? s + 1 : s + 2;
        if (s2 < n_seg) {
            const int r2 = seg_round(s2, n_rounds);
            if (seg_gate(s2, n_rounds))
                setup_gate(s2, r2);
            else
                setup_up(s2, r2);
        }
        __syncthreads();
        if (tid < kRoundWords) sh.bmask[tid] = 0u;  // used again after the next segment's first barrier
        seg_ready = min(n_seg, s2 + 1);
        fill();  // what a short list left of the ring
    }
    if (tid == 0 && a.ent != nullptr) a.ent_n[blockIdx.x] = n_ent;
}

// ---------------------------------------------------------------------------
// down: partial[s][t][n0 .. n0 + 511] over the both-active rows that the
// gate+up CTAs of slice s listed (CTA order, row order).
//
// The 16 warps are column groups of the tile times phases: a warp takes every
// kPhases-th step of 16 rows of its columns, copies its part of a step with
// cp.async into its own ring, and builds the MMA's A operand from it (16
// columns x 16 rows): bf16 rows (64 columns a warp, full 128-byte lines) by
// transposing ldmatrix; INT4 rows (128 columns a warp) from the codes of two
// rows paired in one register, as code - 8, exact in bf16. The B operand is c
// (16 rows x 8 tokens; for INT4 rows times each row's scale for the 32
// columns), split exactly into three bf16 parts (8 significant bits each), so
// that the product keeps its 24 bits; each step's MMAs start from zero and are
// added in fp32. (An infinite weight gives NaN for a token that is not active on
// the row, as zero times it does in fp32.)
// ---------------------------------------------------------------------------
constexpr int kDownTile = 512;  // columns per CTA
constexpr int kMaxSlices = 40;   // narrow rows: more slices would cost the reduction more than they give
template <int NT>
constexpr int kDownPiece = NT <= 8 ? 1024 : 768;  // rows resolved at a time

template <int NT, bool Q4>
struct MidDownShape {
    static constexpr int kCols = Q4 ? 128 : 64;               // columns per warp
    static constexpr int kPhases = kWarps * kCols / kDownTile;  // 2 or 4
    static constexpr int kRow = Q4 ? 80 : 128;                // bytes of a row in a stage (INT4: 64 of codes, 8 of scales)
    static constexpr int kStage = kGroup * kRow;
    static constexpr int kRing = 4;
    static constexpr int kCRow = NT + 4;  // floats per list row of c: two rows 2t apart start 8 banks apart
    static constexpr int kOperand = kDownPiece<NT> * kCRow * 4;
};

template <int NT>
struct MidDownShared {
    const unsigned char* rowp[kDownPiece<NT>];
    int start[kMidMaxGrid + 1];   // rows listed by the slice's gate+up CTAs, as a prefix
};

// The top 16 bits of v: a bf16 and the rest of v in the lower part. With `keep_rest` the bf16 below instead
// where that rest would be zero, unless v is zero (v >= 0, the difference is as exact).
template <bool keep_rest>
__device__ __forceinline__ uint32_t bf16_part(float v) {
    const uint32_t b = __float_as_uint(v);
    return (keep_rest ? max(b, 1u) - 1u : b) & 0xffff0000u;
}
// c[0 .. 3] as three bf16 parts each, whose sum is c exactly: parts[p] holds (c0, c1) and (c2, c3). For bf16
// weights (all c >= 0) the parts of c > 0 are all above zero, an infinite c has an infinite part, and so an
// infinite weight's products add up to infinity as in fp32. INT4 codes are finite: there only an infinite c counts.
template <bool Q4>
__device__ __forceinline__ void split3(const float (&c)[4], uint2 (&parts)[3]) {
    uint32_t hi[4], mi[4], lo[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        hi[r] = bf16_part<!Q4>(c[r]);
        const float r1 = Q4 && (hi[r] & 0x7fffffffu) == 0x7f800000u ? 0.0f : c[r] - __uint_as_float(hi[r]);
        mi[r] = bf16_part<!Q4>(r1);
        lo[r] = __float_as_uint(r1 - __uint_as_float(mi[r]));
    }
    parts[0] = make_uint2(__byte_perm(hi[0], hi[1], 0x7632), __byte_perm(hi[2], hi[3], 0x7632));
    parts[1] = make_uint2(__byte_perm(mi[0], mi[1], 0x7632), __byte_perm(mi[2], mi[3], 0x7632));
    parts[2] = make_uint2(__byte_perm(lo[0], lo[1], 0x7632), __byte_perm(lo[2], lo[3], 0x7632));
}
// (code - 8) of the two codes at bits 0-3 and 16-19, as bf16 (exact)
__device__ __forceinline__ uint32_t q4_weight(uint32_t v, uint32_t magic) {
    const __nv_bfloat162 k = __halves2bfloat162(__ushort_as_bfloat16(0x4308), __ushort_as_bfloat16(0x4308));  // 136
    const uint32_t p = q4_frag(v, magic);
    const __nv_bfloat162 w = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&p), k);
    return *reinterpret_cast<const uint32_t*>(&w);
}

template <int NT, bool Q4>
__global__ void __launch_bounds__(kThreads, 1) k_mid_down(const FfnLaunch a, int n_tiles, int ks, int gu_grid, int masked) {
    using S = MidDownShape<NT, Q4>;
    const uint32_t magic = a.q4_magic;
    constexpr int TL = MidShape<NT>::kTiles;
    constexpr int P = kDownPiece<NT>;
    constexpr int MT = S::kCols / 16;  // 16-column MMA tiles per warp
    extern __shared__ __align__(128) unsigned char dyn[];
    MidDownShared<NT>& sh = *reinterpret_cast<MidDownShared<NT>*>(dyn);
    unsigned char* rings = dyn + (sizeof(MidDownShared<NT>) + 127) / 128 * 128;
    float* cs = reinterpret_cast<float*>(rings + kWarps * S::kRing * S::kStage);  // c: [list row][kCRow]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* ring = rings + warp * S::kRing * S::kStage;
    const int g = lane / 4, t4 = lane & 3;
    const int d = a.d;
    const int n_slots = a.route ? a.batch : a.nt;
    const int n0 = (int)(blockIdx.x % (unsigned)n_tiles) * kDownTile;
    const int sl = (int)(blockIdx.x / (unsigned)n_tiles);
    const int c0 = share_start(gu_grid, ks, sl), n_cta = share_start(gu_grid, ks, sl + 1) - c0;
    int n_items = (a.n_rows + kChunk - 1) / kChunk;
    int per = n_items / gu_grid;  // items of a gate+up CTA; the first `more` have one more
    pdl_wait();
    pdl_launch_dependents();
    if (a.route != nullptr) {
        unsigned used = 0u;
        for (int t = 0; t < a.batch; ++t)
            for (int k = 0; k < a.top_k; ++k) used |= 1u << a.route[t].sel[k];
        n_items *= __popc(used);
        per = n_items / gu_grid;
    }
    const int more = n_items - per * gu_grid;
    // the first entry of gate+up CTA c0 + i, as k_mid_gate_up splits the items, and the most it can list
    auto first_of = [&](int i) { return ((c0 + i) * per + min(c0 + i, more)) * kChunk; };
    auto most_of = [&](int i) { return (per + (c0 + i < more ? 1 : 0)) * kChunk; };
    auto resolve = [&](const int2& en) -> const unsigned char* {
        const int e = (unsigned)en.y >> 28, pos = en.y & 0xfffffff;
        // a mask since the list was made may have left no token on the row
        if (masked && !((a.ubits[(size_t)e * a.nbytes + pos / 8] >> (pos % 8)) & 1)) return nullptr;
        return static_cast<const unsigned char*>(a.ex[e].wd) + (size_t)debug_row(en.x, a.m, a.status) * a.row_bytes;
    };
    auto put = [&](int i, const unsigned char* p, const float4 (&c)[NT / 4]) {  // list row i of the piece
        sh.rowp[i] = p;
#pragma unroll
        for (int k = 0; k < NT / 4; ++k) *reinterpret_cast<float4*>(cs + i * S::kCRow + 4 * k) = c[k];
    };
    // c of list entry `at` (place `src` of the lists): with the entry, or (masked since) from the masked values
    auto load_c = [&](size_t src, int at, float4 (&c)[NT / 4]) {
#pragma unroll
        for (int k = 0; k < NT / 4; ++k) {
            if (a.entc != nullptr) {
                c[k] = __ldcg(reinterpret_cast<const float4*>(a.entc + src * NT) + k);
            } else {
                float v[4];
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    v[x] = 4 * k + x < n_slots ? __ldcg(a.cval + ((size_t)((unsigned)at >> 28) * kMaxPass + 4 * k + x) * a.cval_tok_stride +
                                                        (at & 0xfffffff))
                                               : 0.0f;
                c[k] = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
    };
    // Lists short enough for one piece whatever their counts are read whole, together with the counts (one
    // memory round trip instead of two); places past a CTA's count are dropped.
    const int cap = (per + (more > 0 ? 1 : 0)) * kChunk;  // most entries of one gate+up CTA
    // the count of gate+up CTA c0 + i, held to what it can list of this row space: a replayed graph may have left
    // the lists of a longer one
    auto count = [&](int i) { return min(__ldcg(a.ent_n + c0 + i), most_of(i)); };
    const bool whole = n_cta <= kWarp && cap * n_cta <= P && a.entc != nullptr;
    int total = 0;
    if (whole) {
        constexpr int kEach = (P + kThreads - 1) / kThreads;
        int2 en[kEach];
        float4 c[kEach][NT / 4];
        int of[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            const int i = tid + u * kThreads;
            of[u] = i / max(cap, 1);
            en[u] = make_int2(0, 0);
#pragma unroll
            for (int k = 0; k < NT / 4; ++k) c[u][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (of[u] < n_cta) {
                const int first = first_of(of[u]), idx = i - of[u] * cap;
                if (first + idx < n_items * kChunk) {
                    en[u] = __ldcg(a.ent + first + idx);
                    load_c((size_t)first + idx, 0, c[u]);
                }
            }
        }
        const int cnt = lane < n_cta ? count(lane) : 0;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        total = __shfl_sync(0xffffffffu, incl, kWarp - 1);
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            const int from = min(of[u], kWarp - 1);
            const int n_of = __shfl_sync(0xffffffffu, cnt, from), start = __shfl_sync(0xffffffffu, incl - cnt, from);
            const int idx = tid + u * kThreads - of[u] * cap;
            if (of[u] < n_cta && idx < n_of) put(start + idx, resolve(en[u]), c[u]);
        }
    } else {
        if (warp == 0) {
            int run = 0;
            for (int b = 0; b < n_cta; b += kWarp) {
                const int v = b + lane < n_cta ? count(b + lane) : 0;
                int incl = v;
#pragma unroll
                for (int o = 1; o < kWarp; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += u;
                }
                if (b + lane < n_cta) sh.start[b + lane] = run + incl - v;
                run += __shfl_sync(0xffffffffu, incl, kWarp - 1);
            }
            if (lane == 0) sh.start[n_cta] = run;
        }
        __syncthreads();
        total = sh.start[n_cta];
    }

    constexpr int kGroups = kDownTile / S::kCols;  // column groups
    const int cw = warp % kGroups, kh = warp / kGroups;
    const int col0 = n0 + S::kCols * cw;
    float sum[MT][TL][4];
#pragma unroll
    for (int j = 0; j < MT; ++j)
#pragma unroll
        for (int q = 0; q < TL; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[j][q][i] = 0.0f;

    for (int s = 0; s < total; s += P) {
        const int n = min(P, total - s);
        const int steps = (n + kGroup - 1) / kGroup;
        if (s > 0) __syncthreads();  // the previous piece is done
        if (!whole) {
            for (int i = tid; i < n; i += kThreads) {
                int lo = 0, hi = n_cta - 1;  // the CTA that listed entry s + i
                while (lo < hi) {
                    const int mid = (lo + hi + 1) / 2;
                    if (sh.start[mid] <= s + i)
                        lo = mid;
                    else
                        hi = mid - 1;
                }
                const size_t src = (size_t)first_of(lo) + (s + i - sh.start[lo]);
                const int2 en = __ldcg(a.ent + src);
                float4 c[NT / 4];
                load_c(src, en.y, c);
                put(i, resolve(en), c);
            }
        }
        if (tid < steps * kGroup - n) {
            const float4 zero[NT / 4] = {};
            put(n + tid, nullptr, zero);
        }
        __syncthreads();
        auto issue = [&](int st, int slot) {
            if (st < steps) {
                unsigned char* dst = ring + slot * S::kStage;
                const unsigned char* none = static_cast<const unsigned char*>(a.ex[0].wd);
                if constexpr (!Q4) {
                    const int col = col0 + (lane & 7) * 8;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = 4 * i + lane / 8;
                        const unsigned char* p = sh.rowp[st * kGroup + r];
                        const bool ok = p != nullptr && col < d;
                        cp16(dst + r * S::kRow + (((lane & 7) ^ (r & 7)) << 4), ok ? p + (size_t)col * 2 : none, ok ? 16 : 0);
                    }
                } else {
                    const int col = col0 + (lane & 3) * 32;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int r = 8 * i + lane / 4;
                        const unsigned char* p = sh.rowp[st * kGroup + r];
                        const bool ok = p != nullptr && col < d;
                        cp16(dst + r * S::kRow + (lane & 3) * 16, ok ? p + col / 2 : none, ok ? 16 : 0);
                    }
                    if (lane < kGroup) {  // four scales (d is a multiple of the 128 columns)
                        const unsigned char* p = sh.rowp[st * kGroup + lane];
                        const bool ok = p != nullptr && col0 < d;
                        cp8(dst + lane * S::kRow + 64, ok ? p + d / 2 + col0 / 16 : none, ok ? 8 : 0);
                    }
                }
            }
            cp_commit();
        };
#pragma unroll
        for (int u = 0; u < S::kRing; ++u) issue(kh + S::kPhases * u, u);
        int slot = 0;
        for (int st = kh; st < steps; st += S::kPhases) {
            cp_wait<S::kRing - 1>();
            __syncwarp();
            const unsigned char* sp = ring + slot * S::kStage;
            auto next = [&]() {
                __syncwarp();  // the slot may be refilled
                issue(st + S::kPhases * S::kRing, slot);
                slot = slot + 1 == S::kRing ? 0 : slot + 1;
            };
            // two (INT4) or four column tiles j0 .. of A times B, onto the sums
            auto products = [&](int j, const uint32_t (&w)[4], int q, const uint2 (&b)[3]) {
                float acc[4];
                mma_from(acc, w[0], w[1], w[2], w[3], b[2].x, b[2].y, 0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int x = 1; x >= 0; --x) mma(acc, w[0], w[1], w[2], w[3], b[x].x, b[x].y);
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[j][q][i] += acc[i];
            };
            float cv[TL][4];  // c of token g and rows 2t, 2t+1, 2t+8, 2t+9 of the step
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    cv[q][r] = cs[(st * kGroup + 2 * t4 + (r & 1) + (r >> 1) * 8) * S::kCRow + 8 * q + g];
            if constexpr (!Q4) {
                // A: lane addresses row (lane % 8) + 8 (lane / 16), 16-byte chunk 2 j + (lane / 8) % 2
                const int ar = (lane & 7) + ((lane >> 4) << 3);
                const uint32_t sa = smem_u32(sp) + ar * S::kRow;
                uint32_t w[MT][4];
#pragma unroll
                for (int j = 0; j < MT; ++j) ldsm4t(sa + (((2 * j + ((lane >> 3) & 1)) ^ (ar & 7)) << 4), w[j]);
                next();
#pragma unroll
                for (int q = 0; q < TL; ++q) {
                    uint2 b[3];
                    split3<false>(cv[q], b);
#pragma unroll
                    for (int j = 0; j < MT; ++j) products(j, w[j], q, b);
                }
            } else {
                // rows 2t, 2t+1, 2t+8, 2t+9: half word g of each group of 32 columns (columns 8 s + g at nibble s), scales
                uint32_t cw4[4][4];
                float sc[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const unsigned char* rp = sp + (2 * t4 + (r & 1) + (r >> 1) * 8) * S::kRow;
#pragma unroll
                    for (int p = 0; p < 4; ++p) cw4[r][p] = *reinterpret_cast<const uint32_t*>(rp + p * 16 + (g >> 1) * 4);
                    const uint2 h = *reinterpret_cast<const uint2*>(rp + 64);
                    const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&h.x));
                    const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&h.y));
                    sc[r][0] = f0.x;
                    sc[r][1] = f0.y;
                    sc[r][2] = f1.x;
                    sc[r][3] = f1.y;
                }
                next();
                const uint32_t sel = (g & 1) ? 0x7632 : 0x5410;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint32_t v01 = __byte_perm(cw4[0][p], cw4[1][p], sel), v23 = __byte_perm(cw4[2][p], cw4[3][p], sel);
                    uint32_t w[2][4];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        w[j][0] = q4_weight(v01 >> (8 * j), magic);
                        w[j][1] = q4_weight(v01 >> (8 * j + 4), magic);
                        w[j][2] = q4_weight(v23 >> (8 * j), magic);
                        w[j][3] = q4_weight(v23 >> (8 * j + 4), magic);
                    }
#pragma unroll
                    for (int q = 0; q < TL; ++q) {
                        const float cr[4] = {cv[q][0] * sc[0][p], cv[q][1] * sc[1][p], cv[q][2] * sc[2][p], cv[q][3] * sc[3][p]};
                        uint2 b[3];
                        split3<true>(cr, b);
                        products(2 * p, w[0], q, b);
                        products(2 * p + 1, w[1], q, b);
                    }
                }
            }
        }
        cp_wait<0>();
    }
    // the phases' sums in order, through shared memory: [phase - 1][token][column]
    __syncthreads();
    float* red = reinterpret_cast<float*>(rings);
    auto each = [&](auto&& f) {  // this lane's sums: token, column of the tile
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int c = Q4 ? 32 * (j / 2) + 16 * (j % 2) + 8 * (i >> 1) + g : 16 * j + g + 8 * (i >> 1);
                    f(sum[j][q][i], (8 * q + 2 * t4 + (i & 1)) * kDownTile + S::kCols * cw + c);
                }
    };
    if (kh > 0) each([&](float v, int at) { red[(kh - 1) * NT * kDownTile + at] = v; });
    __syncthreads();
    if (kh == 0)
        each([&](float v, int at) {
#pragma unroll
            for (int p = 0; p < S::kPhases - 1; ++p) v += red[p * NT * kDownTile + at];
            red[at] = v;
        });
    __syncthreads();
    for (int i = tid; i < n_slots * (kDownTile / 4); i += kThreads) {
        const int tok = i / (kDownTile / 4), c = i % (kDownTile / 4) * 4;
        if (n0 + c < d)
            *reinterpret_cast<float4*>(a.partial + ((size_t)sl * n_slots + tok) * d + n0 + c) =
                *reinterpret_cast<const float4*>(red + tok * kDownTile + c);
    }
}

// y (or the residual) from the slices: a warp takes 32 columns (8 lanes of four) and its four groups of 8
// lanes every fourth slice each, so that few loads follow one another; the groups' sums are added in a
// fixed order.
constexpr int kRedThreads = 128;
__global__ void __launch_bounds__(kRedThreads) k_mid_reduce(const FfnLaunch a, int ks) {
    // in a stack the next layer's first kernel may be scheduled at once (it waits before it reads h)
    if (a.trigger_early) pdl_launch_dependents();
    pdl_wait();
    if (!a.trigger_early) pdl_launch_dependents();
    const int n_slots = a.route ? a.batch : a.nt;
    const size_t n4 = (size_t)n_slots * a.d / 4;
    const int lane = threadIdx.x & 31, grp = lane / 8;
    const size_t i = ((size_t)blockIdx.x * (kRedThreads / kWarp) + threadIdx.x / kWarp) * 8 + (lane & 7);
    const bool in = i < n4;
    float* o = (a.residual_out ? a.h : a.y) + (size_t)(a.route ? 0 : a.tok0) * a.d + 4 * i;
    const bool vec = (reinterpret_cast<uintptr_t>(o) & 15u) == 0;
    float4 h = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (in && a.residual_out && grp == 0) h = vec ? *reinterpret_cast<const float4*>(o) : make_float4(o[0], o[1], o[2], o[3]);
    const float4* p = reinterpret_cast<const float4*>(a.partial) + (in ? i : 0);
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    constexpr int kB = 5;  // slices a group loads at once: one round for the 19 slices of d = 4096
    for (int b = grp; b < ks; b += 4 * kB) {
        float4 v[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u)
            v[u] = b + 4 * u < ks ? __ldcg(p + (size_t)(b + 4 * u) * n4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kB; ++u) {
            s.x += v[u].x;
            s.y += v[u].y;
            s.z += v[u].z;
            s.w += v[u].w;
        }
    }
#pragma unroll
    for (int m = 8; m <= 16; m *= 2) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, m);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, m);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, m);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, m);
    }
    if (!in || grp != 0) return;
    if (a.residual_out) s = make_float4(h.x + s.x, h.y + s.y, h.z + s.z, h.w + s.w);
    if (vec) {
        *reinterpret_cast<float4*>(o) = s;
    } else {
        o[0] = s.x;
        o[1] = s.y;
        o[2] = s.z;
        o[3] = s.w;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int g_optin = 0;

// Slices of at least two stages (bf16), or of at most one (INT4, whose stages
// hold four times the weights; a slice may then be empty); a ring of up to kRing stages; the activations
// in shared memory when a slice of them does not fit the registers; ring 0
// when nothing fits.
template <int NT, bool Q4>
MidCfg mid_cfg(int d, int optin, bool* xreg, size_t* smem) {
    // (*xreg on entry: whether registers may hold the activations)
    MidCfg mc;
    mc.nst = (d + kStageK<Q4> - 1) / kStageK<Q4>;
    mc.kw = kWarps;
    while (mc.kw > 1 && (Q4 ? mc.nst <= mc.kw / 2 : mc.nst < 2 * mc.kw)) mc.kw /= 2;
    *xreg = *xreg && (mc.nst + mc.kw - 1) / mc.kw <= kRegStages<Q4>;
    const size_t nblk = (size_t)mc.nst * (kStageK<Q4> / 32), tiles = MidShape<NT>::kTiles;
    const size_t fixed = (sizeof(MidShared<NT>) + 127) / 128 * 128 + (size_t)kRoundRows * mc.kw * NT * sizeof(float) +
                         (Q4 ? tiles * nblk * 8 * sizeof(float) : 0) + (*xreg ? 0 : tiles * nblk * kWarp * sizeof(uint4));
    mc.ring = kRing;
    while (mc.ring > 0 && fixed + (size_t)kWarps * mc.ring * kStageBytes<Q4> > (size_t)optin) --mc.ring;
    *smem = fixed + (size_t)kWarps * mc.ring * kStageBytes<Q4>;
    return mc;
}

template <int NT, bool Q4>
constexpr size_t down_smem() {
    using S = MidDownShape<NT, Q4>;
    const size_t stream = (size_t)kWarps * S::kRing * S::kStage + S::kOperand;
    const size_t sums = (size_t)(S::kPhases - 1) * NT * kDownTile * sizeof(float);
    return (sizeof(MidDownShared<NT>) + 127) / 128 * 128 + (stream > sums ? stream : sums);
}

template <typename K, typename... Args>
cudaError_t launch(K kernel, int grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, args...);
}

template <int NT, bool Q4>
cudaError_t gate_up_t(const FfnLaunch& a, int grid, cudaStream_t stream) {
    size_t smem = 0;
    bool xreg = (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0;  // 16-byte loads
    const MidCfg mc = mid_cfg<NT, Q4>(a.d, g_optin, &xreg, &smem);
    if (mc.ring < 1) return cudaErrorInvalidValue;
    return xreg ? launch(k_mid_gate_up<NT, true, Q4>, grid, kThreads, smem, stream, a, mc)
                : launch(k_mid_gate_up<NT, false, Q4>, grid, kThreads, smem, stream, a, mc);
}

template <int NT, bool Q4>
cudaError_t prepare_gate_up_t(int optin) {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(k_mid_gate_up<NT, true, Q4>, at, optin);
    return e == cudaSuccess ? cudaFuncSetAttribute(k_mid_gate_up<NT, false, Q4>, at, optin) : e;
}

}  // namespace

bool mid_supported(int wdtype, int d, int nt, bool x_aligned, int optin_smem) {
    size_t smem = 0;
    bool xreg = x_aligned;
    if (nt < 1 || nt > kMidMaxTokens || (wdtype == 2 ? d % kStageK<true> != 0 : wdtype != 1 || d % 8 != 0)) return false;
    if (wdtype == 2)
        return (nt <= 8 ? mid_cfg<8, true>(d, optin_smem, &xreg, &smem) : mid_cfg<16, true>(d, optin_smem, &xreg, &smem)).ring >= 1;
    return (nt <= 8 ? mid_cfg<8, false>(d, optin_smem, &xreg, &smem) : mid_cfg<16, false>(d, optin_smem, &xreg, &smem)).ring >= 1;
}

cudaError_t prepare_mid(int optin_smem) {
    g_optin = optin_smem;
    cudaError_t e = prepare_gate_up_t<8, false>(optin_smem);
    if (e == cudaSuccess) e = prepare_gate_up_t<16, false>(optin_smem);
    if (e == cudaSuccess) e = prepare_gate_up_t<8, true>(optin_smem);
    if (e == cudaSuccess) e = prepare_gate_up_t<16, true>(optin_smem);
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<8, false>, at, (int)down_smem<8, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<16, false>, at, (int)down_smem<16, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<8, true>, at, (int)down_smem<8, true>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<16, true>, at, (int)down_smem<16, true>());
    return e;
}

cudaError_t launch_mid_gate_up(const FfnLaunch& a, int wdtype, int grid, cudaStream_t stream) {
    const int nt = a.route ? a.batch : a.nt;
    const bool q4 = wdtype == 2;
    if (nt > kMidMaxTokens || (a.norm_from_h)) return cudaErrorInvalidValue;
    if (q4) return nt <= 8 ? gate_up_t<8, true>(a, grid, stream) : gate_up_t<16, true>(a, grid, stream);
    return nt <= 8 ? gate_up_t<8, false>(a, grid, stream) : gate_up_t<16, false>(a, grid, stream);
}

cudaError_t launch_mid_down(const FfnLaunch& a, int wdtype, int num_sms, int partial_rows, int gu_grid, bool masked,
                            cudaStream_t stream) {
    const int nt = a.route ? a.batch : a.nt;
    const int n_tiles = (a.d + kDownTile - 1) / kDownTile;
    // one CTA per SM, within the partial buffer, at least one gate+up CTA's list each
    int ks = num_sms / n_tiles;
    if (ks > partial_rows / nt) ks = partial_rows / nt;
    if (ks > gu_grid) ks = gu_grid;
    if (ks > kMaxSlices) ks = kMaxSlices;
    if (ks < 1) ks = 1;
    if (nt > kMidMaxTokens || partial_rows < nt || gu_grid > kMidMaxGrid || a.partial == nullptr || a.ent == nullptr || (!masked && a.entc == nullptr))
        return cudaErrorInvalidValue;
    const int grid = n_tiles * ks;
    const int mk = masked ? 1 : 0;
    cudaError_t e;
    if (wdtype == 2)
        e = nt <= 8 ? launch(k_mid_down<8, true>, grid, kThreads, down_smem<8, true>(), stream, a, n_tiles, ks, gu_grid, mk)
                    : launch(k_mid_down<16, true>, grid, kThreads, down_smem<16, true>(), stream, a, n_tiles, ks, gu_grid, mk);
    else
        e = nt <= 8 ? launch(k_mid_down<8, false>, grid, kThreads, down_smem<8, false>(), stream, a, n_tiles, ks, gu_grid, mk)
                    : launch(k_mid_down<16, false>, grid, kThreads, down_smem<16, false>(), stream, a, n_tiles, ks, gu_grid, mk);
    if (e != cudaSuccess) return e;
    const size_t n4 = (size_t)nt * a.d / 4;
    constexpr int kPerCta = kRedThreads / 4;  // float4 columns
    return launch(k_mid_reduce, (int)((n4 + kPerCta - 1) / kPerCta), kRedThreads, 0, stream, a, ks);
}

}  // namespace tsffn
