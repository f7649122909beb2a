// ts_mid.cu -- passes of 3-16 tokens over bf16 rows (Eq. 1 with the dReLU of
// Eq. 2, single FFNs and the grouped experts of an MoE layer), in three
// launches:
//   k_mid_gate_up  persistent, one CTA per SM, each CTA a contiguous range of
//                  8-row chunks: gate rows, union mask, gate-active up rows,
//                  c = w_route g u, bitmaps;
//   k_mid_down     (512 output columns) x (slice of the union both-active
//                  rows) per CTA, gathered W_down rows;
//   k_mid_reduce   the slices added in order into y, or onto the residual.
// Both contractions run on mma.sync m16n8k16 with the weights as the 16-row
// operand and 8 tokens as the columns: at 3-16 tokens the products are far
// below the tensor rate (2 * tokens flop per weight byte) and HBM bounds them.
// Measured at d = 4096, m = 14336 (10% active, calls back to back), against the
// kernels before (one thread issuing a bulk copy per row, then a down kernel
// of 64-byte column slices; at 16 tokens the kernels of ts_wide.cu): 5 tokens
// 96 -> 52 us, 16 tokens 98 -> 79 us, 8 tokens over 8 experts, top-2, 20% active:
// 835 -> 279 us (5.9 TB/s).
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

__device__ __forceinline__ void cp16(void* dst, const void* src, int bytes) {  // 16, or 0: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
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
// in slice order, so results do not depend on timing.
//
// A CTA's chunks go in rounds, and the gate rows of round r (segment G_r) and
// its gate-active up rows (U_r) are streamed in the order G0 G1 U0 G2 U1 ...,
// so the list of the next segment is always known while the present one
// streams and the ring never drains between them.
// At 5 tokens the launch takes 35 us for 195 MB (5.6 TB/s). (Loading 16 rows x
// 32 elements straight into registers ran at 3.7 TB/s: loads that share the
// few scoreboards wait for one another. Pulling the both-active W_down rows
// into L2 at the end of a round changed nothing at 3-16 tokens and cost 28 us
// over 8 experts, whose rows do not fit.)
// ---------------------------------------------------------------------------
constexpr int kStageK = 64;                         // elements of a row per stage
constexpr int kStageBytes = kGroup * kStageK * 2;   // 2 KB
constexpr int kRing = 4;                            // stages in flight per warp
constexpr int kRegStages = 4;                       // stages of a slice whose activations stay in registers
constexpr int kRoundChunks = 8;                     // most chunks per round
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
__device__ __forceinline__ int stage_off(int r, int c) { return r * 128 + ((c ^ (((r & 1) << 2) | ((r >> 1) & 3))) << 4); }

// Segment s of a CTA with n_rounds rounds: its round, and whether it is the gate segment.
__device__ __forceinline__ bool seg_gate(int s, int n_rounds) { return s == 0 || ((s & 1) && s < 2 * n_rounds - 1); }
__device__ __forceinline__ int seg_round(int s, int n_rounds) {
    if (s == 0) return 0;
    if (s == 2 * n_rounds - 1) return n_rounds - 1;
    return (s & 1) ? (s + 1) / 2 : s / 2 - 1;
}

template <int NT, bool XREG>
__global__ void __launch_bounds__(kThreads, 1) k_mid_gate_up(const FfnLaunch a, const MidCfg mc) {
    constexpr int TL = MidShape<NT>::kTiles;
    extern __shared__ __align__(128) unsigned char dyn[];
    MidShared<NT>& sh = *reinterpret_cast<MidShared<NT>*>(dyn);
    unsigned char* ring_all = dyn + (sizeof(MidShared<NT>) + 127) / 128 * 128;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* ring = ring_all + (size_t)warp * mc.ring * kStageBytes;
    float* red = reinterpret_cast<float*>(ring_all + (size_t)kWarps * mc.ring * kStageBytes);  // [groups][kw][16][NT]
    uint4* xf = reinterpret_cast<uint4*>(red + (size_t)kRoundRows * mc.kw * NT);  // !XREG: [TL][2 nst][32]
    const int d = a.d;
    const int n_x = a.route ? a.batch : a.nt;
    const int g = lane / 4, t4 = lane & 3;

    if (tid == 0) {
        mbar_init(&sh.never, 1);
        mbar_fence_init();
        sh.bmask[0] = sh.bmask[1] = 0u;
    }
    // rows known without the previous kernel: the first copies go out before the wait
    const bool early = (a.rows == nullptr || a.rows_ready) && a.route == nullptr;
    if (!early) pdl_wait();
    resolve_experts(a, sh.es);
    pdl_launch_dependents();
    if (tid < kMaxExperts * NT) {
        const int e = tid / NT, t = tid % NT;
        int k_of = -1;
        float w = 0.0f;
        if (a.route == nullptr) {
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

    const int n_chunks = (a.n_rows + kChunk - 1) / kChunk;
    const int n_items = sh.es.n_act * n_chunks;
    const int i0 = (int)((long long)n_items * blockIdx.x / gridDim.x);
    const int i1 = (int)((long long)n_items * (blockIdx.x + 1) / gridDim.x);
    const int n_local = i1 - i0;
    if (n_local == 0) {  // a list shorter than the grid
        if (early) pdl_wait();
        if (tid == 0 && a.ent != nullptr) a.ent_n[blockIdx.x] = 0;
        return;
    }
    // at least three rounds where there are chunks enough, so that every list is ready ahead of its segment
    const int n_rounds = max((n_local + kRoundChunks - 1) / kRoundChunks, min(3, n_local / 2));
    const int n_seg = 2 * n_rounds;

    // the gate rows of round r into the list of its segment s
    auto setup_gate = [&](int s, int r) {
        MidRound<NT>& R = sh.round[r % 3];
        const int base = (int)((long long)n_local * r / n_rounds);
        const int nr = (int)((long long)n_local * (r + 1) / n_rounds) - base;
        if (tid < kRoundRows) {
            const int c = tid / kChunk;
            int j = -1;
            const unsigned char* p = nullptr;
            if (c < nr) {
                const int item = i0 + base + c;
                const int ea = item / n_chunks;
                const int chunk = item - ea * n_chunks;
                const int e = sh.es.act[ea];
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
    auto load_ptrs = [&]() {
        const int n = sh.seg_n[iseg & 1];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = igrp * kGroup + 4 * i + lane / 8;
            const unsigned char* p = r < n ? sh.rowp[iseg & 1][r] : nullptr;
            isz[i] = p ? 16 : 0;
            ip[i] = (p ? p : static_cast<const unsigned char*>(a.ex[0].wg)) + (size_t)(st0 * kStageK + (lane & 7) * 8) * 2;
        }
    };
    // this lane's place in a stage: rows 4 i + lane / 8 are 512 bytes apart, odd i with bit 1 of the chunk flipped
    const int doff = stage_off(lane / 8, lane & 7);
    // copy the next stage, if one is known
    auto issue = [&]() {
        if (ist == 0) {
            while (iseg < seg_ready && igrp * kGroup >= sh.seg_n[iseg & 1]) {
                ++iseg;
                igrp = team;
            }
            if (iseg >= seg_ready) return false;
            load_ptrs();
        }
        unsigned char* dst = ring + islot * kStageBytes;
        // a lane past the end of the rows copies nothing (the address is not read then)
        const bool in = (st0 + ist) * kStageK + (lane & 7) * 8 < d;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cp16(dst + i * 512 + ((i & 1) ? doff ^ 32 : doff), ip[i], in ? isz[i] : 0);
            ip[i] += kStageK * 2;
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
    if (n_rounds > 1) setup_gate(1, 1);
    __syncthreads();
    seg_ready = n_rounds > 1 ? 2 : min(n_seg, 1);
    fill();
    if (early) pdl_wait();
    // the failure-detection test: a wait that can only run out
    if (a.test_stall && tid == 0 && !mbar_wait(&sh.never, 0u)) atomicOr(a.status, kStatusTimeout);

    // activations in operand order; tokens past the pass and elements past d are zero
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(a.x) + (size_t)(a.route ? 0 : a.tok0) * d;
    const bool xvec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
    auto load_x = [&](int q, int b) {  // tile q, 32-element block b of the row
        const int t = 8 * q + g, col = b * 32 + t4 * 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (t < n_x && col < d) {
            const __nv_bfloat16* src = x + (size_t)t * d + col;
            if (xvec) {
                v = *reinterpret_cast<const uint4*>(src);
            } else {
                const unsigned short* h = reinterpret_cast<const unsigned short*>(src);
                v = make_uint4(h[0] | (unsigned)h[1] << 16, h[2] | (unsigned)h[3] << 16, h[4] | (unsigned)h[5] << 16,
                               h[6] | (unsigned)h[7] << 16);
            }
        }
        return v;
    };
    uint4 xr[XREG ? TL : 1][XREG ? 2 * kRegStages : 1];
    if constexpr (XREG) {
#pragma unroll
        for (int q = 0; q < TL; ++q)
#pragma unroll
            for (int b = 0; b < 2 * kRegStages; ++b)
                xr[q][b] = b < 2 * ns ? load_x(q, 2 * st0 + b) : make_uint4(0u, 0u, 0u, 0u);
    } else {
        for (int i = warp; i < TL * 2 * mc.nst; i += kWarps) xf[(size_t)i * kWarp + lane] = load_x(i / (2 * mc.nst), i % (2 * mc.nst));
        __syncthreads();
    }

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
            auto stage = [&](const uint4 (&x0)[TL], const uint4 (&x1)[TL]) {
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
                const unsigned char* sp = ring + cslot * kStageBytes;
                const uint4 w0 = lds128(sp + roff0), w1 = lds128(sp + roff0 + 1024);
                const uint4 v0 = lds128(sp + roff1), v1 = lds128(sp + roff1 + 1024);
                __syncwarp();  // the slot may be refilled
                cslot = cslot + 1 == mc.ring ? 0 : cslot + 1;
                --in_flight;
                issue();
#pragma unroll
                for (int q = 0; q < TL; ++q) {
                    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    mma(acc, w0.x, w1.x, w0.y, w1.y, x0[q].x, x0[q].y);
                    mma(acc, w0.z, w1.z, w0.w, w1.w, x0[q].z, x0[q].w);
                    mma(acc, v0.x, v1.x, v0.y, v1.y, x1[q].x, x1[q].y);
                    mma(acc, v0.z, v1.z, v0.w, v1.w, x1[q].z, x1[q].w);
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum[q][i] += acc[i];
                }
            };
            if constexpr (XREG) {
#pragma unroll
                for (int k = 0; k < kRegStages; ++k) {
                    if (k < ns) {
                        uint4 x0[TL], x1[TL];
#pragma unroll
                        for (int q = 0; q < TL; ++q) {
                            x0[q] = xr[q][2 * k];
                            x1[q] = xr[q][2 * k + 1];
                        }
                        stage(x0, x1);
                    }
                }
            } else {
                for (int k = 0; k < ns; ++k) {
                    uint4 x0[TL], x1[TL];
#pragma unroll
                    for (int q = 0; q < TL; ++q) {
                        x0[q] = xf[((size_t)q * 2 * mc.nst + 2 * (st0 + k)) * kWarp + lane];
                        x1[q] = xf[((size_t)q * 2 * mc.nst + 2 * (st0 + k) + 1) * kWarp + lane];
                    }
                    stage(x0, x1);
                }
            }
            // rows g and g + 8, tokens 2t and 2t + 1 of each tile: [token][16 rows], the
            // halves of the rows swapped for every second pair of tokens (fewer bank conflicts)
            float* o = red + ((size_t)grp * mc.kw + slice) * (kGroup * NT) + 2 * t4 * kGroup + (g ^ ((t4 & 1) << 3));
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float* oi = o + (8 * q + (i & 1)) * kGroup;
                    *((i & 2) ? red + ((oi - red) ^ 8) : oi) = sum[q][i];
                }
        }
        __syncthreads();
        MidRound<NT>& R = sh.round[r % 3];
        // Warp t finishes token t of the segment: lane = row of each 32, so that the bitmaps are ballots.
        const int n_rows = R.n_chunks * kChunk;
        if (warp < n_x) {
            const int t = warp;
            // the slices' sums in slice order
            auto total = [&](int i) {
                const float* p = red + (size_t)(i / kGroup) * mc.kw * (kGroup * NT) + t * kGroup +
                                 ((i % kGroup) ^ (((t >> 1) & 1) << 3));
                float tot = 0.0f;
#pragma unroll 4
                for (int k = 0; k < mc.kw; ++k) tot += p[(size_t)k * (kGroup * NT)];
                return tot;
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
                const int pos = chunk * kChunk + row % kChunk;
                if (!gate && on && pos < a.n_rows)
                    a.cval[((size_t)e * kMaxPass + t) * a.cval_tok_stride + pos] = bk ? sh.wt[e][t] * (gt * ut) : 0.0f;
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
            if (((m[tid / 32] >> (tid % 32)) & 1u) && a.ent != nullptr)
                a.ent[(size_t)i0 * kChunk + n_ent + mask_before(m, tid)] =
                    make_int2(R.jrow[tid], (e << 28) | (chunk * kChunk + tid % kChunk));
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
// Warp (w % 8, w / 8) takes 64 columns and every second step of 16 rows: it
// copies its 16 x 128 bytes of a step with four cp.async instructions of full
// lines into its own ring of kRing stages, and reads them with transposing
// ldmatrix as the MMA's A operand (16 columns x 16 rows). The B operand is c
// (16 rows x 8 tokens), split exactly into three bf16 parts (8 significant bits
// each), so that the product keeps the 24 bits of c; each step's MMAs start
// from zero and are added in fp32. (A weight of infinity times a part that is
// zero gives NaN here, as a token that is not active on the row does in the
// fp32 kernel.)
// ---------------------------------------------------------------------------
constexpr int kDownTile = 512;  // columns per CTA
template <int NT>
constexpr int kDownPiece = NT <= 8 ? 1024 : 512;  // rows resolved at a time

template <int NT>
struct MidDownShared {
    const unsigned char* rowp[kDownPiece<NT>];
    int at[kDownPiece<NT>];       // (expert << 28) | row of the row space
    int start[kMidMaxGrid + 1];   // rows listed by the slice's gate+up CTAs, as a prefix
};

__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

template <int NT>
__global__ void __launch_bounds__(kThreads, 1) k_mid_down(const FfnLaunch a, int n_tiles, int ks, int gu_grid, int masked) {
    constexpr int TL = MidShape<NT>::kTiles;
    constexpr int P = kDownPiece<NT>;
    extern __shared__ __align__(128) unsigned char dyn[];
    MidDownShared<NT>& sh = *reinterpret_cast<MidDownShared<NT>*>(dyn);
    unsigned char* rings = dyn + (sizeof(MidDownShared<NT>) + 127) / 128 * 128;
    uint2* cf = reinterpret_cast<uint2*>(rings + kWarps * kRing * kStageBytes);  // [step][tile][part][32 lanes] B operands
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* ring = rings + warp * kRing * kStageBytes;
    const int g = lane / 4, t4 = lane & 3;
    const int d = a.d;
    const int n_slots = a.route ? a.batch : a.nt;
    const int n0 = (int)(blockIdx.x % (unsigned)n_tiles) * kDownTile;
    const int sl = (int)(blockIdx.x / (unsigned)n_tiles);
    const int c0 = (int)((long long)gu_grid * sl / ks), n_cta = (int)((long long)gu_grid * (sl + 1) / ks) - c0;
    pdl_wait();
    pdl_launch_dependents();
    // the first entry of a gate+up CTA, as k_mid_gate_up splits the items
    int n_act = 1;
    if (a.route != nullptr) {
        unsigned used = 0u;
        for (int t = 0; t < a.batch; ++t)
            for (int k = 0; k < a.top_k; ++k) used |= 1u << a.route[t].sel[k];
        n_act = __popc(used);
    }
    const long long n_items = (long long)n_act * ((a.n_rows + kChunk - 1) / kChunk);
    if (warp == 0) {
        int run = 0;
        for (int b = 0; b < n_cta; b += kWarp) {
            const int v = b + lane < n_cta ? __ldcg(a.ent_n + c0 + b + lane) : 0;
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
    const int total = sh.start[n_cta];

    const int cw = warp & 7, kh = warp >> 3;
    const int col0 = n0 + 64 * cw;
    const int ccol = col0 + (lane & 7) * 8;  // this lane's copies
    const bool ccol_in = ccol < d;
    float sum[4][TL][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < TL; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[j][q][i] = 0.0f;

    for (int s = 0; s < total; s += P) {
        const int n = min(P, total - s);
        const int steps = (n + kGroup - 1) / kGroup;
        if (s > 0) __syncthreads();  // the previous piece is done
        for (int i = tid; i < steps * kGroup; i += kThreads) {
            const unsigned char* p = nullptr;
            int at = 0;
            if (i < n) {
                int lo = 0, hi = n_cta - 1;  // the CTA that listed entry s + i
                while (lo < hi) {
                    const int mid = (lo + hi + 1) / 2;
                    if (sh.start[mid] <= s + i)
                        lo = mid;
                    else
                        hi = mid - 1;
                }
                const long long i0 = n_items * (c0 + lo) / gu_grid;
                const int2 en = __ldcg(a.ent + i0 * kChunk + (s + i - sh.start[lo]));
                at = en.y;
                const int e = (unsigned)en.y >> 28, pos = en.y & 0xfffffff;
                // a mask since the list was made may have left no token on the row
                if (!masked || ((a.ubits[(size_t)e * a.nbytes + pos / 8] >> (pos % 8)) & 1))
                    p = static_cast<const unsigned char*>(a.ex[e].wd) + (size_t)debug_row(en.x, a.m, a.status) * a.row_bytes;
            }
            sh.rowp[i] = p;
            sh.at[i] = at;
        }
        __syncthreads();
        auto issue = [&](int st, int slot) {
            if (st < steps) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = 4 * i + lane / 8;
                    const unsigned char* p = sh.rowp[st * kGroup + r];
                    const bool ok = p != nullptr && ccol_in;
                    cp16(ring + slot * kStageBytes + r * 128 + (((lane & 7) ^ (r & 7)) << 4),
                         ok ? p + (size_t)ccol * 2 : static_cast<const unsigned char*>(a.ex[0].wd), ok ? 16 : 0);
                }
            }
            cp_commit();
        };
#pragma unroll
        for (int u = 0; u < kRing; ++u) issue(kh + 2 * u, u);
        // c in operand order: lane (g, t) holds token g of rows 2t, 2t+1, 2t+8, 2t+9
        for (int i = tid; i < steps * TL * kWarp; i += kThreads) {
            const int ln = i % kWarp, q = i / kWarp % TL, st = i / (kWarp * TL);
            const int tok = 8 * q + ln / 4;
            float c[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int li = st * kGroup + 2 * (ln & 3) + (r & 1) + (r >> 1) * 8;
                const int at = sh.at[li];
                c[r] = sh.rowp[li] != nullptr && tok < n_slots
                           ? __ldcg(a.cval + ((size_t)((unsigned)at >> 28) * kMaxPass + tok) * a.cval_tok_stride + (at & 0xfffffff))
                           : 0.0f;
            }
            uint32_t hi[4], mi[4], lo[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                hi[r] = __float_as_uint(c[r]) & 0xffff0000u;
                const float r1 = hi[r] == 0x7f800000u ? 0.0f : c[r] - __uint_as_float(hi[r]);
                mi[r] = __float_as_uint(r1) & 0xffff0000u;
                lo[r] = __float_as_uint(r1 - __uint_as_float(mi[r]));
            }
            uint2* o = cf + ((size_t)(st * TL + q) * 3) * kWarp + ln;
            o[0] = make_uint2(__byte_perm(hi[0], hi[1], 0x7632), __byte_perm(hi[2], hi[3], 0x7632));
            o[kWarp] = make_uint2(__byte_perm(mi[0], mi[1], 0x7632), __byte_perm(mi[2], mi[3], 0x7632));
            o[2 * kWarp] = make_uint2(__byte_perm(lo[0], lo[1], 0x7632), __byte_perm(lo[2], lo[3], 0x7632));
        }
        __syncthreads();
        int slot = 0;
        for (int st = kh; st < steps; st += 2) {
            cp_wait<kRing - 1>();
            __syncwarp();
            // A: lane addresses row (lane % 8) + 8 (lane / 16), 16-byte chunk 2 j + (lane / 8) % 2
            const int ar = (lane & 7) + ((lane >> 4) << 3);
            const uint32_t sa = smem_u32(ring + slot * kStageBytes) + ar * 128;
            uint32_t w[4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) ldsm4t(sa + (((2 * j + ((lane >> 3) & 1)) ^ (ar & 7)) << 4), w[j]);
            __syncwarp();  // the slot may be refilled
            issue(st + 2 * kRing, slot);
            slot = slot + 1 == kRing ? 0 : slot + 1;
#pragma unroll
            for (int q = 0; q < TL; ++q) {
                uint2 b[3];
#pragma unroll
                for (int x = 0; x < 3; ++x) b[x] = cf[((size_t)(st * TL + q) * 3 + x) * kWarp + lane];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int x = 2; x >= 0; --x) mma(acc, w[j][0], w[j][1], w[j][2], w[j][3], b[x].x, b[x].y);
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum[j][q][i] += acc[i];
                }
            }
        }
        cp_wait<0>();
    }
    // the odd steps' sums onto the even steps', through shared memory: [token][column]
    __syncthreads();
    float* red = reinterpret_cast<float*>(rings);  // [NT][512]
    auto each = [&](auto&& f) {  // this lane's sums: token, column of the tile
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < TL; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    f(sum[j][q][i], 8 * q + 2 * t4 + (i & 1), 64 * cw + 16 * j + g + 8 * (i >> 1));
    };
    if (kh == 1) each([&](float v, int tok, int c) { red[tok * kDownTile + c] = v; });
    __syncthreads();
    if (kh == 0) each([&](float v, int tok, int c) { red[tok * kDownTile + c] = v + red[tok * kDownTile + c]; });
    __syncthreads();
    for (int i = tid; i < n_slots * (kDownTile / 4); i += kThreads) {
        const int tok = i / (kDownTile / 4), c = i % (kDownTile / 4) * 4;
        if (n0 + c < d)
            *reinterpret_cast<float4*>(a.partial + ((size_t)sl * n_slots + tok) * d + n0 + c) =
                *reinterpret_cast<const float4*>(red + tok * kDownTile + c);
    }
}

// y (or the residual) from the slices, in slice order; four columns a thread
constexpr int kRedThreads = 128;
__global__ void __launch_bounds__(kRedThreads) k_mid_reduce(const FfnLaunch a, int ks) {
    // in a stack the next layer's first kernel may be scheduled at once (it waits before it reads h)
    if (a.trigger_early) pdl_launch_dependents();
    pdl_wait();
    if (!a.trigger_early) pdl_launch_dependents();
    const int n_slots = a.route ? a.batch : a.nt;
    const size_t n4 = (size_t)n_slots * a.d / 4;
    const size_t i = (size_t)blockIdx.x * kRedThreads + threadIdx.x;
    if (i >= n4) return;
    const float4* p = reinterpret_cast<const float4*>(a.partial) + i;
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    constexpr int kB = 10;  // slices loaded at once
    for (int b = 0; b < ks; b += kB) {
        float4 v[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) v[u] = b + u < ks ? __ldcg(p + (size_t)(b + u) * n4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kB; ++u) {
            s.x += v[u].x;
            s.y += v[u].y;
            s.z += v[u].z;
            s.w += v[u].w;
        }
    }
    float* o = (a.residual_out ? a.h : a.y) + (size_t)(a.route ? 0 : a.tok0) * a.d + 4 * i;
    const bool vec = (reinterpret_cast<uintptr_t>(o) & 15u) == 0;
    if (a.residual_out) {
        const float4 h = vec ? *reinterpret_cast<const float4*>(o) : make_float4(o[0], o[1], o[2], o[3]);
        s = make_float4(h.x + s.x, h.y + s.y, h.z + s.z, h.w + s.w);
    }
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

// Slices of at least two stages; a ring of kRing stages, fewer for rows so
// long that their activations go to shared memory; ring 0 when it does not fit.
template <int NT>
MidCfg mid_cfg(int d, int optin, bool* xreg, size_t* smem) {
    MidCfg mc;
    mc.nst = (d + kStageK - 1) / kStageK;
    mc.kw = kWarps;
    while (mc.kw > 1 && mc.nst / mc.kw < 2) mc.kw /= 2;
    *xreg = mc.nst <= kWarps * kRegStages;
    const size_t fixed = (sizeof(MidShared<NT>) + 127) / 128 * 128 + (size_t)kRoundRows * mc.kw * NT * sizeof(float) +
                         (*xreg ? 0 : (size_t)MidShape<NT>::kTiles * 2 * mc.nst * kWarp * sizeof(uint4));
    mc.ring = kRing;
    if (fixed + (size_t)kWarps * mc.ring * kStageBytes > (size_t)optin) mc.ring = 1;
    if (fixed + (size_t)kWarps * mc.ring * kStageBytes > (size_t)optin) mc.ring = 0;
    *smem = fixed + (size_t)kWarps * mc.ring * kStageBytes;
    return mc;
}

template <int NT>
constexpr size_t down_smem() {
    return (sizeof(MidDownShared<NT>) + 127) / 128 * 128 + (size_t)kWarps * kRing * kStageBytes +
           (size_t)kDownPiece<NT> / kGroup * MidShape<NT>::kTiles * 3 * kWarp * sizeof(uint2);
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

template <int NT>
cudaError_t gate_up_t(const FfnLaunch& a, int grid, cudaStream_t stream) {
    size_t smem = 0;
    bool xreg = false;
    const MidCfg mc = mid_cfg<NT>(a.d, g_optin, &xreg, &smem);
    if (mc.ring < 1) return cudaErrorInvalidValue;
    return xreg ? launch(k_mid_gate_up<NT, true>, grid, kThreads, smem, stream, a, mc)
                : launch(k_mid_gate_up<NT, false>, grid, kThreads, smem, stream, a, mc);
}

}  // namespace

bool mid_supported(int wdtype, int d, int nt, int optin_smem) {
    size_t smem = 0;
    bool xreg = false;
    if (wdtype != 1 || d % 8 != 0 || nt < 1 || nt > kMidMaxTokens) return false;
    return (nt <= 8 ? mid_cfg<8>(d, optin_smem, &xreg, &smem) : mid_cfg<16>(d, optin_smem, &xreg, &smem)).ring >= 1;
}

cudaError_t prepare_mid(int optin_smem) {
    g_optin = optin_smem;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_mid_gate_up<8, true>, at, optin_smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_gate_up<8, false>, at, optin_smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_gate_up<16, true>, at, optin_smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_gate_up<16, false>, at, optin_smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<8>, at, (int)down_smem<8>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mid_down<16>, at, (int)down_smem<16>());
    return e;
}

cudaError_t launch_mid_gate_up(const FfnLaunch& a, int grid, cudaStream_t stream) {
    const int nt = a.route ? a.batch : a.nt;
    if (nt > kMidMaxTokens || a.norm_from_h) return cudaErrorInvalidValue;
    return nt <= 8 ? gate_up_t<8>(a, grid, stream) : gate_up_t<16>(a, grid, stream);
}

cudaError_t launch_mid_down(const FfnLaunch& a, int num_sms, int partial_rows, int gu_grid, bool masked,
                            cudaStream_t stream) {
    const int nt = a.route ? a.batch : a.nt;
    const int n_tiles = (a.d + kDownTile - 1) / kDownTile;
    // one CTA per SM, within the partial buffer, at least one gate+up CTA's list each
    int ks = num_sms / n_tiles;
    if (ks > partial_rows / nt) ks = partial_rows / nt;
    if (ks > gu_grid) ks = gu_grid;
    if (ks < 1) ks = 1;
    if (nt > kMidMaxTokens || partial_rows < nt || gu_grid > kMidMaxGrid || a.partial == nullptr || a.ent == nullptr)
        return cudaErrorInvalidValue;
    const cudaError_t e =
        nt <= 8 ? launch(k_mid_down<8>, n_tiles * ks, kThreads, down_smem<8>(), stream, a, n_tiles, ks, gu_grid, (int)masked)
                : launch(k_mid_down<16>, n_tiles * ks, kThreads, down_smem<16>(), stream, a, n_tiles, ks, gu_grid, (int)masked);
    if (e != cudaSuccess) return e;
    const size_t n4 = (size_t)nt * a.d / 4;
    return launch(k_mid_reduce, (int)((n4 + kRedThreads - 1) / kRedThreads), kRedThreads, 0, stream, a, ks);
}

}  // namespace tsffn
