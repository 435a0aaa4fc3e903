// chain: the chunk form in ONE kernel without any hand-off through memory, on warp-level tensor-core products.
//
// A sequence is walked in blocks of up to 64 rows (64 / r tokens).  From Theorem 3.2, with rows m, S the state before the block:
//     T  = (I + Mstrict (.) (diag(beta) K K^T))^{-1} diag(beta)                      (does not depend on S)
//     P  = (Q K^T) (.) Mincl                                                         (does not depend on S)
//     U' = T (V - K S^T),       O = Q S^T + P U',       S <- S + U'^T K
// i.e. W and Uh are never formed: T is applied to V - K S^T instead.  Of the block's operations only three products depend on
// S one after another, and their operands fit the register layout of mma.sync: with S held as [j][i] accumulators, S K^T,
// then T applied, then the update are each "registers times shared memory", and the accumulator of one product, packed
// to fp16, is the A operand of the next.  So a warp carries 16 rows j of S through the whole sequence without exchanging
// anything with other warps: the serial step has no barrier, no shared-memory round trip and no tensor-memory latency.
//
//   chain warps   16 rows j of S each (IS = 2: two warps share the 16 rows, each holds half of the columns i; they add
//                 their halves of S K^T and Q S^T through shared memory once per block)
//   prep warps    teams of four: K, Q -> fp16 in place, G = K K^T, the inverse, P; a few blocks ahead
// A stage of shared memory holds what the chain needs of one block: K, Q (fp16), T, P (fp16), V (bf16 as it came).
//
// What bounds it: where every SM has a CTA (d = 128, r = 2, 128 columns per CTA) a block of 32 tokens takes 6.5 k cycles, of
// which the shared-memory pipe is busy for 80 % and the mma.sync pipe for 58 %; with few CTAs it is the latency of the chain's
// dependent products (1.8 us a block at d = 128, 1.3 at 64).  Measured (kernel time, against the tcgen05 kernels in two
// launches or one): 256 sequences of 1024 tokens, d = 128, r = 2: 0.23 ms against 0.63; 128 sequences of 4096, d = 64, r = 4: 0.34
// against 0.93; 48 sequences of 1999, 64 x 128, r = 3: 0.145 against 0.33.  Measured and not taken: chain warps of 32 rows (half the
// shared-memory reads, but one such warp per scheduler does not hide its own latencies: 0.31 ms at the first size), fragments
// requested two to six ahead by hand (0.243), G from the bf16 tiles with the conversion after it (0.27).  Where the tcgen05 kernel
// in one launch has few sequences and enough SMs to build flows ahead (d = 128), it is the faster one: see the estimates.
//
// Range: V - K S^T and U' are packed to fp16 like every other operand, and K S^T reaches sqrt(d_k) times the largest entry of S, so
// that a state well inside fp16's 65504 can overflow them.  What overflows leaves its row of S infinite or NaN to the end of the walk
// (infinity times anything is infinite or NaN), so one look at each row when the walk is over finds it and the blocks pay nothing:
// the warp then walks its 16 rows once more, token by token in fp32 (walk_fp32).
//
// The inverse: warp i of a team owns rows 16 i .. 16 i + 15.  D_i = (I + A_ii)^{-1} by its Neumann product and
// E_ij = D_i A_ij in registers, then X_ij = -sum_k E_ik X_kj row block by row block (three exchanges through shared memory).
#include <float.h>

#include <atomic>

#include "pf_common.cuh"
#include "pf_tc.cuh"
#include "pf_tc_prims.cuh"

namespace pf {

using namespace tc;

namespace {

constexpr int NB = 64;               // rows per block

struct ChainMaps {
    CUtensorMap q, k, v;
};

struct ChainGeo {
    int L, d_v, nblk;
    int nseg, seg_blk;  // segments per sequence (1: none) and blocks per segment
    int rm;             // strict-mask group size (Problem::mask_group)
    int exact;          // PF_STEP_EXACT
    int clear;          // set the status word to 0
    const __nv_bfloat16 *q, *k, *v, *beta;      // the inputs once more, for walk_fp32
    const float* S0;
    float *O, *S_final;
};

__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// (a predicated store, not a branch: a branch would keep the compiler from moving anything across it)
__device__ __forceinline__ void store2_if(float* p, float x, float y, bool pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.global.v2.f32 [%0], {%1, %2};\n\t}" ::"l"(p), "f"(x), "f"(y),
                 "r"((unsigned)pred));
}
__device__ __forceinline__ void store_h2_if(__half* p, uint32_t x, bool pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.u32 [%0], %1;\n\t}" ::"l"(p), "r"(x), "r"((unsigned)pred));
}
// eight bf16 -> eight fp16 (sign: 0x80008000 to negate them)
__device__ __forceinline__ uint4 bf16_to_half8(uint4 x, uint32_t sign) {
    uint32_t* w = (uint32_t*)&x;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = pack_h2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u)) ^ sign;
    return x;
}

template <int DK, int R, int JS>
struct ChainSmem {
    static constexpr int C = NB / R;                              // tokens per block
    static constexpr int CP = (C + 15) / 16 * 16;                 // ... in tiles of 16
    static constexpr int k_bytes = NB * DK * 2, q_bytes = CP * DK * 2;
    static constexpr int t_bytes = NB * 128, p_bytes = CP * 128, v_bytes = NB * JS * 2;
    static constexpr int k_off = 0, q_off = k_off + k_bytes, t_off = q_off + q_bytes, p_off = t_off + t_bytes, v_off = p_off + p_bytes;
    static constexpr int stage = v_off + v_bytes;
    static constexpr int tx_bytes = k_bytes + C * DK * 2 + v_bytes;         // what the copies of a block bring
};

template <int DK, int R, int JS, int IS, int TEAMS, int NS>
struct ChainCfg {
    using SM = ChainSmem<DK, R, JS>;
    static constexpr int NCW = JS / 16 * IS;                      // chain warps
    static constexpr int threads = 32 * NCW + 128 * TEAMS;
    static constexpr int xs_off = NS * SM::stage;                 // per team: X (unscaled) while it is being formed
    static constexpr int beta_off = xs_off + TEAMS * NB * 128;    // per team: 64 step sizes, of two blocks in turn
    // IS = 2: partial sums on their way to the other warp of the pair, [pair][parity][warp][thread-linear 16-byte pieces]
    static constexpr int x_piece = 8 + SM::CP / 16;               // 16-byte pieces per thread: 32 of S K^T, 4 per 16 tokens of Q S^T
    static constexpr int ex_off = beta_off + TEAMS * 512;
    static constexpr int ex_bytes = IS == 2 ? (JS / 16) * 2 * 2 * x_piece * 512 : 0;
    static constexpr int total = ex_off + ex_bytes;
};
// as many stages as fit, up to six
template <int DK, int R, int JS, int IS, int TEAMS>
constexpr int chain_stages() {
    constexpr int left = 226 * 1024 - ChainCfg<DK, R, JS, IS, TEAMS, 0>::total;
    constexpr int n = left / ChainSmem<DK, R, JS>::stage;
    return n < 6 ? n : 6;
}

// What one CTA of the kernel works on.
struct ChainPart {
    int b0, nblk;       // first block of the sequence's, number of blocks
    int j0;             // first of its JS rows j of the state
    int width;          // d_v, or d_k for the response to the segment's start state
    bool response;
    const float* S0;    // start state of this sequence, or null
    float* O;           // rows of O of the first block (response: fp16 rows)
    float* S_end;       // end state [i][j] (response: fp16 [j][i] without its diagonal), or null
    float* D;           // response: the end state's diagonal
};

// Segments (Section 3, "Scan"; Proposition 2.1): the flow of an interval is the pair (P, Xi) with S_end = S_start P + Xi.  A
// sequence is cut into segments that are walked side by side: for each the state from zero (S0 for the first segment), whose
// outputs go to O and whose end is Xi, and, for all but the first, the state from the identity with v = 0, whose "outputs"
// R_t = P_t q_t are what each token makes of its segment's start state and whose end is P.  Then one kernel composes the
// segments' start states and another adds start R_t to O.
// The diagonal of P is kept apart, in fp32, and fp16 is for the rest: where the step sizes are small P is close to the identity, and
// rounding all of it (and the start state before it) would round the whole state once per segment (step sizes of 0.01, 8000
// tokens in 9 segments: relative error of S_final 7.2e-4, this way 6.1e-5, 4.6e-5 in the tcgen05 kernels; at step sizes around 0.5
// 3.49e-4 and 3.44e-4).
struct ChainSeg {
    __half* R;          // [nseq][L][d_k]
    __half* P;          // [nseq][nseg][d_k j][d_k i], zeros on the diagonal
    float* D;           // [nseq][nseg][d_k]: the diagonal
    float* Xi;          // [nseq][nseg][d_k i][d_v j]
    __half* start;      // [nseq][nseg][d_v j][d_k i]
};

// The kernel's arguments, for walk_fp32.
struct ChainArgs {
    ChainGeo g;
    ChainSeg seg;
};

// What this CTA works on; seq: its sequence.
template <int DK, int JS, int C, bool SEG>
__device__ __forceinline__ ChainPart chain_part(const ChainGeo& g, const ChainSeg& sg, const float* S0, float* O, float* S_final, long long& seq) {
    ChainPart part;
    const int slices = g.d_v / JS;
    if constexpr (!SEG) {
        seq = blockIdx.x / slices;
        part = {0, g.nblk, (int)(blockIdx.x % slices) * JS, g.d_v, false, S0 ? S0 + seq * DK * g.d_v : nullptr, O + seq * g.L * g.d_v,
                S_final ? S_final + seq * DK * g.d_v : nullptr, nullptr};
    } else {
        constexpr int rs = DK / JS;
        const int per_seq = g.nseg * slices + (g.nseg - 1) * rs, x = (int)(blockIdx.x % per_seq), y = x - g.nseg * slices;
        seq = blockIdx.x / per_seq;
        part.response = y >= 0;
        const int s = part.response ? 1 + y / rs : x / slices;
        part.b0 = s * g.seg_blk;
        part.nblk = min(g.seg_blk, g.nblk - part.b0);
        part.j0 = (part.response ? y % rs : x % slices) * JS;
        part.width = part.response ? DK : g.d_v;
        const long long row0 = seq * g.L + (long long)part.b0 * C, slot = seq * g.nseg + s;
        part.S0 = s == 0 && S0 ? S0 + seq * DK * g.d_v : nullptr;
        part.O = part.response ? (float*)(sg.R + row0 * DK) : O + row0 * g.d_v;
        part.S_end = part.response ? (float*)(sg.P + slot * DK * DK) : sg.Xi + slot * DK * g.d_v;
        part.D = sg.D + slot * DK;
    }
    return part;
}

// How they reach it.  The call is never made in ordinary use, but how it is written decides which registers the chain has.  us by value, from
// shared memory, and without the call: 250 sequences of 1000, d = 128, r = 2 (128 columns per CTA): 243, 227, 226; 64 x 128, r = 4: 235, 246,
// 236; 19 of 6950 in segments, 64 x 128: r = 1 139, 144, 130, r = 2 193, 183, 181, r = 3 278, 263, 269; 64 x 64, r = 2 108, 103, 102; at d_k = 128
// in segments both alike.
template <int DK, int R, int JS, bool SEG>
constexpr bool WALK_BY_REF = SEG ? !(DK == 64 && R == 1) : DK == 128 && JS == 128;

// 16 rows of S from row `row0` of the CTA's on, once more: the recurrence token by token in fp32, by one warp, two lanes to a row.  Not
// a fast path (1.3 us a token at d_k = 128, r = 1, 3.0 at 64, r = 4): it is there so that every state that fp16 can hold gives a finite
// result, whatever the products with it reach.
template <int DK, int R, int JS, bool SEG, class Args>
__device__ __noinline__ void walk_fp32(Args args, int row0) {
    constexpr int C = NB / R, NI = DK / 2;                        // columns i per lane
    const ChainGeo g = args.g;
    const ChainSeg sg = args.seg;
    long long seq;
    const ChainPart part = chain_part<DK, JS, C, SEG>(g, sg, g.S0, g.O, g.S_final, seq);
    const int lane = threadIdx.x & 31, i0 = (lane & 1) * NI, j = part.j0 + row0 + (lane >> 1);
    const long long tok0 = seq * g.L + (long long)part.b0 * C;
    const int tokens = min(part.nblk * C, g.L - part.b0 * C), group = g.rm == 1 ? 1 : R;      // (group: factors that read the same state)
    auto dot = [&](const float (&S)[NI], const __nv_bfloat16* x, bool self) {
        float d = 0.f;
#pragma unroll
        for (int n = 0; n < NI; n += 8) {
            const uint4 y = *(const uint4*)(x + i0 + n);
            const uint32_t* w = (const uint32_t*)&y;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float z = __uint_as_float(e & 1 ? w[e / 2] & 0xFFFF0000u : w[e / 2] << 16);
                d = fmaf(self ? z : S[n + e], z, d);
            }
        }
        return d + __shfl_xor_sync(0xffffffffu, d, 1);
    };
    float S[NI];
#pragma unroll
    for (int n = 0; n < NI; ++n) S[n] = part.S0 ? part.S0[(long long)(i0 + n) * g.d_v + j] : 0.f;
#pragma unroll 1
    for (int t = 0; t < tokens; ++t) {
#pragma unroll 1
        for (int f = 0; f < R; f += group) {
            const long long m0 = (tok0 + t) * R + f;
            float u[R];
#pragma unroll
            for (int x = 0; x < R; ++x) {
                if (x >= group) break;
                const __nv_bfloat16* kr = g.k + (m0 + x) * DK;
                float b = __bfloat162float(g.beta[m0 + x]);
                if (g.exact) {
                    const float n2 = dot(S, kr, true);
                    if (n2 > 0.f) b = -expm1f(-b * n2) / n2;
                }
                u[x] = b * (__bfloat162float(g.v[(m0 + x) * g.d_v + j]) - dot(S, kr, false));
            }
#pragma unroll
            for (int x = 0; x < R; ++x) {
                if (x >= group) break;
                const __nv_bfloat16* kr = g.k + (m0 + x) * DK + i0;
#pragma unroll
                for (int n = 0; n < NI; n += 8) {
                    const uint4 y = *(const uint4*)(kr + n);
                    const uint32_t* w = (const uint32_t*)&y;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        S[n + e] = fmaf(u[x], __uint_as_float(e & 1 ? w[e / 2] & 0xFFFF0000u : w[e / 2] << 16), S[n + e]);
                }
            }
        }
        const float o = dot(S, g.q + (tok0 + t) * DK, false);
        if ((lane & 1) == 0) part.O[(long long)t * g.d_v + j] = o;
    }
    if (part.S_end)
#pragma unroll
        for (int n = 0; n < NI; ++n) part.S_end[(long long)(i0 + n) * g.d_v + j] = S[n];
}

// K, Q and V of block b (of this part) into stage b mod NS (one thread); rows past the sequence arrive as zeros
template <int DK, int R, int JS, int NS>
__device__ __forceinline__ void load_block(const ChainMaps& maps, uint8_t* smem, uint64_t* land, int b, int seq, const ChainPart& part) {
    using SM = ChainSmem<DK, R, JS>;
    const int st = b % NS;
    uint8_t* sg = smem + st * SM::stage;
    const int bb = part.b0 + b;
    mbar_expect_tx(&land[st], SM::tx_bytes - (part.response ? SM::v_bytes : 0));
    tma_load_4d(sg + SM::k_off, &maps.k, 0, bb * SM::C * R, 0, seq, &land[st]);
    // (r = 3: a block's 21 tokens sit in slabs of 32 rows, one copy each)
    constexpr int QS = SM::CP == SM::C ? 1 : DK / 64;
#pragma unroll
    for (int h = 0; h < QS; ++h) tma_load_4d(sg + SM::q_off + h * (SM::CP * 128), &maps.q, 0, bb * SM::C, h, seq, &land[st]);
    if (!part.response) tma_load_4d(sg + SM::v_off, &maps.v, 0, bb * SM::C * R, part.j0 / (JS < 64 ? JS : 64), seq, &land[st]);
}
// offset of the 16-byte piece c8 (= column / 8) of row `row` of the V tile: 128-byte rows (JS >= 64) or 64-byte rows
template <int JS>
__device__ __forceinline__ uint32_t v_piece(int row, int c8) {
    if (JS >= 64) return (uint32_t)((c8 >> 3) * (NB * 128) + row * 128 + (((c8 & 7) ^ (row & 7)) << 4));
    return (uint32_t)(row * 64 + ((c8 ^ ((row >> 1) & 3)) << 4));
}

// byte offsets of a lane's row address for ldmatrix.x4 within a slab of 128-byte swizzled rows; the K-step kk of 16 columns
// is at off ^ (kk << 5), everything else is added
__device__ __forceinline__ uint32_t lane_off(int row, int half) { return (uint32_t)row * 128u + (uint32_t)((half ^ (row & 7)) << 4); }

// Which warp of a team forms block (16 tokens tt, 16 rows nb) of P: warp w has w + 1 blocks of G, so that all have about as
// many.  Blocks whose rows are all later than the tile's tokens are nobody's.
template <int R>
__host__ __device__ constexpr int p_owner(int tt, int nb) {
    if (nb >= (tt + 1) * R) return -1;
    if (R == 1) return 3 - tt;
    if (R == 2) return tt == 0 ? nb + 1 : nb < 3 ? 0 : 1;
    if (R == 3) return tt == 0 ? (nb < 2 ? 1 : 2) : nb < 3 ? 0 : 3;
    return nb < 2 ? 0 : nb - 1;
}
// G[rows of block W][row blocks 0 .. W] into ga, and warp W's blocks of -P = (-Q K^T) (.) Mincl, negated back, into shared
// memory.  All blocks advance together along the contraction, so that eight to ten accumulators are independent and a key
// fragment serves both.
template <int DK, int R, int CP, int W>
__device__ __forceinline__ void gram_blocks(uint32_t k_b, uint32_t q_b, uint8_t* sp, uint32_t offA, uint32_t offN, int gq, int t4,
                                            float (&ga)[4][2][4]) {
    constexpr int KT = DK / 16, TT = CP / 16;
    float pc[TT][4][2][4];
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
        uint32_t ka[4], qa[TT][4];
        ldmatrix_x4(ka, k_b + (offA ^ ((kk & 3) << 5)) + W * 2048 + (kk >> 2) * (NB * 128));
#pragma unroll
        for (int tt = 0; tt < TT; ++tt)
            if (p_owner<R>(tt, 0) == W || p_owner<R>(tt, 1) == W || p_owner<R>(tt, 2) == W || p_owner<R>(tt, 3) == W)
                ldmatrix_x4(qa[tt], q_b + (offA ^ ((kk & 3) << 5)) + tt * 2048 + (kk >> 2) * (CP * 128));
#pragma unroll
        for (int nb = 0; nb < 4; ++nb) {
            bool used = nb <= W;
#pragma unroll
            for (int tt = 0; tt < TT; ++tt) used = used || p_owner<R>(tt, nb) == W;
            if (!used) continue;
            // (the warp's own rows as columns: the fragment it has, its two middle pieces exchanged, where holding it that long costs
            //  no other register.  us with it and with a second load, 250 sequences of 1000 and 3 of 8192 tokens: d_k = 64, r = 2: 145
            //  and 147, r = 4: 236 and 238.5; d_k = 128: r = 1 154 and 155, but 128 x 64 119 and 108; r = 2 228 and 227, 128 x 64 157 and
            //  160; r = 3 348 and 339, 136 and 114; r = 4 410 and 388, 121 and 123)
            uint32_t x[4] = {ka[0], ka[2], ka[1], ka[3]};
            if (nb != W || (DK == 128 && R != 2)) ldmatrix_x4(x, k_b + (offN ^ ((kk & 3) << 5)) + nb * 2048 + (kk >> 2) * (NB * 128));
            if (nb <= W) {
                mma_acc(ga[nb][0], ka, x[0], x[1], kk > 0);
                mma_acc(ga[nb][1], ka, x[2], x[3], kk > 0);
            }
#pragma unroll
            for (int tt = 0; tt < TT; ++tt)
                if (p_owner<R>(tt, nb) == W) {
                    mma_acc(pc[tt][nb][0], qa[tt], x[0], x[1], kk > 0);
                    mma_acc(pc[tt][nb][1], qa[tt], x[2], x[3], kk > 0);
                }
        }
    }
#pragma unroll
    for (int tt = 0; tt < TT; ++tt)
#pragma unroll
        for (int nb = 0; nb < 4; ++nb) {
            if (p_owner<R>(tt, nb) != W) continue;
            const int ta = 16 * tt + gq, la = (ta + 1) * R, lb = (ta + 9) * R;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = 16 * nb + 8 * h + 2 * t4;
                const bool all = 16 * nb + 15 < (16 * tt + 1) * R;        // (every row is visible to every token of the block)
                *(uint32_t*)(sp + chunk_off(ta, 2 * nb + h, CP) + 4 * t4) =
                    pack_h2(all || m < la ? -pc[tt][nb][h][0] : 0.f, all || m + 1 < la ? -pc[tt][nb][h][1] : 0.f);
                *(uint32_t*)(sp + chunk_off(ta + 8, 2 * nb + h, CP) + 4 * t4) =
                    pack_h2(all || m < lb ? -pc[tt][nb][h][2] : 0.f, all || m + 1 < lb ? -pc[tt][nb][h][3] : 0.f);
            }
        }
}

// ---------------------------------------------------------------------------------------------------------------------
// prep team: blocks b = team, team + TEAMS, ...
// ---------------------------------------------------------------------------------------------------------------------
template <int DK, int R, int JS, int IS, int TEAMS, int NS>
__device__ __forceinline__ void prep_role(const ChainGeo& g, const ChainPart& part, const __nv_bfloat16* __restrict__ beta, int* err, uint8_t* smem,
                                          uint64_t* land, uint64_t* full, long long seq, int team, int tid) {
    using CFG = ChainCfg<DK, R, JS, IS, TEAMS, NS>;
    using SM = ChainSmem<DK, R, JS>;
    constexpr int C = SM::C, CP = SM::CP;
    const int w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const int L = g.L;
    const int bar_id = 1 + team;
    uint8_t* xs = smem + CFG::xs_off + team * NB * 128;
    const uint32_t xs_b = smem_u32(xs);
    const uint32_t offA = lane_off(lane & 15, lane >> 4);
    const uint32_t offN = lane_off((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
    const uint32_t offT = lane_off((lane & 7) + (((lane >> 3) & 1) << 3), lane >> 4);
    const __nv_bfloat16* bs = beta + seq * L * R;
    // (the bits as loaded: a conversion next to the load would make every thread wait for it there, a block ahead of its use)
    auto read_beta = [&](int b) {                                 // rows past the block or the sequence have step size zero
        uint16_t x = 0;
        if (tid < min(C, L - (part.b0 + b) * C) * R)
            asm volatile("ld.global.nc.b16 %0, [%1];" : "=h"(x) : "l"(bs + (long long)(part.b0 + b) * C * R + tid));
        return x;
    };
    uint16_t breg = team < part.nblk ? read_beta(team) : 0;
    const int lim0 = (16 * w + gq) / g.rm * g.rm, lim1 = (16 * w + gq + 8) / g.rm * g.rm;      // (edges of the strict mask)
#pragma unroll 1
    for (int b = team; b < part.nblk; b += TEAMS) {
        const int st = b % NS;
        uint8_t* sg = smem + st * SM::stage;
        const uint32_t k_b = smem_u32(sg + SM::k_off), q_b = smem_u32(sg + SM::q_off);
        // (two in turn: another warp may still be scaling T of the block before)
        float* sBeta = (float*)(smem + CFG::beta_off + team * 512 + (b / TEAMS & 1) * 256);
        // (a failed wait must not strand the others at a barrier: the next one carries the outcome)
        const bool ok = mbar_wait_clk(&land[st], (uint32_t)(b / NS) & 1, err, 311);
        // ---- K, Q: bf16 -> fp16 in place (elementwise, so the swizzled layout is untouched), several pieces per round, so that
        //      their loads are in flight together; Q as -Q: the chain multiplies it with -S
        {
            uint4* p = (uint4*)(sg + SM::k_off) + tid;
            constexpr int PIECES = (SM::k_bytes + SM::q_bytes) / 2048, ROUND = 8;
#pragma unroll
            for (int e0 = 0; e0 < PIECES; e0 += ROUND) {
                uint4 x[ROUND];
#pragma unroll
                for (int e = 0; e < ROUND; ++e)
                    if (e0 + e < PIECES) x[e] = p[(e0 + e) * 128];
#pragma unroll
                for (int e = 0; e < ROUND; ++e)
                    if (e0 + e < PIECES) p[(e0 + e) * 128] = bf16_to_half8(x[e], (e0 + e) * 2048 < SM::k_bytes ? 0u : 0x80008000u);
            }
        }
        fence_async_smem();                                       // (the stage's next copy is ordered after these writes)
        if (tid < NB) sBeta[tid] = __uint_as_float((uint32_t)breg << 16);
        if (b + TEAMS < part.nblk) breg = read_beta(b + TEAMS);
        if (!named_bar_and(bar_id, 128, ok)) return;

        // ---- G (row block w) and this warp's blocks of P
        float ga[4][2][4];
        {
            uint8_t* sp = sg + SM::p_off;
            if (w == 0) gram_blocks<DK, R, CP, 0>(k_b, q_b, sp, offA, offN, gq, t4, ga);
            else if (w == 1) gram_blocks<DK, R, CP, 1>(k_b, q_b, sp, offA, offN, gq, t4, ga);
            else if (w == 2) gram_blocks<DK, R, CP, 2>(k_b, q_b, sp, offA, offN, gq, t4, ga);
            else gram_blocks<DK, R, CP, 3>(k_b, q_b, sp, offA, offN, gq, t4, ga);
        }
        if (g.exact) {
            // |k|^2 is the diagonal of G; beta' = (1 - e^{-beta |k|^2}) / |k|^2
#pragma unroll
            for (int nb = 0; nb < 4; ++nb)
                if (nb == w && (gq >> 1) == t4) {
                    const float n0 = (gq & 1) ? ga[nb][0][1] : ga[nb][0][0], n1 = (gq & 1) ? ga[nb][1][3] : ga[nb][1][2];
                    const int m = 16 * w + gq;
                    if (n0 > 0.f) sBeta[m] = -expm1f(-sBeta[m] * n0) / n0;
                    if (n1 > 0.f) sBeta[m + 8] = -expm1f(-sBeta[m + 8] * n1) / n1;
                }
            __syncwarp();
        }
        // ---- A = Mstrict (.) (diag(beta) G) as A-operand fragments
        uint32_t af[4][4];
        {
            const int m0 = 16 * w + gq, m1 = m0 + 8;
            const float b0 = sBeta[m0], b1 = sBeta[m1];
#pragma unroll
            for (int nb = 0; nb < 4; ++nb)
                if (nb <= w) {
                    // (with groups of three rows the edge also cuts into the block to the left of the diagonal one)
                    const bool edge = nb == w || (R == 3 && nb + 1 == w);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int c = 16 * nb + 8 * h + 2 * t4 + e;
                            ga[nb][h][e] = !edge || c < lim0 ? b0 * ga[nb][h][e] : 0.f;
                            ga[nb][h][2 + e] = !edge || c < lim1 ? b1 * ga[nb][h][2 + e] : 0.f;
                        }
                    frag_pack(af[nb], ga[nb]);
                }
        }
        // ---- D = (I + A_ww)^{-1} (Neumann product, A nilpotent), E_j = D A_wj
        uint32_t df[4], ef[3][4];
        float dd[2][4];
        {
            uint32_t a[4], at[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e] = w == 0 ? af[0][e] : w == 1 ? af[1][e] : w == 2 ? af[2][e] : af[3][e];
            at[0] = movmatrix(a[0]); at[1] = movmatrix(a[2]); at[2] = movmatrix(a[1]); at[3] = movmatrix(a[3]);
            neumann16(dd, a, at, lane, g.rm == 1);
            frag_pack(df, dd);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (j < w) {
                float c[2][4];
                frag_zero(c);
                mma_16816(c[0], df, movmatrix(af[j][0]), movmatrix(af[j][1]));
                mma_16816(c[1], df, movmatrix(af[j][2]), movmatrix(af[j][3]));
                frag_pack(ef[j], c);
            }
        // ---- X_w,j row block by row block; X is left unscaled in the scratch for the row blocks below, T = X diag(beta) in the stage
        auto put_x = [&](int j, const uint32_t (&f)[4]) {         // (f: packed accumulator fragment)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                *(uint32_t*)(xs + chunk_off(16 * w + gq, 2 * j + h, NB) + 4 * t4) = f[2 * h];
                *(uint32_t*)(xs + chunk_off(16 * w + gq + 8, 2 * j + h, NB) + 4 * t4) = f[2 * h + 1];
            }
        };
        auto put_t = [&](int j, const float (&x)[2][4]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 bb = *(const float2*)(sBeta + 16 * j + 8 * h + 2 * t4);
                *(uint32_t*)(sg + SM::t_off + chunk_off(16 * w + gq, 2 * j + h, NB) + 4 * t4) = pack_h2(x[h][0] * bb.x, x[h][1] * bb.y);
                *(uint32_t*)(sg + SM::t_off + chunk_off(16 * w + gq + 8, 2 * j + h, NB) + 4 * t4) = pack_h2(x[h][2] * bb.x, x[h][3] * bb.y);
            }
        };
        float xa[3][2][4];
        auto add_ex = [&](int k2, int j) {                        // xa[j] += E_k2 X_k2,j
            uint32_t x[4];
            ldmatrix_x4_trans(x, xs_b + (offT ^ (j << 5)) + k2 * 2048);
            mma_16816(xa[j][0], ef[k2], x[0], x[1]);
            mma_16816(xa[j][1], ef[k2], x[2], x[3]);
        };
        auto finish = [&](int j, bool later) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) xa[j][h][e] = -xa[j][h][e];
            if (later) {
                uint32_t f[4];
                frag_pack(f, xa[j]);
                put_x(j, f);
            }
            put_t(j, xa[j]);
        };
#pragma unroll
        for (int j = 0; j < 3; ++j) frag_zero(xa[j]);
        put_x(w, df);
        named_bar(bar_id, 128);
        put_t(w, dd);                                             // (after the barrier: beta' of the exact step is complete)
        if (w == 1) {
            add_ex(0, 0);
            finish(0, true);
        } else if (w == 2) {
            add_ex(1, 1);
            finish(1, true);
            add_ex(0, 0);
        } else if (w == 3) {
            add_ex(2, 2);
            finish(2, false);
            add_ex(1, 1);
            add_ex(0, 0);
        }
        named_bar(bar_id, 128);
        if (w == 2) {
            add_ex(1, 0);
            finish(0, true);
        } else if (w == 3) {
            add_ex(1, 0);
            add_ex(2, 1);
            finish(1, false);
        }
        named_bar(bar_id, 128);
        if (w == 3) {
            add_ex(2, 0);
            finish(0, false);
        }
        mbar_arrive(&full[st]);
    }
}

// ---------------------------------------------------------------------------------------------------------------------
// chain warp: rows j of the 16-column group `grp` of the CTA's JS columns, columns i of half `hi` (IS = 2)
// ---------------------------------------------------------------------------------------------------------------------
template <int DK, int R, int JS, int IS, int TEAMS, int NS, bool SEG>
__device__ __forceinline__ void chain_role(const ChainMaps& maps, const ChainGeo& g, const ChainPart& part, int* err, uint8_t* smem,
                                           uint64_t* land, uint64_t* full, uint64_t* empty, const ChainSeg& seg, ChainArgs& args, int seq, int warp,
                                           int lane) {
    using CFG = ChainCfg<DK, R, JS, IS, TEAMS, NS>;
    using SM = ChainSmem<DK, R, JS>;
    constexpr int C = SM::C, CP = SM::CP, TT = CP / 16;
    constexpr int DI = DK / IS, KT = DI / 16;                     // columns i of this warp, in K-steps of 16
    const int grp = warp / IS, hi = warp % IS;
    const int gq = lane >> 2, t4 = lane & 3;
    const uint32_t offA = lane_off(lane & 15, lane >> 4);
    const uint32_t offN = lane_off((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
    const uint32_t offT = lane_off((lane & 7) + (((lane >> 3) & 1) << 3), lane >> 4);
    // V, read transposed: matrix id = lane >> 3: rows + 8 (id >> 1), columns 8 (id & 1)
    const uint32_t offV = v_piece<JS>((lane & 7) + ((lane >> 4) << 3), 2 * grp + ((lane >> 3) & 1));
    constexpr uint32_t V_STEP = 16 * (JS >= 64 ? 128 : 64);
    const uint32_t smem_b = smem_u32(smem);
    // K-step kk of this warp = step hi KT + kk of the row: slab and 32-byte position within it
    auto kpos = [&](int kk, int slab_bytes) { return (uint32_t)((hi * KT + kk) >> 2) * (uint32_t)slab_bytes; };
    auto kxor = [&](int kk) { return (uint32_t)(((hi * KT + kk) & 3) << 5); };

    float S[2 * KT][4];                                           // [8 columns i][c]: rows j = gq, gq + 8, columns 2 t4, 2 t4 + 1
    const int jr = part.j0 + 16 * grp + gq, i0 = hi * DI + 2 * t4, width = part.width;
#pragma unroll
    for (int n = 0; n < 2 * KT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = i0 + 8 * n + (e & 1), j = jr + 8 * (e >> 1);
            if (SEG && part.response) S[n][e] = i == j ? 1.f : 0.f;
            else S[n][e] = part.S0 ? part.S0[(long long)i * width + j] : 0.f;
        }
    float* ob = part.O + part.j0 + 16 * grp + 2 * t4 + (IS == 2 ? 8 * hi : 0);     // O of the current block (response: in halves)
    __half* rb = (__half*)part.O + part.j0 + 16 * grp + 2 * t4 + (IS == 2 ? 8 * hi : 0);
    auto put_o = [&](int t, int dj, float x, float y, bool pred) {     // token t of the current block
        // (both forms, predicated: a branch at every store would keep the products on either side of it apart)
        if (SEG) store_h2_if(rb + (long long)t * width + dj, pack_h2(x, y), pred && part.response);
        store2_if(ob + (long long)t * width + dj, x, y, pred && !(SEG && part.response));
    };

    // IS = 2: what this warp keeps of O of the block before (8 of the 16 columns j), without the other warp's part of Q S^T
    float ok8[TT][4];
    int Cv_prev = 0;
    uint8_t* exw = smem + CFG::ex_off + grp * (4 * CFG::x_piece * 512) + lane * 16;
    auto store8 = [&](const float4* other) {                      // ob points one block further than what is stored
#pragma unroll
        for (int tt = 0; tt < TT; ++tt) {
            const float4 x = other[(8 + tt) * 32];
            const int t = 16 * tt + gq;
            put_o(t - C, 0, ok8[tt][0] + x.x, ok8[tt][1] + x.y, t < Cv_prev);
            put_o(t - C + 8, 0, ok8[tt][2] + x.z, ok8[tt][3] + x.w, t + 8 < Cv_prev);
        }
    };
    if (IS == 2)
#pragma unroll
        for (int tt = 0; tt < TT; ++tt) {
            ((float4*)(exw + (2 + hi) * (CFG::x_piece * 512)))[(8 + tt) * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 4; ++e) ok8[tt][e] = 0.f;
        }

    int st = 0, phase = 0, st_prev = 0, ph_prev = 0;
#pragma unroll 1
    for (int b = 0; b < part.nblk; ++b) {
        const uint32_t sg = smem_b + st * SM::stage;
        const uint32_t k_b = sg + SM::k_off, q_b = sg + SM::q_off, t_b = sg + SM::t_off, p_b = sg + SM::p_off, v_b = sg + SM::v_off;
        uint32_t s16[KT][4];                                      // fp16 copy of -S: A operand of -S K^T, B operand of (-Q)(-S)^T
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
            s16[kk][0] = pack_h2(-S[2 * kk][0], -S[2 * kk][1]);
            s16[kk][1] = pack_h2(-S[2 * kk][2], -S[2 * kk][3]);
            s16[kk][2] = pack_h2(-S[2 * kk + 1][0], -S[2 * kk + 1][1]);
            s16[kk][3] = pack_h2(-S[2 * kk + 1][2], -S[2 * kk + 1][3]);
        }
        // (IS = 2: the pair's barrier below carries the outcome, so that a failed wait never strands the other warp there; V, which
        //  the team does not touch, had landed before the team arrived: the second wait makes it visible here)
        const bool ok = mbar_wait_clk(&full[st], (uint32_t)phase, err, 312) && mbar_wait_clk(&land[st], (uint32_t)phase, err, 313);
        if (IS == 1 && !ok) return;
        // ---- R = V^T - S K^T: the accumulators start from V (in one warp of a pair)
        float r[8][4];
        if (IS == 1 || hi == 0) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                uint32_t x[4];
                ldmatrix_x4_trans(x, v_b + offV + kk * V_STEP);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    r[2 * kk + (e >> 1)][2 * (e & 1)] = __uint_as_float(x[e] << 16);
                    r[2 * kk + (e >> 1)][2 * (e & 1) + 1] = __uint_as_float(x[e] & 0xFFFF0000u);
                }
            }
        } else {
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) r[n][e] = 0.f;
        }
#pragma unroll
        for (int kk = 0; kk < KT; ++kk)
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                uint32_t x[4];
                ldmatrix_x4(x, k_b + (offN ^ kxor(kk)) + np * 2048 + kpos(kk, NB * 128));
                mma_16816(r[2 * np], s16[kk], x[0], x[1]);
                mma_16816(r[2 * np + 1], s16[kk], x[2], x[3]);
            }
        if (IS == 2) {
            // the other warp of the pair has the other half of the sum; with it goes the half of Q S^T of the block before that
            // the other warp stores
            float4* mine = (float4*)(exw + ((b & 1) * 2 + hi) * (CFG::x_piece * 512));
            const float4* other = (const float4*)(exw + ((b & 1) * 2 + (hi ^ 1)) * (CFG::x_piece * 512));
            const float4* other_o = (const float4*)(exw + (((b & 1) ^ 1) * 2 + (hi ^ 1)) * (CFG::x_piece * 512));
#pragma unroll
            for (int n = 0; n < 8; ++n) mine[n * 32] = make_float4(r[n][0], r[n][1], r[n][2], r[n][3]);
            if (!named_bar_and(1 + TEAMS + grp, 64, ok)) return;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                const float4 x = other[n * 32];
                r[n][0] += x.x; r[n][1] += x.y; r[n][2] += x.z; r[n][3] += x.w;
            }
            store8(other_o);
        }
        // ---- the block NS - 1 further on into the stage that every chain warp has left (a block ago)
        if (warp == 0 && lane == 0 && b > 0 && b - 1 + NS < part.nblk && mbar_wait_clk(&empty[st_prev], (uint32_t)ph_prev, err, 314))
            load_block<DK, R, JS, NS>(maps, smem, land, b - 1 + NS, seq, part);
        __syncwarp();
        // ---- U'^T = R T^T (T lower triangular)
        uint32_t r16[4][4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            r16[kk][0] = pack_h2(r[2 * kk][0], r[2 * kk][1]);
            r16[kk][1] = pack_h2(r[2 * kk][2], r[2 * kk][3]);
            r16[kk][2] = pack_h2(r[2 * kk + 1][0], r[2 * kk + 1][1]);
            r16[kk][3] = pack_h2(r[2 * kk + 1][2], r[2 * kk + 1][3]);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int nb = kk; nb < 4; ++nb) {
                uint32_t x[4];
                ldmatrix_x4(x, t_b + (offN ^ (kk << 5)) + nb * 2048);
                mma_acc(r[2 * nb], r16[kk], x[0], x[1], kk > 0);
                mma_acc(r[2 * nb + 1], r16[kk], x[2], x[3], kk > 0);
            }
        uint32_t u16[4][4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            u16[kk][0] = pack_h2(r[2 * kk][0], r[2 * kk][1]);
            u16[kk][1] = pack_h2(r[2 * kk][2], r[2 * kk][3]);
            u16[kk][2] = pack_h2(r[2 * kk + 1][0], r[2 * kk + 1][1]);
            u16[kk][3] = pack_h2(r[2 * kk + 1][2], r[2 * kk + 1][3]);
        }
        // ---- S += U'^T K
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int ip = 0; ip < KT; ++ip) {
                uint32_t x[4];
                ldmatrix_x4_trans(x, k_b + (offT ^ kxor(ip)) + kk * 2048 + kpos(ip, NB * 128));
                mma_16816(S[2 * ip], u16[kk], x[0], x[1]);
                mma_16816(S[2 * ip + 1], u16[kk], x[2], x[3]);
            }
        // ---- O = Q S^T + P U' with the state before the update (these products fill the latency of the update).  Two tiles of 16
        //      tokens at a time, or one with its sums in two halves: at least four independent accumulators, the depth of the
        //      product's pipeline (one tile at a time took 2.8 k cycles of a step of 6.5 k at d_k = 128, r = 1)
        const int Cv = min(C, g.L - (part.b0 + b) * C);
        constexpr int TG = TT >= 2 ? 2 : 1, SP = 3 - TG;
#pragma unroll
        for (int tg = 0; tg < TT; tg += TG) {
            float o[TG][SP][2][4];
#pragma unroll
            for (int kk = 0; kk < KT; ++kk)
#pragma unroll
                for (int u = 0; u < TG; ++u) {
                    uint32_t a[4];
                    ldmatrix_x4(a, q_b + (offA ^ kxor(kk)) + (tg + u) * 2048 + kpos(kk, CP * 128));
                    mma_acc(o[u][kk % SP][0], a, s16[kk][0], s16[kk][2], kk >= SP);
                    mma_acc(o[u][kk % SP][1], a, s16[kk][1], s16[kk][3], kk >= SP);
                }
            if (IS == 2) {
                // (the warp keeps 8 of the 16 columns j and hands its half of the sum for the others over)
#pragma unroll
                for (int u = 0; u < TG; ++u) {
                    if (SP == 2)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o[u][0][0][e] += o[u][SP - 1][0][e];
                            o[u][0][1][e] += o[u][SP - 1][1][e];
                        }
                    float4* mine = (float4*)(exw + ((b & 1) * 2 + hi) * (CFG::x_piece * 512));
                    mine[(8 + tg + u) * 32] = hi ? make_float4(o[u][0][0][0], o[u][0][0][1], o[u][0][0][2], o[u][0][0][3])
                                                 : make_float4(o[u][0][1][0], o[u][0][1][1], o[u][0][1][2], o[u][0][1][3]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) ok8[tg + u][e] = hi ? o[u][0][1][e] : o[u][0][0][e];
                }
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int u = 0; u < TG; ++u) {
                    if (kk >= (tg + u + 1) * R) continue;
                    uint32_t a[4];
                    ldmatrix_x4(a, p_b + (offA ^ (kk << 5)) + (tg + u) * 2048);
                    if (IS == 2) {
                        mma_16816(ok8[tg + u], a, hi ? u16[kk][1] : u16[kk][0], hi ? u16[kk][3] : u16[kk][2]);
                    } else {
                        mma_16816(o[u][kk % SP][0], a, u16[kk][0], u16[kk][2]);
                        mma_16816(o[u][kk % SP][1], a, u16[kk][1], u16[kk][3]);
                    }
                }
            if (IS == 1)
#pragma unroll
                for (int u = 0; u < TG; ++u) {
                    if (SP == 2)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o[u][0][0][e] += o[u][SP - 1][0][e];
                            o[u][0][1][e] += o[u][SP - 1][1][e];
                        }
                    const int t = 16 * (tg + u) + gq;
                    put_o(t, 0, o[u][0][0][0], o[u][0][0][1], t < Cv);
                    put_o(t, 8, o[u][0][1][0], o[u][0][1][1], t < Cv);
                    put_o(t + 8, 0, o[u][0][0][2], o[u][0][0][3], t + 8 < Cv);
                    put_o(t + 8, 8, o[u][0][1][2], o[u][0][1][3], t + 8 < Cv);
                }
        }
        Cv_prev = Cv;
        ob += (long long)C * width;
        rb += (long long)C * width;
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
        st_prev = st;
        ph_prev = phase;
        if (++st == NS) {
            st = 0;
            phase ^= 1;
        }
    }
    if (IS == 2) {
        named_bar(1 + TEAMS + grp, 64);                           // (both warps are here: a failed wait left through the barrier above)
        store8((const float4*)(exw + (((part.nblk & 1) ^ 1) * 2 + (hi ^ 1)) * (CFG::x_piece * 512)));
    }
    if (SEG && part.response) {
        __half* P = (__half*)part.S_end;
#pragma unroll
        for (int n = 0; n < 2 * KT; ++n)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const int j = jr + 4 * e, i = i0 + 8 * n;
                *(uint32_t*)(P + (long long)j * DK + i) = pack_h2(i == j ? 0.f : S[n][e], i + 1 == j ? 0.f : S[n][e + 1]);
                if (i == j) part.D[j] = S[n][e];
                if (i + 1 == j) part.D[j] = S[n][e + 1];
            }
        return;
    }
    // (one entry tells for its row.  The end state may replace the start state, which is still needed where rows are lost)
    bool lost = __any_sync(0xffffffffu, !(fabsf(S[0][0]) <= FLT_MAX) || !(fabsf(S[0][2]) <= FLT_MAX));
    if (IS == 2) lost = !named_bar_and(1 + TEAMS + grp, 64, !lost);   // (both warps of a pair have written their last O)
    if (lost) {
        if (hi == 0) {
            if constexpr (WALK_BY_REF<DK, R, JS, SEG>) walk_fp32<DK, R, JS, SEG, const ChainArgs&>(args, 16 * grp);
            else walk_fp32<DK, R, JS, SEG, ChainArgs>(ChainArgs{g, seg}, 16 * grp);
        }
    } else if (part.S_end) {
#pragma unroll
        for (int n = 0; n < 2 * KT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) part.S_end[(long long)(i0 + 8 * n + (e & 1)) * width + jr + 8 * (e >> 1)] = S[n][e];
    }
}

template <int DK, int R, int JS, int IS, int TEAMS, int NS, bool SEG>
__global__ void __launch_bounds__(ChainCfg<DK, R, JS, IS, TEAMS, NS>::threads, 1)
chain_kernel(const __grid_constant__ ChainMaps maps, const __nv_bfloat16* __restrict__ beta, const float* __restrict__ S0,
             float* __restrict__ O, float* __restrict__ S_final, int* __restrict__ status, ChainGeo g, ChainSeg sg) {
    using CFG = ChainCfg<DK, R, JS, IS, TEAMS, NS>;
    using SM = ChainSmem<DK, R, JS>;
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t land[NS], full[NS], empty[NS];
    __shared__ ChainArgs args;
    const int tid = threadIdx.x, warp = tid >> 5;
    long long seq;
    const ChainPart part = chain_part<DK, JS, SM::C, SEG>(g, sg, S0, O, S_final, seq);
    if ((smem_u32(smem) & 1023u) != 0) {                          // (the swizzled layouts need a 1024-byte aligned base)
        wait_for_previous_kernel();
        if (tid == 0) atomicCAS(status, 0, 99);
        return;
    }
    if (WALK_BY_REF<DK, R, JS, SEG> && tid == 32) args = {g, sg};
    if (tid == 0) {
        for (int x = 0; x < NS; ++x) {
            mbar_init(&land[x], 1);
            mbar_init(&full[x], 128);
            mbar_init(&empty[x], CFG::NCW);
        }
        mbar_fence_init();
        prefetch_tmap(&maps.q);
        prefetch_tmap(&maps.k);
        prefetch_tmap(&maps.v);
    }
    if (SM::CP > SM::C || part.response) {                        // (r = 3: query rows that no copy writes are read; a response: v = 0)
        for (int e = tid; e < NS * SM::stage / 16; e += CFG::threads) ((uint4*)smem)[e] = make_uint4(0, 0, 0, 0);
        fence_async_smem();
    }
    wait_for_previous_kernel();
    if (!SEG) let_next_kernel_start();      // (chain_compose's blocks would crowd on what few multiprocessors have room: 144 us instead of 140)
    if (tid == 0 && blockIdx.x == 0 && g.clear) *status = 0;      // (the call's status word: a wait expires a second from now at the earliest)
    __syncthreads();
    if (tid == 0)
        for (int b = 0; b < NS && b < part.nblk; ++b) load_block<DK, R, JS, NS>(maps, smem, land, b, (int)seq, part);
    __syncwarp();
    if (warp < CFG::NCW)
        chain_role<DK, R, JS, IS, TEAMS, NS, SEG>(maps, g, part, status, smem, land, full, empty, sg, args, (int)seq, warp, tid & 31);
    else
        prep_role<DK, R, JS, IS, TEAMS, NS>(g, part, beta, status, smem, land, full, seq, (warp - CFG::NCW) >> 2, (tid - 32 * CFG::NCW) & 127);
}

// Start states of the segments: one CTA per sequence and 16 rows j, serial over the segments; four warps with a quarter of the
// columns i each.  start(1) = Xi_0, start(s+1) = start(s) P_s + Xi_s; the last one is S_final.  The diagonal's part of the product is
// fp32, the rest has fp16 operands.  The next P and Xi come while the present ones are used.
template <int DK>
__global__ void __launch_bounds__(128) chain_compose(ChainSeg sg, float* __restrict__ S_final, int nseg, int d_v) {
    constexpr int LD = DK + 8, NT = DK / 32, PIECES = DK * DK / 8 / 128;
    extern __shared__ __align__(16) uint8_t smem_tail[];
    __half* sP = (__half*)smem_tail;                                   // [2][DK][LD]
    __half* sA = sP + 2 * DK * LD;                                // [2][16][LD]  fp16 rows of the start state
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const int groups = d_v / 16;
    const long long seq = blockIdx.x / groups;
    const int j = (int)(blockIdx.x % groups) * 16 + gq, i0 = w * (DK / 4) + 2 * t4;
    auto load_p = [&](int s) {
        const __half* src = sg.P + (seq * nseg + s) * DK * DK;
        __half* dst = sP + (s & 1) * DK * LD;
#pragma unroll
        for (int e = 0; e < PIECES; ++e) {
            const int p = e * 128 + tid, row = p / (DK / 8), c = p % (DK / 8);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + row * LD + c * 8)), "l"(src + row * DK + c * 8) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float S[NT][4];
    auto xi = [&](int s, float (&x)[NT][4]) {
        const float* src = sg.Xi + (seq * nseg + s) * DK * d_v;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) x[n][e] = src[(long long)(i0 + 8 * n + (e & 1)) * d_v + j + 8 * (e >> 1)];
    };
    auto diagonal = [&](int s, float2 (&x)[NT]) {
#pragma unroll
        for (int n = 0; n < NT; ++n) x[n] = *(const float2*)(sg.D + (seq * nseg + s) * DK + i0 + 8 * n);
    };
    float X[NT][4], Xn[NT][4];                                    // Xi of this step and of the next
    float2 D[NT], Dn[NT];                                         // the diagonal of P likewise
    wait_for_previous_kernel();
    load_p(1);
    xi(0, S);
    xi(1, X);
    diagonal(1, D);
#pragma unroll 1
    for (int s = 1; s < nseg; ++s) {
        __half* a_s = sA + (s & 1) * 16 * LD;
        __half* out = sg.start + (seq * nseg + s) * d_v * DK;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t x = pack_h2(S[n][2 * h], S[n][2 * h + 1]);
                *(uint32_t*)(a_s + (gq + 8 * h) * LD + i0 + 8 * n) = x;
                *(uint32_t*)(out + (long long)(j + 8 * h) * DK + i0 + 8 * n) = x;
            }
        if (s + 1 < nseg) {
            xi(s + 1, Xn);
            diagonal(s + 1, Dn);
            load_p(s + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const __half* P = sP + (s & 1) * DK * LD;
        float M[NT][4];
#pragma unroll
        for (int kk = 0; kk < DK / 16; ++kk) {
            uint32_t a[4];
            ldmatrix_x4(a, smem_u32(a_s + (lane & 15) * LD + 16 * kk + 8 * (lane >> 4)));
#pragma unroll
            for (int np = 0; np < NT / 2; ++np) {
                uint32_t x[4];
                ldmatrix_x4_trans(x, smem_u32(P + (16 * kk + (lane & 7) + (((lane >> 3) & 1) << 3)) * LD + w * (DK / 4) + 16 * np + 8 * (lane >> 4)));
                mma_acc(M[2 * np], a, x[0], x[1], kk > 0);
                mma_acc(M[2 * np + 1], a, x[2], x[3], kk > 0);
            }
        }
        // (Xi and the diagonal last: their loads have had the whole step)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                S[n][e] = fmaf(S[n][e], e & 1 ? D[n].y : D[n].x, X[n][e]) + M[n][e];
                if (s + 1 < nseg) X[n][e] = Xn[n][e];
            }
            if (s + 1 < nseg) D[n] = Dn[n];
        }
        __syncthreads();                                          // (P of this step is replaced after the next one's first barrier)
    }
    if (S_final) {
        float* out = S_final + seq * DK * d_v;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) out[(long long)(i0 + 8 * n + (e & 1)) * d_v + j + 8 * (e >> 1)] = S[n][e];
    }
}

// O[t][j] += sum_i R[t][i] start[j][i] for the tokens of all segments but the first: grid (128-token tiles, nseq (nseg - 1)), a
// warp per 16 tokens.  Bound by the traffic: per token R once, O read and written.
template <int DK, int DV>
__global__ void __launch_bounds__(256) chain_apply(ChainSeg sg, float* __restrict__ O, int L, int seg_tokens, int nseg) {
    constexpr int LD = DK + 8, KT = DK / 16;
    extern __shared__ __align__(16) uint8_t smem_tail[];
    __half* sS = (__half*)smem_tail;                                   // [DV][LD]
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const long long seq = blockIdx.y / (nseg - 1);
    const int s = 1 + (int)(blockIdx.y % (nseg - 1));
    const int t_end = min(L, (s + 1) * seg_tokens), t0 = s * seg_tokens + blockIdx.x * 128 + w * 16 + gq;
    const __half* src = sg.start + (seq * nseg + s) * DV * DK;
    wait_for_previous_kernel();
#pragma unroll
    for (int e = 0; e < DV * DK / 8 / 256; ++e) {
        const int p = e * 256 + tid, row = p / (DK / 8), c = p % (DK / 8);
        *(uint4*)(sS + row * LD + c * 8) = *(const uint4*)(src + row * DK + c * 8);
    }
    uint32_t a[KT][4];
    const bool in0 = t0 < t_end, in1 = t0 + 8 < t_end;
    const __half* r0 = sg.R + (seq * L + t0) * DK + 2 * t4;
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
        a[kk][0] = in0 ? *(const uint32_t*)(r0 + 16 * kk) : 0u;
        a[kk][1] = in1 ? *(const uint32_t*)(r0 + 8 * DK + 16 * kk) : 0u;
        a[kk][2] = in0 ? *(const uint32_t*)(r0 + 16 * kk + 8) : 0u;
        a[kk][3] = in1 ? *(const uint32_t*)(r0 + 8 * DK + 16 * kk + 8) : 0u;
    }
    // (every load is requested before the first is used: a store to O between them would hold back those behind it)
    float* o0 = O + (seq * L + t0) * DV + 2 * t4;
    float c[DV / 8][4];
#pragma unroll
    for (int n = 0; n < DV / 8; ++n) {
        const float2 x = in0 ? *(const float2*)(o0 + 8 * n) : make_float2(0.f, 0.f);
        const float2 y = in1 ? *(const float2*)(o0 + 8 * DV + 8 * n) : make_float2(0.f, 0.f);
        c[n][0] = x.x; c[n][1] = x.y; c[n][2] = y.x; c[n][3] = y.y;
    }
    __syncthreads();
    // (calls one after another, us with an early start of the next and without: 15 blocks 30.6 and 31.3, 62: 43.2 and 43.7 (d = 128,
    //  r = 1), 26.2 and 27.1 (d = 64).  Where the blocks are many the next kernel's come to multiprocessors in the order in which
    //  these leave, apart from their neighbours with the same inputs: at d = 128 1 - 4 % slower, 256 blocks 101.2 and 99.5, 1024: 350 and
    //  337 (r = 2); at d = 64 1 - 2 % faster, 256 blocks 37.3 and 38.0.  The line is below the first shape that loses)
    if (gridDim.x * gridDim.y <= 128) let_next_kernel_start();
#pragma unroll
    for (int np = 0; np < DV / 16; ++np) {
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
            uint32_t x[4];
            ldmatrix_x4(x, smem_u32(sS + (16 * np + (lane & 7) + ((lane >> 4) << 3)) * LD + 16 * kk + 8 * ((lane >> 3) & 1)));
            mma_16816(c[2 * np], a[kk], x[0], x[1]);
            mma_16816(c[2 * np + 1], a[kk], x[2], x[3]);
        }
#pragma unroll
        for (int n = 2 * np; n < 2 * np + 2; ++n) {
            if (in0) *(float2*)(o0 + 8 * n) = make_float2(c[n][0], c[n][1]);
            if (in1) *(float2*)(o0 + 8 * DV + 8 * n) = make_float2(c[n][2], c[n][3]);
        }
    }
}

// How a sequence is spread over CTAs: columns per CTA, and segments.  The time is (waves of CTAs) x (blocks of a segment) x
// (time of a block), plus what composing segments costs.
// Columns: fewer per CTA make a shorter step but more CTAs.  Measured with one wave, us per block for d_k = d_v = 128, r = 1 .. 4: 32
// columns by pairs of warps 2.35, 1.82, 1.74, 1.70; 64 columns 3.3, 2.5, 2.55, 2.3; 128 columns 4.4, 3.4, 3.4, 3.0.  At d_k = 64 a step
// is short enough that 32 columns gain nothing over 64, and 128 columns cost 1.53 times as much.
// Segments: as many as one wave of CTAs holds pay for the second walk (the responses) and for two more kernels when few
// sequences are long: taken where the estimate falls (d = 64, r = 1, one sequence: 1200 tokens 17 us instead of 38; d = 128: 600 tokens
// 20.5 instead of 26).
enum { COLS_32, COLS_64, COLS_128 };
struct ChainPlan {
    int cols, nseg, seg_blk;
    double us;
    double short_us;          // the kernel alone without segments, the start of each wave counted: what a call of a few blocks takes
};
ChainPlan make_plan(const Problem& p) {
    static const double step[2][4] = {{1.9, 1.45, 1.42, 1.32}, {3.3, 2.5, 2.55, 2.3}};      // us per block, 64 columns, d_k = 64 and 128
    const long long nseq = (long long)p.B * p.H, sms = sm_count();
    const int C = NB / p.r, nblk = (p.L + C - 1) / C;
    const double st = step[p.d_k == 128][p.r - 1];
    auto waves = [&](int js) { return (double)((nseq * (p.d_v / js) + sms - 1) / (sms > 0 ? sms : 1)); };
    double best = waves(64);
    ChainPlan plan{COLS_64, 1, nblk, 0.0, 0.0};
    double turns = best;
    if (p.d_k == 128 && 0.72 * waves(32) < best) {
        turns = waves(32);
        best = 0.72 * turns;
        plan.cols = COLS_32;
    }
    if (p.d_v == 128) {
        const double w = (p.d_k == 128 ? 1.34 : 1.53) * waves(128);
        if (w < best) {
            best = w;
            turns = waves(128);
            plan.cols = COLS_128;
        }
    }
    plan.us = 7.0 + nblk * st * best;
    plan.short_us = 5.0 * turns + nblk * st * best;
    const double limit = 0.92 * plan.us;
    // (kernels and their gaps, then the traffic of the responses and of O at about 4 TB/s)
    const double extra = (p.d_k == 128 ? 14.0 : 9.0) + (double)nseq * p.L * (4.0 * p.d_k + 8.0 * p.d_v) / 4e6;
    // (calls of up to 512 tokens at d_k = 128 are one launch, as they are specified to be: 400 tokens, r = 2 take 27 us instead of 20)
    if (p.d_k == 128 && p.L <= 512) return plan;
    for (int cols = p.d_k == 128 ? COLS_32 : COLS_64; cols <= COLS_64; ++cols) {
        const int js = cols == COLS_32 ? 32 : 64, vs = p.d_v / js, rs = p.d_k / js;
        const long long most = (sms / nseq + rs) / (vs + rs);
        for (int want = 2; want <= most && want <= 64 && want <= nblk; ++want) {
            const int seg_blk = (nblk + want - 1) / want, nseg = (nblk + seg_blk - 1) / seg_blk;
            const double us = extra + 0.8 * nseg + seg_blk * st * (cols == COLS_32 ? 0.72 : 1.0);
            if (us < limit && us < plan.us) plan = {cols, nseg, seg_blk, us, plan.short_us};
        }
    }
    return plan;
}

struct ChainCarve {
    size_t R, P, D, Xi, start, total;
};
ChainCarve carve(const Problem& p, const ChainPlan& plan) {
    ChainCarve c{};
    size_t off = 1024;                                            // (word 0 of a caller's workspace is the status word)
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += align_up(bytes, 256);
        return at;
    };
    if (plan.nseg > 1) {
        const size_t nseq = (size_t)p.B * p.H, slots = nseq * plan.nseg;
        c.R = take(nseq * p.L * p.d_k * 2);
        c.P = take(slots * p.d_k * p.d_k * 2);
        c.D = take(slots * p.d_k * 4);
        c.Xi = take(slots * p.d_k * p.d_v * 4);
        c.start = take(slots * p.d_v * p.d_k * 2);
    }
    c.total = off;
    return c;
}

template <int DK, int R, int JS, int IS, int TEAMS, bool SEG>
int launch(const Problem& p, const ChainPlan& plan, const ChainSeg& sg) {
    constexpr int NS = chain_stages<DK, R, JS, IS, TEAMS>();
    using CFG = ChainCfg<DK, R, JS, IS, TEAMS, NS>;
    static_assert(CFG::total <= 227 * 1024 && NS >= 2, "shared memory budget");
    const void* fn = (const void*)chain_kernel<DK, R, JS, IS, TEAMS, NS, SEG>;
    constexpr int C = NB / R;
    ChainGeo g{p.L, p.d_v, (p.L + C - 1) / C, plan.nseg, plan.seg_blk, p.mask_group(), p.exact ? 1 : 0, p.clear_status ? 1 : 0,
               (const __nv_bfloat16*)p.q, (const __nv_bfloat16*)p.k, (const __nv_bfloat16*)p.v, (const __nv_bfloat16*)p.beta,
               p.S0, p.O, p.S_final};
    const long long nseq = (long long)p.B * p.H, grid = nseq * (plan.nseg * (p.d_v / JS) + (plan.nseg - 1) * (DK / JS));
    ChainMaps maps;
    constexpr int VC = JS < 64 ? JS : 64;
    if (!make_slab_map(&maps.k, p.k, nseq, (uint64_t)p.L * R, DK, 64, NB, DK / 64) ||
        !make_slab_map(&maps.q, p.q, nseq, p.L, DK, 64, C, R == 3 ? 1 : DK / 64) ||
        !make_slab_map(&maps.v, p.v, nseq, (uint64_t)p.L * R, p.d_v, VC, NB, JS / VC))
        return record_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    static std::atomic<uint64_t> opted_in{0};
    const int st = allow_smem(opted_in, fn, CFG::total);
    if (st != PF_OK) return st;
    void* args[] = {(void*)&maps, (void*)&p.beta, (void*)&p.S0, (void*)&p.O, (void*)&p.S_final, (void*)&p.status, (void*)&g, (void*)&sg};
    prof_begin("chain", p.stream);
    PF_CUDA_TRY(launch_early(fn, dim3((unsigned)grid), CFG::threads, args, (size_t)CFG::total, p.stream));
    prof_end(p.stream);
    count_launch(1);
    return PF_OK;
}

template <int DK, int R>
int launch_plan(const Problem& p, const ChainPlan& plan, const ChainSeg& sg) {
    if (plan.nseg > 1) {
        if constexpr (DK == 128)
            if (plan.cols == COLS_32) return launch<DK, R, 32, 2, 2, true>(p, plan, sg);
        return launch<DK, R, 64, 1, 2, true>(p, plan, sg);
    }
    if constexpr (DK == 128)
        if (plan.cols == COLS_32) return launch<DK, R, 32, 2, 2, false>(p, plan, sg);
    if (plan.cols == COLS_64) return launch<DK, R, 64, 1, 2, false>(p, plan, sg);
    return launch<DK, R, 128, 1, DK == 64 ? 2 : 1, false>(p, plan, sg);
}
template <int DK>
int launch_rank(const Problem& p, const ChainPlan& plan, const ChainSeg& sg) {
    switch (p.r) {
        case 1: return launch_plan<DK, 1>(p, plan, sg);
        case 2: return launch_plan<DK, 2>(p, plan, sg);
        case 3: return launch_plan<DK, 3>(p, plan, sg);
        default: return launch_plan<DK, 4>(p, plan, sg);
    }
}

template <int DK, int DV>
int launch_seg_tail(const Problem& p, const ChainPlan& plan, const ChainSeg& sg) {
    const int nseq = p.B * p.H, dv = DV, seg_tokens = plan.seg_blk * (NB / p.r);
    constexpr int LD = DK + 8;
    {
        constexpr int smem = (2 * DK + 2 * 16) * LD * 2;
        static std::atomic<uint64_t> opted_in{0};
        const int st = allow_smem(opted_in, (const void*)chain_compose<DK>, smem);
        if (st != PF_OK) return st;
        prof_begin("chain_compose", p.stream);
        void* args[] = {(void*)&sg, (void*)&p.S_final, (void*)&plan.nseg, (void*)&dv};
        PF_CUDA_TRY(launch_early((const void*)chain_compose<DK>, dim3((unsigned)(nseq * (DV / 16))), 128, args, smem, p.stream));
        prof_end(p.stream);
    }
    constexpr int smem = DV * LD * 2;
    prof_begin("chain_apply", p.stream);
    void* args[] = {(void*)&sg, (void*)&p.O, (void*)&p.L, (void*)&seg_tokens, (void*)&plan.nseg};
    PF_CUDA_TRY(launch_early((const void*)chain_apply<DK, DV>, dim3((unsigned)((seg_tokens + 127) / 128), (unsigned)(nseq * (plan.nseg - 1))), 256,
                             args, smem, p.stream));
    prof_end(p.stream);
    count_launch(2);
    return PF_OK;
}

}  // namespace

double chain_estimate_us(const Problem& p) { return make_plan(p).us; }
double chain_short_us(const Problem& p) { return make_plan(p).short_us; }

size_t chain_workspace_bytes(const Problem& p) { return carve(p, make_plan(p)).total; }
bool chain_needs_workspace(const Problem& p) { return make_plan(p).nseg > 1; }

bool chain_supported(const Problem& p) {
    return p.in_dtype == PF_DTYPE_BF16 && p.L >= 1 && (long long)p.B * p.H * (p.d_v / 32) <= 0x7fffffffLL &&
           (long long)p.L * p.r <= 0x7fffffffLL;
}

int chain_forward(const Problem& p, void* workspace) {
    const ChainPlan plan = make_plan(p);
    ChainSeg sg{};
    if (plan.nseg > 1) {
        const ChainCarve c = carve(p, plan);
        uint8_t* ws = (uint8_t*)workspace;
        sg = {(__half*)(ws + c.R), (__half*)(ws + c.P), (float*)(ws + c.D), (float*)(ws + c.Xi), (__half*)(ws + c.start)};
    }
    const int st = p.d_k == 128 ? launch_rank<128>(p, plan, sg) : launch_rank<64>(p, plan, sg);
    if (st != PF_OK || plan.nseg == 1) return st;
    if (p.d_k == 128) return p.d_v == 128 ? launch_seg_tail<128, 128>(p, plan, sg) : launch_seg_tail<128, 64>(p, plan, sg);
    return p.d_v == 128 ? launch_seg_tail<64, 128>(p, plan, sg) : launch_seg_tail<64, 64>(p, plan, sg);
}

}  // namespace pf
