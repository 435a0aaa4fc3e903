// chain: the chunk form in ONE kernel without any hand-off through memory; a CTA walks a sequence (or a segment of one).
//
// A sequence is walked in blocks of up to 64 rows (64 / r tokens).  From Theorem 3.2, with rows m, S the state before the block:
//     T  = (I + Mstrict (.) (diag(beta) K K^T))^{-1} diag(beta)                      (does not depend on S)
//     P  = (Q K^T) (.) Mincl                                                         (does not depend on S)
//     U' = T (V - K S^T),       O = Q S^T + P U',       S <- S + U'^T K
// W = T K and Uh = T V are never formed: T is applied to V - K S^T, which is rounded when what the state predicts of V is out of it.  Three products of a
// block depend on S one after another: R = V - K S^T, U' = T R and the update.  All are tcgen05 products of 128 rows j (d_v = 64: half of them nobody's) whose A operand lies
// in tensor memory and whose B operand is a tile of shared memory as TMA or the preparing warps left it.  S stays in tensor memory as the
// fp32 accumulator of its update; between two products the chain warps convert an accumulator to the next one's fp16 operand.
//
// Warps (their registers moved to where they are needed):
//   chain (8)     fp32 accumulators -> fp16 operands: -S, R, U' in turn, 32 rows j and half of the columns each
//   products (3)  one warp each for the chain's, the output's (O^T = S Q^T + U'^T P^T) and the Gram products ([G | P^T] = K [K^T | Q^T], 64
//                 rows, from the bf16 tiles as they land)
//   solve (2 x 4) T of every other block: G from tensor memory, the inverse on mma.sync
//   convert (4)   K, Q -> fp16 in place, P out of tensor memory into shared memory
//   output (4)    O^T out of tensor memory into the rows of O;  and one warp issues the copies
// A stage of shared memory holds what the chain needs of one block: K, Q (fp16, the rows of Q behind those of K), P, T (fp16), V (bf16 as
// it came, added to R's accumulator as V^T times an identity).
//
// What bounds it: the three trips of a block (issue 4 to 8 products at 30 cycles each, tensor memory to registers and back), 2.2 k cycles at
// d = 128 with everything but the chain's own warps switched off, drawn out to 2.6 - 3 k by the others: all products go through one
// queue, in which those of 64 rows or few columns take as long as large ones (26 - 32 cycles; so G and P^T are one product: 16 products less
// a block, 133.8 -> 131.3 us at the first size below), and the warps share issue slots (so whoever waits off the chain's path does it at
// named barriers) and the instruction cache (so what is off the chain's path is written small).  148 CTAs at r = 1 move 5.5 TB/s, 84 % of
// what a copy reaches.  Measured (us, before: the same blocks on
// warp-level products, a warp carrying 16 rows j in registers; a shared-memory read of every tile by every such warp): 256 sequences of
// 1024, d = 128, r = 2: 227 -> 130 (calls on other inputs one after another; 228 -> 113 on the same); 128 of 4096, d = 64, r = 4: 340 -> 282 (336 -> 275); 48 of 1999, 64 x 128,
// r = 3: 144 -> 81 (2 segments); 4 of 16384, d = 128, r = 1: 135 -> 76 (segments); 32 of 2048, d = 128, r = 1: 68 -> 53 (the tcgen05 kernel in one launch before).
// Measured and not taken: the update's and V - K S^T's products in halves, so that one half is converted while the other is being multiplied (the
// probe's 1.6 k cycles have it; here 412 us against 389 at 32 sequences of 8192: more instructions); the output's products issued by the chain's
// warp (462); one election per product instead of per group (427 against 420 then, 179 against 146 with all SMs busy); products in loops on
// the chain's path too (489).  S K^T and S Q^T as one product (8 products less a block, but the larger one on the chain's path: 131 -> 136 at 256
// sequences, 290 -> 322 at d = 64, r = 4).  The chain's warps at named barriers too, one warp watching the products' ends for them (293 -> 328).
// V in one buffer apart from the stages, which makes room for one more (142.6 -> 152.4, 128 sequences of 2048, d = 64, r = 4).  The
// state before the last block's update in V - K S^T, with U'^T K K^T of the two blocks in its place (172 us at 256 sequences: 20 products more).
// What counts besides the chain's latency: instructions that are fetched (what all warps execute in a block is about 40 KB; 49 KB of it, in a form with one more role, missed
// the instruction cache in 23 % of the requests instead of 5 and took 20 % more time), so that a wait is a few instructions and its failure is reported once a
// role; and no warps that poll mbarriers but those that watch for others.
// Measured and not taken: the chain's warps meeting at a named barrier and the first of them issuing (128 us against 116 at 256 sequences, 314 against 264 at
// 128 of 4096, d = 64); a predicate on every product instead of a branch around all of a step (twice the instructions); an L2 prefetch of the next tiles (128 of 4096, d = 64:
// 359 against 338 without, at the time; level elsewhere); W = T K formed ahead, U' = T V - W S^T, two dependent products instead of three (128 of 4096, d = 64, r = 4: 298, in turn with 291 without; slower at d = 128): T is then
// applied to all of V and not to what the state leaves of it, and W is rounded, which costs up to 1.4 times the error where the state predicts V
// (d = 64, r = 4, beta to 2, V = S* K, relative L2 error of O: 3.7e-4, 2.7e-4 without).
//
// Range: V - K S^T and U' are packed to fp16 like every other operand, and K S^T reaches sqrt(d_k) times the largest entry of S, so
// that a state well inside fp16's 65504 can overflow them.  What overflows leaves its row of S infinite or NaN to the end of the walk
// (infinity times anything is infinite or NaN), so one look at each row when the walk is over finds it and the blocks pay nothing:
// its rows are then walked once more, token by token in fp32 (walk_fp32).
//
// The inverse of I - N, N = -A: warp w of a team owns rows 16 w .. 16 w + 15 of G, forms N's blocks there and D_w = (I - N_ww)^{-1} by its Neumann product,
// and after one exchange through shared memory column block w of X: X_ww = D_w, X_iw = D_i sum_k N_ik X_kw, each X_iw^T left in
// registers as the operand of the next (through shared memory and in loops: 58.1 us instead of 56.5, 148 sequences of 1024, r = 2).
#include <float.h>

#include <atomic>

#include "pf_common.cuh"
#include "pf_tc.cuh"
#include "pf_tc_prims.cuh"

namespace pf {

using namespace tc;

namespace {

constexpr int NB = 64;               // rows per block
constexpr int MOST_PARTS = 30;       // parts of walks in a CTA's share

struct ChainMaps {
    CUtensorMap q, k, v;
};

struct ChainGeo {
    int L, d_v, nblk;
    int nseg, seg_blk;  // segments per sequence (1: none) and blocks per segment
    int first_blk;      // blocks of the first segment
    int share;          // SHARED: blocks of a CTA, and
    int total;          // of all of them
    float* hand;        // [CTAs] states that go from one CTA to another, [d_k i][d_v j]
    int *handed, *finished;     // [CTAs] each: warps that have handed over; the CTA's outputs are written
    int* lost;          // [sequences] a response has left fp16's range (null: nobody asks, ChainPlan::rewalk)
    int rm;             // strict-mask group size (Problem::mask_group)
    int exact;          // PF_STEP_EXACT
    int clear;          // set the status word to 0
    const __nv_bfloat16 *q, *k, *v, *beta;      // the inputs once more, for walk_fp32
    const float* S0;
    float *O, *S_final;
};

// four 8 x 8 matrices to shared memory (transposed): lane l has the address of row l % 8 of matrix l / 8
__device__ __forceinline__ void stmatrix_x4(uint32_t saddr, const uint32_t (&r)[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(saddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t saddr, const uint32_t (&r)[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(saddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// eight bf16 -> eight fp16
__device__ __forceinline__ uint4 bf16_to_half8(uint4 x) {
    uint32_t* w = (uint32_t*)&x;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = pack_h2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
    return x;
}

template <int DK, int R, int JS>
struct ChainSmem {
    static constexpr int C = NB / R;                              // tokens per block
    static constexpr int CP = (C + 15) / 16 * 16;                 // ... in tiles of 16
    static constexpr int k_bytes = NB * DK * 2, q_bytes = CP * DK * 2;
    static constexpr int t_bytes = NB * 128, p_bytes = CP * 128, v_bytes = NB * JS * 2;
    // slabs of 64 columns, in each the rows of K and then those of Q: one operand of NB + CP rows
    static constexpr int rows = NB + CP, k_off = 0, q_off = NB * 128, p_off = k_bytes + q_bytes;
    static constexpr int stage = p_off + p_bytes;
    static constexpr int tx_bytes = k_bytes + C * DK * 2;         // what the copies of a block's K and Q bring
};

// Barriers (mbarriers); those of the rings of shared memory follow (ChainCfg).
enum {
    B_SP = 0,       // chain: fp16 copy of S published
    B_UD = 1,       // products: U' complete
    B_UP = 2,       // chain: its fp16 copy published
    B_SD = 3,       // products: S complete
    B_QD = 4,       // output products: Q S^T complete
    B_OD = 5,       // [2] output products: O^T complete
    B_OFREE = 7,    // [2] output: O^T read
    B_GD = 9,       // Gram products: G and P^T complete
    B_RD = 10,      // products: V^T - S K^T complete
    B_RP = 11,      // chain: its fp16 copy published
    B_END = 12,     // [4] the two chain warps of a quarter, when a walk is over
    B_RINGS = 16
};
constexpr int TEAMS = 2;             // solve teams
// warps: 0-7 chain, 8-11 output, 12-15 conversion, then the solve teams, then products of the chain, products of the output, Gram products,
// copies
constexpr int W_OUT = 8, W_CONV = 12, W_SOLVE = 16, W_MMA = W_SOLVE + 4 * TEAMS, W_MMA_OUT = W_MMA + 1, W_GRAM = W_MMA + 2, W_LOAD = W_MMA + 3,
              CHAIN_THREADS = 32 * (W_MMA + 4);

// Registers per thread: the launch's, and what each warpgroup makes of them (the sum is the launch's)
constexpr int REGS = 72, REGS_CHAIN = 80, REGS_OUT = 48, REGS_CONV = 48, REGS_ISSUE = 48, REGS_SOLVE = 88;
static_assert(2 * REGS_CHAIN + REGS_OUT + REGS_CONV + REGS_ISSUE + TEAMS * REGS_SOLVE <= REGS * CHAIN_THREADS / 128, "registers of the launch");
template <int N>
__device__ __forceinline__ void set_registers() {
    if (N > REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// X while it is being formed: the ten 16 x 16 blocks on and below the diagonal, one after another, rows of 32 bytes whose halves are exchanged in
// every other group of four rows (so that eight rows of a half meet no bank twice)
constexpr int XS_BYTES = 10 * 512;
__device__ __forceinline__ uint32_t xs_block(int i, int k) { return (uint32_t)((i * (i + 1) / 2 + k) * 512); }
__device__ __forceinline__ uint32_t xs_lane(int row, int half) { return (uint32_t)(row * 32 + ((half ^ ((row >> 2) & 1)) << 4)); }
// Rows n = 0 .. 63, columns k = 16 c .. 16 c + 15 of the identity (bf16, unswizzled K-major) for c = 0 .. 3 out of one strip of 8 x 8 blocks, zeros but
// for two: the columns' halves come from places 7 blocks apart, the four operands start two blocks apart.
struct IdStrip {
    static constexpr int blocks = 21, bytes = blocks * 128;
    // (block 6 - 2 c + g + 7 h is rows 8 g .., half h of the columns: the identity's where g = 2 c + h)
    __device__ static bool one(int e) { return (e >> 6 == 6 || e >> 6 == 14) && (e >> 3 & 7) == (e & 7); }     // element e of the strip
    __device__ static uint64_t desc(uint32_t base, int c) { return make_desc_ns(base + (6 - 2 * c) * 128, 7 * 128, 128); }
};

constexpr int SMEM_MOST = 226 * 1024;
template <int DK, int R, int DV>
struct ChainCfg {
    using SM = ChainSmem<DK, R, DV>;
    // as many stages as fit, up to six; their V and T behind all of the rest
    static constexpr int fit = (SMEM_MOST - TEAMS * (XS_BYTES + 512) - IdStrip::bytes) / (SM::stage + SM::v_bytes + SM::t_bytes), NS = fit < 6 ? fit : 6;
    static constexpr int v_off = NS * SM::stage, t_off = v_off + NS * SM::v_bytes;
    static constexpr int xs_off = t_off + NS * SM::t_bytes;       // per team: X (unscaled) while it is being formed
    static constexpr int beta_off = xs_off + TEAMS * XS_BYTES;    // per team: 64 step sizes, of two blocks in turn
    static constexpr int id_off = beta_off + TEAMS * 512;         // identity (IdStrip)
    static constexpr int total = id_off + IdStrip::bytes;
    // barriers of the stages, after the others: a block's tiles landed, a block prepared, a block's stage free
    static constexpr int LAND = B_RINGS, FULL = LAND + NS, EMPTY = FULL + NS, count = EMPTY + NS;
};
// a ring's slot and the parity of its present round
template <int N>
struct RingPos {
    int i = 0, phase = 0;
    __device__ __forceinline__ void next() {
        if (++i == N) {
            i = 0;
            phase ^= 1;
        }
    }
};

// Tensor memory: columns.  All 512 are this CTA's, so that they are these very addresses: constants, where a base read from shared memory
// would go through a register to each product.
constexpr uint32_t T_S = 0;          // S, fp32 [j][i]
constexpr uint32_t T_S16 = 128;      // -S, fp16 pairs
constexpr uint32_t T_R = 192;        // V^T - S K^T, then U'^T over it, fp32 [j][m]
constexpr uint32_t T_R16 = 256;      // V^T - S K^T and
constexpr uint32_t T_U16 = 288;      // U'^T in fp16 pairs
constexpr uint32_t T_G = 320;        // G, fp32 [m][m'] (16 rows in each quarter of the lanes, as products of 64 rows are laid out)
constexpr uint32_t T_P = 384;        // P^T before its mask, fp32 [m][t], likewise: behind T_G, one product
template <int CP> constexpr int O_BUFS = CP > 32 ? 1 : 2;         // O^T, fp32 [j][t]: of two blocks in turn where there is room
template <int CP> __device__ __forceinline__ uint32_t o_cols(int b) { return CP > 32 ? 448u : 448u + 32u * (b & 1); }

// How the walks are given to CTAs: a sequence each; a segment's walk each; or all walks, one after another, in equal shares.
enum { WHOLE = 0, SEGMENTS = 1, SHARED = 2 };

// A walk, or the part of one, that a CTA of the kernel works on.
struct ChainPart {
    int b0, nblk;       // first block of the sequence's, number of blocks
    int width;          // rows j of the state: d_v, or d_k for the response to the segment's start state
    bool response;
    const float* S0;    // start state of this sequence, or null
    float* O;           // rows of O of the first block (response: fp16 rows)
    float* S_end;       // end state [i][j] (response: fp16 [j][i] without its diagonal), or null
    float* D;           // response: the end state's diagonal
    long long seq;
    // SHARED:
    int hand_in, hand_out;      // the state comes from there, goes there (-1: does not)
    int before, walk;           // blocks of the walk before this part, and of all of it
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

// A walk: segment s of sequence seq, the walk itself or the response to its start state, n blocks from block b0 of the sequence on.
template <int DK, int C, int MODE>
__device__ __forceinline__ ChainPart walk_of(const ChainGeo& g, const ChainSeg& sg, const float* S0, float* O, float* S_final, long long seq, int s, bool response, int b0, int n) {
    const long long row0 = seq * g.L + (long long)b0 * C, slot = seq * g.nseg + s;
    ChainPart part;
    part.seq = seq;
    part.b0 = b0;
    part.nblk = part.walk = n;
    part.response = MODE != WHOLE && response;
    part.width = part.response ? DK : g.d_v;
    part.S0 = s == 0 && S0 ? S0 + seq * DK * g.d_v : nullptr;
    part.O = part.response ? (float*)(sg.R + row0 * DK) : O + row0 * g.d_v;
    if (MODE == WHOLE || (MODE == SHARED && g.nseg == 1)) part.S_end = S_final ? S_final + seq * DK * g.d_v : nullptr;
    else part.S_end = part.response ? (float*)(sg.P + slot * DK * DK) : sg.Xi + slot * DK * g.d_v;
    part.D = MODE == WHOLE ? nullptr : sg.D + slot * DK;
    part.hand_in = part.hand_out = -1;
    part.before = 0;
    return part;
}
// WHOLE, SEGMENTS: the walk of this CTA
template <int DK, int C, int MODE>
__device__ __forceinline__ ChainPart own_walk(const ChainGeo& g, const ChainSeg& sg, const float* S0, float* O, float* S_final) {
    if (MODE == WHOLE) return walk_of<DK, C, MODE>(g, sg, S0, O, S_final, blockIdx.x, 0, false, 0, g.nblk);
    const int per_seq = 2 * g.nseg - 1, x = (int)(blockIdx.x % per_seq), s = x >= g.nseg ? 1 + x - g.nseg : x, b0 = s * g.seg_blk;
    return walk_of<DK, C, MODE>(g, sg, S0, O, S_final, blockIdx.x / per_seq, s, x >= g.nseg, b0, min(g.seg_blk, g.nblk - b0));
}
// SHARED: the walks lie one after another on a line of blocks (per sequence the first segment's, then of each further one the walk from zero and the response) that
// is cut into shares of equal length, no shorter than any walk, so that a walk lies in one share or across one cut.  The share behind a cut comes first in its CTA's
// time and takes the walk's first blocks; the one before it has the rest, at its end, when the state has long been handed over: nobody waits, and no SM idles while
// others walk (the wrap-around rule for preemptive schedules, R. McNaughton, 1959).  Shares go to CTAs from the last one on, so that who waits has the higher index.
__device__ __forceinline__ int share_of_cta() { return (int)(gridDim.x - 1 - blockIdx.x); }
// The part that holds block x of the line.
template <int DK, int C>
__device__ __forceinline__ ChainPart part_at(const ChainGeo& g, const ChainSeg& sg, const float* S0, float* O, float* S_final, int x, int lo, int hi) {
    const int per_seq = 2 * g.nblk - g.first_blk, seq = x / per_seq;
    int off = x - seq * per_seq, s = 0, n = g.first_blk, start = 0;
    bool response = false;
    if (off >= g.first_blk) {
        off -= g.first_blk;
        s = off / (2 * g.seg_blk);
        off -= s * 2 * g.seg_blk;
        n = min(g.seg_blk, g.nblk - g.first_blk - s * g.seg_blk);
        response = off >= n;
        start = g.first_blk + s * 2 * g.seg_blk + (response ? n : 0);
        ++s;
    }
    start += seq * per_seq;                                       // the walk's place on the line
    ChainPart part = walk_of<DK, C, SHARED>(g, sg, S0, O, S_final, seq, s, response, s == 0 ? 0 : g.first_blk + (s - 1) * g.seg_blk, n);
    part.nblk = min(start + n, hi) - max(start, lo);
    if (start < lo) part.hand_out = share_of_cta() - 1;           // the first blocks of the walk, whose rest the share before this one has
    else if (start + n > hi) {
        part.hand_in = share_of_cta();
        part.before = n - part.nblk;
        part.b0 += part.before;
        part.O = response ? (float*)((__half*)part.O + (long long)part.before * C * DK) : part.O + (long long)part.before * C * g.d_v;
    }
    return part;
}
// What a CTA works on: one walk, or the parts of its share.
template <int MODE>
struct ChainWork {
    static constexpr bool shared = MODE == SHARED;
    const ChainPart& own;       // (of the first part, SHARED)
    const ChainPart* parts;     // SHARED
    int n, count;               // parts, and blocks of all of them
    __device__ __forceinline__ int size() const { return shared ? n : 1; }
    __device__ __forceinline__ const ChainPart& operator[](int i) const { return shared ? parts[i] : own; }
};

// Eight rows of S from row `row0` on, once more: the recurrence token by token in fp32, by one warp, four lanes to a row.  Not a fast
// path: it is there so that every state that fp16 can hold gives a finite result, whatever the products with it reach.
template <int DK, int R>
__device__ __forceinline__ void walk_fp32(const ChainArgs& args, const ChainPart& part, long long seq, int row0) {
    constexpr int C = NB / R, NI = DK / 4;                        // columns i per lane
    const ChainGeo& g = args.g;
    const int lane = threadIdx.x & 31, i0 = (lane & 3) * NI, j = row0 + (lane >> 2);
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
        d += __shfl_xor_sync(0xffffffffu, d, 1);
        return d + __shfl_xor_sync(0xffffffffu, d, 2);
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
        if ((lane & 3) == 0) part.O[(long long)t * g.d_v + j] = o;
    }
    if (part.S_end)
#pragma unroll
        for (int n = 0; n < NI; ++n) part.S_end[(long long)(i0 + n) * g.d_v + j] = S[n];
}

// A role's waits on mbarriers.  The first that runs out leaves its code; those after it give up at the first try, so that each CTA ends by itself.
struct Waits {
    uint32_t bar;           // shared address of the first barrier
    int tries = WAIT_TRIES, code = 0;
    __device__ __forceinline__ explicit Waits(uint32_t bar) : bar(bar) {}
    template <bool LAZY = true>
    __device__ __forceinline__ void wait(int which, int parity, int code_if_not) {
        if (!mbar_wait_tries<LAZY>(bar + 8 * which, (uint32_t)parity, tries)) {
            if (code == 0) code = code_if_not;
            tries = 1;
        }
    }
    __device__ __forceinline__ bool ok() const { return code == 0; }
};

// byte offsets of a lane's row address for ldmatrix.x4 within a slab of 128-byte swizzled rows; the K-step kk of 16 columns
// is at off ^ (kk << 5), everything else is added
__device__ __forceinline__ uint32_t lane_off(int row, int half) { return (uint32_t)row * 128u + (uint32_t)((half ^ (row & 7)) << 4); }

// Most warps wait at named barriers, which take no issue slots: of all that watch mbarriers (which has to be done in a loop) for the end of
// a product there is one warp, the one that issued it, and it passes the news on.  Those that wait at named barriers never give up, so
// whoever watches an mbarrier takes part in them to the end, also when it has given up (`ok`).
enum {
    N_TEAM = 1,     // [2] solve teams
    N_GD = 5,       // [team] Gram products -> solve: G complete
    N_GFREE = 7,    // solve and conversion -> Gram products: G and P^T read
    N_PD = 8,       // Gram products -> conversion: P^T complete (and nothing reads the block's K and Q as bf16 any more)
    N_OD = 10       // [2] output products -> output: O^T complete
};
__device__ __forceinline__ void named_arrive(int id, int nthreads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory"); }
// (after a wait for a product's mbarrier, by a whole warp)
__device__ __forceinline__ void pass_on(int id, int nthreads) {
    tc_fence_after();
    tc_fence_before();
    named_arrive(id, nthreads);
}
// Products over several K-steps, by one elected thread, descriptors by their low words (a stage's address changes nothing else).  One election for all products of
// a step and their commits: an election each is half as many instructions again, and a predicate on each instead of a branch around all twice as many.
// Products execute in the order of their issue only where accumulator and shape are the same.  So all products that add to one
// accumulator without a wait between them have the same N and the same columns: the upper triangles of T and P are zeros that are multiplied (a
// product of few columns takes 26 - 32 cycles, one of 64 columns 35).
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);          // SBO 1024 bytes, version, 128-byte swizzle
__device__ __forceinline__ uint64_t desc_lo(uint32_t lo) { return ((uint64_t)DESC_HI << 32) | lo; }
__device__ __forceinline__ uint32_t lo_of(uint32_t saddr, uint32_t slab_bytes = 16) { return (saddr >> 4) | (slab_bytes >> 4 << 16); }
// D [128 x N] (+)= A (tensor memory; NEG: -A) B^T: B K-major (MN false) or MN-major, KSTEPS K-steps, slabs of B_ROWS rows
template <bool MN, int N, int KSTEPS, int B_ROWS, bool NEG = false>
__device__ __forceinline__ void products_ta(uint32_t d, uint32_t a, uint32_t b_lo, bool acc) {
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk)
        mma_f16_ta(d, a + 8 * kk, desc_lo(b_lo + (kstep_off<MN ? L_SWMN : L_SWK, B_ROWS>(kk) >> 4)), make_idesc(N, false, MN, NEG), acc || kk > 0);
}
// D [64 x N] = A B^T, B [N rows] K-major bf16 in shared memory, in slabs of ROWS rows, A its first 64 rows
template <int N, int K, int ROWS>
__device__ __forceinline__ void products_ss(uint32_t d, uint32_t b_base) {
    constexpr uint32_t idesc = (make_idesc(N, false, false, false) & ~(31u << 24)) | (4u << 24) | (1u << 7) | (1u << 10);     // (64 rows, bf16)
    const uint32_t b = lo_of(b_base);
#pragma unroll
    for (int kk = 0; kk < K / 16; ++kk)
        mma_f16(d, desc_lo(b + (kstep_off<L_SWK, ROWS>(kk) >> 4)), desc_lo(b + (kstep_off<L_SWK, ROWS>(kk) >> 4)), idesc, kk > 0);
}
__device__ __forceinline__ void commit_at(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// a warp's part of an operand in shared memory is written
__device__ __forceinline__ void publish_smem(uint32_t b) {
    fence_async_smem();
    mbar_arrive_at(b);
}
// PIECES 16-byte pieces of each of THREADS threads: bf16 -> fp16 in place (elementwise, so the swizzled layout is untouched), several per
// round, so that their loads are in flight together
template <int PIECES, int THREADS>
__device__ __forceinline__ void convert_pieces(uint8_t* at, int tid) {
    uint4* p = (uint4*)at + tid;
    constexpr int ROUND = PIECES % 4 == 0 ? 4 : PIECES % 3 == 0 ? 3 : 5;
    static_assert(PIECES % ROUND == 0, "pieces per round");
#pragma unroll 1
    for (int e0 = 0; e0 < PIECES; e0 += ROUND) {
        uint4 y[ROUND];
#pragma unroll
        for (int e = 0; e < ROUND; ++e) y[e] = p[(e0 + e) * THREADS];
#pragma unroll
        for (int e = 0; e < ROUND; ++e) p[(e0 + e) * THREADS] = bf16_to_half8(y[e]);
    }
}

// r = (I - N)^{-1} of a strictly lower triangular 16 x 16 block as an accumulator fragment, from the A-operand fragments of N and N^T: the product
// (I + N)(I + N^2)(I + N^4)(I + N^8) as far as N's powers are not zero (LAST: the last of them; `deep`: up to N^8).  The diagonals of N and N^2 are +0, so that adding
// the identity (`one`: its part of elements 0 and 3) is an OR, exact in fp16, and the first two factors need no start value.
template <int LAST>
__device__ __forceinline__ void neumann_product(float (&r)[2][4], const uint32_t (&n)[4], const uint32_t (&nt)[4], uint32_t one, bool deep) {
    auto mul = [](float (&c)[2][4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {     // (b: fragment of the second factor transposed)
        mma_acc(c[0], a, b0, b2, false);
        mma_acc(c[1], a, b1, b3, false);
    };
    float c[2][4];
    uint32_t p[4], pt[4], q[4];                                   // the power at hand, its transpose, what has been multiplied
    mul(c, nt, n[0], n[1], n[2], n[3]);                           // (N^2)^T
    frag_pack(pt, c);
    q[0] = n[0] | one; q[1] = n[1]; q[2] = n[2]; q[3] = n[3] | one;
    mul(r, q, pt[0] | one, pt[1], pt[2], pt[3] | one);
    if (LAST == 2 && !deep) return;
    mul(c, n, nt[0], nt[1], nt[2], nt[3]);                        // N^2
    frag_pack(p, c);
    float c4[2][4];
    mul(c, pt, p[0], p[1], p[2], p[3]);                           // (N^4)^T
    if (deep) mul(c4, p, pt[0], pt[1], pt[2], pt[3]);             // N^4
    frag_pack(q, r);
    frag_pack(pt, c);
    frag_mul(r, q, pt);                                           // (r stays fp32: only what is added to it has passed through fp16)
    if (!deep) return;
    frag_pack(p, c4);
    mul(c, pt, p[0], p[1], p[2], p[3]);                           // (N^8)^T
    frag_pack(q, r);
    frag_pack(pt, c);
    frag_mul(r, q, pt);
}

// ---------------------------------------------------------------------------------------------------------------------
// solve team: T of blocks b = team, team + TEAMS, ...
// ---------------------------------------------------------------------------------------------------------------------
template <int DK, int R, int JS, int MODE>
__device__ __forceinline__ void solve_role(const ChainGeo& g, ChainWork<MODE> work, const __nv_bfloat16* __restrict__ beta, uint8_t* smem,
                                           uint32_t bar, int team, int tid) {
    using CFG = ChainCfg<DK, R, JS>;
    using SM = ChainSmem<DK, R, JS>;
    constexpr int C = SM::C;
    const int w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const int L = g.L;
    const uint32_t xs_b = smem_u32(smem) + CFG::xs_off + team * XS_BYTES;
    const uint32_t offA = lane_off(lane & 15, lane >> 4), offN = lane_off((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
    const uint32_t xs_a = xs_b + xs_lane(lane & 15, lane >> 4) + xs_block(w, 0), xs_n = xs_b + xs_lane((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
    // the strict mask on the packed values of the diagonal tile, and of the one left of it (groups of three rows reach across the edge of a tile)
    uint32_t keep[4], keep_left[4];
    {
        const int lim0 = (16 * w + gq) / g.rm * g.rm - 16 * w, lim1 = (16 * w + gq + 8) / g.rm * g.rm - 16 * w;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = 8 * (e / 2) + 2 * t4, lim = e % 2 ? lim1 : lim0;
            keep[e] = (c < lim ? 0xFFFFu : 0u) | (c + 1 < lim ? 0xFFFF0000u : 0u);
            keep_left[e] = (c < lim + 16 ? 0xFFFFu : 0u) | (c + 1 < lim + 16 ? 0xFFFF0000u : 0u);
        }
    }
    const uint32_t one = gq == 2 * t4 ? 0x3C00u : gq == 2 * t4 + 1 ? 0x3C000000u : 0u;      // the identity's part of elements 0 and 3 of a fragment
    int b = team;                                                 // (of the CTA's blocks)
#pragma unroll 1
    for (int i = 0, at = 0; i < work.size(); at += work[i].nblk, ++i) {
    const ChainPart& part = work[i];
    const int end = at + part.nblk;
    const __nv_bfloat16* bs = beta + part.seq * L * R;
    // (the bits as loaded: a conversion next to the load would make every thread wait for it there, a block ahead of its use)
    auto read_beta = [&](int b) {                                 // rows past the block or the sequence have step size zero
        uint16_t x = 0;
        const int tok = (part.b0 + b - at) * C;
        if (tid < min(C, L - tok) * R)
            asm volatile("ld.global.nc.b16 %0, [%1];" : "=h"(x) : "l"(bs + (long long)tok * R + tid));
        return x;
    };
    uint16_t breg = b < end ? read_beta(b) : 0;
#pragma unroll 1
    for (; b < end; b += TEAMS) {
        const int st = b % CFG::NS;
        const uint32_t t_b = smem_u32(smem) + CFG::t_off + st * SM::t_bytes;
        // (two in turn: another warp may still be scaling T of the block before)
        float* sBeta = (float*)(smem + CFG::beta_off + team * 512 + (b / TEAMS & 1) * 256);
        if (tid < NB) sBeta[tid] = __uint_as_float((uint32_t)breg << 16);
        if (b + TEAMS < end) breg = read_beta(b + TEAMS);
        named_bar(N_GD + team, 160);                              // (and the step sizes)
        tc_fence_after();
        const uint32_t t_g = T_G + ((uint32_t)(32 * w) << 16);
        uint32_t x[8];                                            // 16 columns of G, rows 16 w .. 16 w + 15, as mma.sync's accumulators
        const int m0 = 16 * w + gq, m1 = m0 + 8;
        if (g.exact) {
            // |k|^2 is the diagonal of G; beta' = (1 - e^{-beta |k|^2}) / |k|^2
            tmem_ld_frag<16>(t_g + 16 * w, x);
            tmem_ld_wait();
            if ((gq >> 1) == t4)
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const float n = __uint_as_float(h == 0 ? (gq & 1 ? x[1] : x[0]) : (gq & 1 ? x[7] : x[6]));
                    if (n > 0.f) sBeta[m0 + 8 * h] = -expm1f(-sBeta[m0 + 8 * h] * n) / n;
                }
            __syncwarp();
        }
        // ---- N = -A = -Mstrict (.) (diag(beta) G): its blocks left of the diagonal go to the other warps, the diagonal one stays as an A operand
        const float b0 = -sBeta[m0], b1 = -sBeta[m1];
        uint32_t nf[4];
#pragma unroll 1
        for (int nb = 0;; ++nb) {
            tmem_ld_frag<16>(t_g + 16 * nb, x);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 4; ++e) nf[e] = pack_h2((e % 2 ? b1 : b0) * __uint_as_float(x[2 * e]), (e % 2 ? b1 : b0) * __uint_as_float(x[2 * e + 1]));
            if (R == 3 && nb + 1 == w)
#pragma unroll
                for (int e = 0; e < 4; ++e) nf[e] &= keep_left[e];
            if (nb == w) break;
            stmatrix_x4(xs_a + nb * 512, nf);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) nf[e] &= keep[e];
        tc_fence_before();
        if (b + 1 < work.count) named_arrive(N_GFREE, 288);
        // ---- D_w = (I - N_ww)^{-1} (Neumann product, N nilpotent) for the other warps
        uint32_t y0[4];                                           // X_ww^T as an A operand
        {
            uint32_t nt[4], df[4];
            float dd[2][4];
            nt[0] = movmatrix(nf[0]); nt[1] = movmatrix(nf[2]); nt[2] = movmatrix(nf[1]); nt[3] = movmatrix(nf[3]);
            neumann_product<(R == 4 ? 2 : 4)>(dd, nf, nt, one, g.rm == 1);
            frag_pack(df, dd);
            stmatrix_x4(xs_a + w * 512, df);
            y0[0] = movmatrix(df[0]); y0[1] = movmatrix(df[2]); y0[2] = movmatrix(df[1]); y0[3] = movmatrix(df[3]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 bb = *(const float2*)(sBeta + 16 * w + 8 * h + 2 * t4);
                dd[h][0] *= bb.x; dd[h][1] *= bb.y; dd[h][2] *= bb.x; dd[h][3] *= bb.y;
            }
            frag_pack(df, dd);
            stmatrix_x4(t_b + w * 2048 + (offA ^ (uint32_t)(w << 5)), df);
        }
        named_bar(N_TEAM + team, 128);
        // ---- down the column: X_iw = D_i sum_k N_ik X_kw, transposed, in registers; T = X diag(beta)
        uint32_t y[3][4];                                         // X_kw^T of k = w, w + 1, w + 2
#pragma unroll
        for (int e = 0; e < 4; ++e) y[0][e] = y0[e];
#pragma unroll
        for (int n = 1; n < 4; ++n) {
            const int i = w + n;
            if (i > 3) break;
            float c[2][4], z[2][4];
            uint32_t f[4], a[4];
#pragma unroll
            for (int k = 0; k < n; ++k) {
                ldmatrix_x4(a, xs_n + xs_block(i, w + k));
                mma_acc(c[0], y[k], a[0], a[1], k > 0);
                mma_acc(c[1], y[k], a[2], a[3], k > 0);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = pack_h2(c[e / 2][e % 2 * 2], c[e / 2][e % 2 * 2 + 1]);
            ldmatrix_x4(a, xs_n + xs_block(i, i));
            mma_acc(z[0], f, a[0], a[1], false);
            mma_acc(z[1], f, a[2], a[3], false);
            if (n < 3) frag_pack(y[n < 3 ? n : 0], z);
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = pack_h2(-z[e / 2][e % 2 * 2] * (e % 2 ? b1 : b0), -z[e / 2][e % 2 * 2 + 1] * (e % 2 ? b1 : b0));
            stmatrix_x4_trans(t_b + i * 2048 + (offN ^ (uint32_t)(w << 5)), f);
        }
        publish_smem(bar + 8 * (CFG::FULL + st));
    }
    }
}

// Conversion: K and Q of every block to fp16 in place, once the Gram products have read them as they came, and P.  Four warps.
template <int DK, int R, int JS>
__device__ __forceinline__ void convert_role(int count, uint8_t* smem, uint32_t bar, int tid) {
    using SM = ChainSmem<DK, R, JS>;
    using CFG = ChainCfg<DK, R, JS>;
    constexpr int CP = SM::CP;
    const int w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const uint32_t p_at = smem_u32(smem) + SM::p_off + (lane_off((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1) ^ (uint32_t)(w << 5));
    int st = 0;
#pragma unroll 1
    for (int b = 0; b < count; ++b) {
        uint8_t* sg = smem + st * SM::stage;
        named_bar(N_PD, 160);
        tc_fence_after();
        // ---- P^T rows m = 16 w .. 16 w + 15, columns t; P = its transpose (.) Mincl: row m is seen by tokens t with m < (t + 1) R
        constexpr int PC = CP < 32 ? CP : 32;                     // (columns at a time)
#pragma unroll 1
        for (int t0 = 0; t0 < CP; t0 += PC) {
            uint32_t x[PC / 2];
            tmem_ld_frag<PC>(T_P + t0 + ((uint32_t)(32 * w) << 16), x);
            tmem_ld_wait();
            if (t0 + PC == CP) {
                tc_fence_before();
                if (b + 1 < count) named_arrive(N_GFREE, 288);
            }
#pragma unroll
            for (int n = 0; n < PC / 8; n += 2) {
                if (16 * w >= (t0 + 8 * n + 16) * R) continue;    // (nothing of the block of 16 tokens sees these rows: zeros from the start)
                uint32_t y[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) y[e] = pack_h2(__uint_as_float(x[4 * n + 2 * e]), __uint_as_float(x[4 * n + 2 * e + 1]));
                if (16 * w + 15 >= (t0 + 8 * n + 1) * R)          // (not all of them are seen by all tokens of the tile)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int t = t0 + 8 * (n + e / 2) + 2 * t4, m = 16 * w + 8 * (e % 2) + gq;
                        y[e] &= (m < (t + 1) * R ? 0xFFFFu : 0u) | (m < (t + 2) * R ? 0xFFFF0000u : 0u);
                    }
                stmatrix_x4_trans(p_at + st * SM::stage + t0 * 128 + n * 1024, y);
            }
        }
        convert_pieces<(SM::k_bytes + SM::q_bytes) / 2048, 128>(sg + SM::k_off, tid);
        publish_smem(bar + 8 * (CFG::FULL + st));
        if (++st == CFG::NS) st = 0;
    }
}

// Gram products (one warp): G = K K^T and K Q^T from the bf16 tiles as they landed, in products of 64 rows and NB + CP columns.
template <int DK, int R, int JS>
__device__ __forceinline__ void gram_role(int count, int* err, uint8_t* smem, uint32_t bar) {
    using SM = ChainSmem<DK, R, JS>;
    using CFG = ChainCfg<DK, R, JS>;
    const uint32_t smem_b = smem_u32(smem);
    RingPos<CFG::NS> ks;
    Waits waits(bar);
#pragma unroll 1
    for (int b = 0; b < count; ++b) {
        waits.wait(CFG::LAND + ks.i, ks.phase, 316);
        if (b > 0) named_bar(N_GFREE, 288);
        tc_fence_after();
        if (waits.ok() && elect_one()) {
            products_ss<SM::rows, DK, SM::rows>(T_G, smem_b + ks.i * SM::stage);
            commit_at(bar + 8 * B_GD);
        }
        __syncwarp();
        waits.wait(B_GD, b & 1, 311);
        pass_on(N_GD + b % TEAMS, 160);
        named_arrive(N_PD, 160);
        ks.next();
    }
    if (!waits.ok()) atomicCAS(err, 0, waits.code);
}

// The copies (one warp).  K and Q of a block are asked for when the block before in their stage is done, V with them; rows past the sequence arrive as zeros.  (Issuing a copy takes the warp some 200 cycles, five a block at d = 128.)
template <int DK, int R, int JS, int MODE>
__device__ __forceinline__ void load_role(const ChainMaps& maps, ChainWork<MODE> work, int* err, uint8_t* smem, uint32_t bar) {
    using SM = ChainSmem<DK, R, JS>;
    using CFG = ChainCfg<DK, R, JS>;
    constexpr int NS = CFG::NS;
    const uint32_t smem_b = smem_u32(smem);
    Waits waits(bar);
    RingPos<NS> ks;
    auto copy_kq = [&](const ChainPart& part, int b) {
        const uint32_t land = bar + 8 * (CFG::LAND + ks.i), at = smem_b + ks.i * SM::stage;
        const int tok = (part.b0 + b) * SM::C, seq = (int)part.seq;
        if (waits.ok() && elect_one()) {
            mbar_expect_tx_at(land, SM::tx_bytes + (part.response ? 0 : SM::v_bytes));
#pragma unroll
            for (int h = 0; h < DK / 64; ++h) {
                tma_load_4d(at + SM::k_off + h * (SM::rows * 128), &maps.k, 0, tok * R, h, seq, land);
                tma_load_4d(at + SM::q_off + h * (SM::rows * 128), &maps.q, 0, tok, h, seq, land);
            }
            if (!part.response) tma_load_4d(smem_b + CFG::v_off + ks.i * SM::v_bytes, &maps.v, 0, tok * R, 0, seq, land);
        }
        __syncwarp();
        ks.next();
    };
    int c = -NS;
#pragma unroll 1
    for (int i = 0; i < work.size(); ++i) {
        const ChainPart& part = work[i];
        const int nblk = part.nblk;
#pragma unroll 1
        for (int b = 0; b < nblk; ++b, ++c) {
            if (c >= 0) waits.wait(CFG::EMPTY + ks.i, ks.phase ^ 1, 341);
            copy_kq(part, b);
        }
    }
    if (!waits.ok()) atomicCAS(err, 0, waits.code);
}

// ---------------------------------------------------------------------------------------------------------------------
// The serial part: S in tensor memory, row j = lane j.
// ---------------------------------------------------------------------------------------------------------------------
// N columns of an fp32 accumulator, in fp16 pairs (negated) as the A operand of the next product.  (A load and its wait cost about the
// same whatever the width.)
template <int N, bool NEG>
__device__ __forceinline__ void to_operand(uint32_t src, uint32_t dst) {
    uint32_t x[N / 32][32], h[16];
#pragma unroll
    for (int c = 0; c < N / 32; ++c) tmem_ld32(src + 32 * c, x[c]);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < N / 32; ++c) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float lo = __uint_as_float(x[c][2 * e]), hi = __uint_as_float(x[c][2 * e + 1]);
            h[e] = NEG ? pack_h2(-lo, -hi) : pack_h2(lo, hi);
        }
        tmem_st16(dst + 16 * c, h);
    }
}

constexpr uint32_t HALF_INF = 0x477FF000u;     // 65520 as fp32: from there on fp16 is infinite (bits of magnitudes, so that NaN is above)

// Waits until *p >= want (one thread), about a second at most.
__device__ __forceinline__ bool wait_for_count(const int* p, int want) {
    const long long t0 = clock64();
    while (ld_acquire_gpu(p) < want)
        if (clock64() - t0 > WAIT_CYCLES) return false;
    return true;
}
__device__ __forceinline__ void add_release_gpu(int* p, int v) { asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }

// The end state (its last update is the chain's last product, so that this goes on beside the last block's output); lost: gets a bit for each quarter of the rows j that has to be walked again.
// end_bar, met: where the two warps of a quarter meet, and its parity.  Returns false if the other one does not come.
template <int DK, bool SHARE>
__device__ __forceinline__ bool end_state(const ChainGeo& g, const ChainPart& part, uint32_t* lost, uint32_t end_bar, int& met, int warp, int lane) {
    constexpr int HC = DK / 2;
    const int h = warp >> 2, quarter = warp & 3, j = 32 * quarter + lane;
    const uint32_t t_s = T_S + h * HC + ((uint32_t)(32 * quarter) << 16);
    if (SHARE && part.hand_out >= 0) {
        // (to the CTA that has the rest of the walk, as it is: what is lost is found at the walk's end)
        float* out = g.hand + (long long)part.hand_out * DK * part.width + (long long)h * HC * part.width + j;
#pragma unroll 1
        for (int c = 0; c < HC; c += 32) {
            uint32_t x[32];
            tmem_ld32(t_s + c, x);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) out[(c + e) * part.width] = __uint_as_float(x[e]);
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) add_release_gpu(g.handed + part.hand_out, 1);
        return true;
    }
    if (part.response) {
        uint32_t most = 0;                                        // (an infinity or NaN on the diagonal is not alone in its row)
        __half* P = (__half*)part.S_end + (long long)j * DK + h * HC;
#pragma unroll 1
        for (int c = 0; c < HC; c += 32) {
            uint32_t x[32];
            tmem_ld32(t_s + c, x);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (h * HC + c + e == j) {
                    part.D[j] = __uint_as_float(x[e]);
                    x[e] = 0;
                }
            if (SHARE)
#pragma unroll
                for (int e = 0; e < 32; ++e) most = max(most, x[e] & 0x7fffffffu);
#pragma unroll
            for (int e = 0; e < 32; e += 8)
                *(uint4*)(P + c + e) = make_uint4(pack_h2(__uint_as_float(x[e]), __uint_as_float(x[e + 1])), pack_h2(__uint_as_float(x[e + 2]), __uint_as_float(x[e + 3])),
                                                  pack_h2(__uint_as_float(x[e + 4]), __uint_as_float(x[e + 5])), pack_h2(__uint_as_float(x[e + 6]), __uint_as_float(x[e + 7])));
        }
        if (SHARE && most >= HALF_INF && g.lost) g.lost[part.seq] = 1;
        return true;
    }
    // (one entry tells for its row.  The end state may replace the start state, which is still needed where rows are lost, so that both warps have to know before
    //  either writes.  They meet at an mbarrier, whose wait has a limit: one of them may have given up)
    uint32_t x[32];
    tmem_ld32(t_s, x);
    tmem_ld_wait();
    const bool finite = __all_sync(0xffffffffu, fabsf(__uint_as_float(x[0])) <= FLT_MAX);
    if (lane == 0) {
        if (!finite) atomicOr(lost, 1u << quarter);
        mbar_arrive_at(end_bar);
    }
    if (!mbar_wait_tries<false>(end_bar, met)) return false;
    met ^= 1;
    if (part.S_end && !(*(volatile uint32_t*)lost >> quarter & 1)) {
#pragma unroll 1
        for (int c = 0; c < HC; c += 32) {
            tmem_ld32(t_s + c, x);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) part.S_end[(long long)(h * HC + c + e) * part.width + j] = __uint_as_float(x[e]);
        }
    }
    return true;
}

// warp `warp` of eight: rows j = 32 (warp & 3) + lane, half warp >> 2 of the columns of everything.  Returns the code of the wait that ran out, or 0.
template <int DK, int MODE>
__device__ __forceinline__ int chain_role(const ChainGeo& g, ChainWork<MODE> work, uint32_t* lost, uint32_t bar, int warp, int lane) {
    constexpr int HC = DK / 2;                                    // columns i of this warp
    const int h = warp >> 2, j = 32 * (warp & 3) + lane;
    const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
    const uint32_t t_s = T_S + h * HC + lanes, t_s16 = T_S16 + h * HC / 2 + lanes;
    const uint32_t t_r = T_R + 32 * h + lanes, t_r16 = T_R16 + 16 * h + lanes, t_u16 = T_U16 + 16 * h + lanes;
    auto publish = [&](int b) {
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_at(bar + 8 * b);
    };
    int code = 0, parity = 0, met = 0;
#pragma unroll 1
    for (int i = 0; i < work.size(); ++i) {
        const ChainPart& part = work[i];
        const float* s0 = part.S0;
        if (work.shared && part.hand_in >= 0) {
            bool ok = true;
            if (lane == 0) ok = wait_for_count(g.handed + part.hand_in, part.width / 16);
            if (!__all_sync(0xffffffffu, ok)) code = 336;
            s0 = g.hand + (long long)part.hand_in * DK * part.width;
        }
        const int width = part.width;
        // (Every further round is a trip to memory, but at d_k = 64, where there are one or two, the shorter code of two is the faster one, us with one and two: 48 sequences of
        //  1999, 64 x 64, r = 4: 88.1 and 85.2, 140 of 1000: 72.9 and 71.1; of 300, r = 2, in segments: 17.1 and 16.4.  At d_k = 128 with two and four: 16 of 333, r = 2: 21.0 and 21.2)
        constexpr int SC = DK == 64 && MODE != SHARED ? 16 : 32;  // columns a round
#pragma unroll 1
        for (int c = 0; c < HC; c += SC) {
            uint32_t x[SC], y[SC / 2];
            const float* at = s0 + (long long)(h * HC + c) * width + j;
#pragma unroll
            for (int e = 0; e < SC; ++e)
                x[e] = __float_as_uint(s0 ? (work.shared ? ld_cg_f32(at + e * width) : at[e * width]) : part.response && h * HC + c + e == j ? 1.f : 0.f);
#pragma unroll
            for (int e = 0; e < SC / 2; ++e) y[e] = pack_h2(-__uint_as_float(x[2 * e]), -__uint_as_float(x[2 * e + 1]));
            if constexpr (SC == 32) {
                tmem_st32(t_s + c, x);
                tmem_st16(t_s16 + c / 2, y);
            } else {
                tmem_st16(t_s + c, x);
                tmem_st8(t_s16 + c / 2, y);
            }
        }
        if (work.shared && i + 1 < work.size() && work[i + 1].S0 && work[i + 1].hand_in < 0)       // (the next part's, to the L2: a line of 128 bytes for each row i and quarter)
            for (int e = lane; e < HC; e += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(work[i + 1].S0 + (long long)(h * HC + e) * width + 32 * (warp & 3)));
        const int nblk = part.nblk;
#pragma unroll 1
        for (int b = 0;; parity ^= 1) {
            publish(B_SP);
            if (!mbar_wait_tries<false>(bar + 8 * B_RD, parity)) return 312;
            tc_fence_after();
            to_operand<32, false>(t_r, t_r16);
            publish(B_RP);
            if (!mbar_wait_tries<false>(bar + 8 * B_UD, parity)) return 313;
            tc_fence_after();
            to_operand<32, false>(t_r, t_u16);
            publish(B_UP);
            if (!mbar_wait_tries<false>(bar + 8 * B_SD, parity)) return 314;
            tc_fence_after();
            if (++b == nblk) break;
            to_operand<HC, true>(t_s, t_s16);
        }
        parity ^= 1;
        if (!end_state<DK, ChainWork<MODE>::shared>(g, part, lost + i, bar + 8 * (B_END + (warp & 3)), met, warp, lane)) return 315;
    }
    return code;
}

// The products of the chain (one warp).  Returns the code of the wait that ran out, or 0.
template <int DK, int R, int DV, int MODE>
__device__ __forceinline__ int mma_role(ChainWork<MODE> work, uint8_t* smem, uint32_t bar) {
    using CFG = ChainCfg<DK, R, DV>;
    using SM = ChainSmem<DK, R, DV>;
    constexpr int V_SLAB = NB * 128, K_SLAB = SM::rows * 128, CP = SM::CP, OB = O_BUFS<CP>;
    const uint32_t smem_b = smem_u32(smem);
    RingPos<CFG::NS> ks;
    auto wait = [&](int which, int parity) { return mbar_wait_tries<false>(bar + 8 * which, (uint32_t)parity); };
    int b = 0;                                                    // (of the CTA's blocks)
#pragma unroll 1
    for (int i = 0; i < work.size(); ++i) {
    const int end = b + work[i].nblk;
    const bool response = work[i].response;
#pragma unroll 1
    for (; b < end; ++b) {
        const uint32_t k_at = smem_b + ks.i * SM::stage + SM::k_off, v_lo = lo_of(smem_b + CFG::v_off + ks.i * SM::v_bytes, DV == 128 ? V_SLAB : 0),
                       t_lo = lo_of(smem_b + CFG::t_off + ks.i * SM::t_bytes);
        // (at d_v = 64 the 64 columns of V's tile are read twice: rows j past d_v are nobody's)
        // ---- V^T into the accumulator, as V^T times an identity, both bf16 (V as it came; the accumulator's last reader is done)
        if (!response) {
            if (!wait(CFG::LAND + ks.i, ks.phase)) return 327;
            tc_fence_after();
            if (elect_one()) {
                constexpr uint32_t idesc = make_idesc(NB, true, false, false) | (1u << 7) | (1u << 10);
#pragma unroll
                for (int c = 0; c < 4; ++c) mma_f16(T_R, desc_lo(v_lo + c * (2048 >> 4)), IdStrip::desc(smem_b + CFG::id_off, c), idesc, c > 0);
            }
            __syncwarp();
        }
        // ---- R = V^T - S K^T
        if (!wait(CFG::FULL + ks.i, ks.phase)) return 322;
        if (!wait(B_SP, b & 1)) return 323;
        tc_fence_after();
        if (elect_one()) {
            products_ta<false, NB, DK / 16, SM::rows>(T_R, T_S16, lo_of(k_at), !response);
            commit_at(bar + 8 * B_RD);
        }
        __syncwarp();
        // ---- U'^T = R T^T
        // (U' completes only after the last reader of the block before's, P U', so that the chain warps need not wait for that)
        if (b > 0 && !wait(B_OD + (b - 1) % OB, ((b - 1) / OB) & 1)) return 319;
        if (!wait(B_RP, b & 1)) return 326;
        tc_fence_after();
        if (elect_one()) {
            products_ta<false, NB, NB / 16, NB>(T_R, T_R16, t_lo, false);
            commit_at(bar + 8 * B_UD);
        }
        __syncwarp();
        // ---- S += U'^T K
        // (and S only after Q S^T)
        if (!wait(B_QD, b & 1)) return 320;
        if (!wait(B_UP, b & 1)) return 328;
        tc_fence_after();
        if (elect_one()) {
            products_ta<true, DK, NB / 16, SM::rows>(T_S, T_U16, lo_of(k_at, K_SLAB), true);
            commit_at(bar + 8 * B_SD);
            commit_at(bar + 8 * (CFG::EMPTY + ks.i));
        }
        __syncwarp();
        ks.next();
    }
    }
    return 0;
}

// The products of the output (one warp): O^T = S Q^T + U'^T P^T with the state before the update.
template <int DK, int R, int DV>
__device__ __forceinline__ void mma_out_role(int count, int width, int* err, uint8_t* smem, uint32_t bar) {
    using SM = ChainSmem<DK, R, DV>;
    using CFG = ChainCfg<DK, R, DV>;
    constexpr int CP = SM::CP, OB = O_BUFS<CP>;
    const uint32_t smem_b = smem_u32(smem);
    const int parties = width + 32;
    RingPos<CFG::NS> ks;
    RingPos<OB> os;
    Waits waits(bar);
#pragma unroll 1
    for (int b = 0; b < count; ++b) {
        const uint32_t sg = smem_b + ks.i * SM::stage, t_o = o_cols<CP>(os.i);
        waits.wait(CFG::FULL + ks.i, ks.phase, 351);
        if (b >= OB) waits.wait(B_OFREE + os.i, os.phase ^ 1, 325);
        waits.wait(B_RD, b & 1, 352);
        tc_fence_after();
        if (waits.ok() && elect_one()) {
            products_ta<false, CP, DK / 16, SM::rows, true>(t_o, T_S16, lo_of(sg + SM::q_off), false);
            commit_at(bar + 8 * B_QD);
        }
        __syncwarp();
        waits.wait(B_UP, b & 1, 354);
        tc_fence_after();
        if (waits.ok() && elect_one()) {
            products_ta<false, CP, NB / 16, CP>(t_o, T_U16, lo_of(sg + SM::p_off), true);
            commit_at(bar + 8 * (B_OD + os.i));
            commit_at(bar + 8 * (CFG::EMPTY + ks.i));
        }
        __syncwarp();
        waits.wait(B_OD + os.i, os.phase, 331);
        // (also when it has given up: the output's warps must have passed this barrier before it is arrived at again)
        if (!waits.ok() && b >= OB) mbar_wait_tries<true>(bar + 8 * (B_OFREE + os.i), os.phase ^ 1);
        pass_on(N_OD + os.i, parties);
        ks.next();
        os.next();
    }
    if (!waits.ok()) atomicCAS(err, 0, waits.code);
}

// O of each block from tensor memory to global memory: warp `warp` of four has rows j = 32 warp + lane, and one store of a warp is
// 128 contiguous bytes of a token's row (64 of a response's).
template <int DK, int R, int DV, int MODE>
__device__ __forceinline__ void out_role(const ChainGeo& g, ChainWork<MODE> work, uint32_t bar, int warp, int lane) {
    using SM = ChainSmem<DK, R, DV>;
    constexpr int C = SM::C, CP = SM::CP, OB = O_BUFS<CP>;
    const int j = 32 * warp + lane, parties = work[0].width + 32;
    RingPos<OB> os;
    const uint32_t lanes = (uint32_t)(32 * warp) << 16;
#pragma unroll 1
    for (int i = 0; i < work.size(); ++i) {
    const ChainPart& part = work[i];
    float* o = part.O + j;
    __half* oh = (__half*)part.O + j;
    const int nblk = part.nblk, b0 = part.b0;
    const bool response = part.response;
    uint32_t most = 0;                                            // (bits of the response's largest magnitude)
#pragma unroll 1
    for (int b = 0; b < nblk; ++b) {
        named_bar(N_OD + os.i, parties);
        tc_fence_after();
        const int Cv = min(C, g.L - (b0 + b) * C);
#pragma unroll 1
        for (int c = 0; c < CP; c += 16) {
            uint32_t x[16];
            tmem_ld16(o_cols<CP>(os.i) + lanes + c, x);
            tmem_ld_wait();
            if (c + 16 == CP) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(bar + 8 * (B_OFREE + os.i));
            }
            if (response) {
                if (MODE == SHARED)
#pragma unroll
                    for (int t = 0; t < 16; ++t) most = max(most, x[t] & 0x7fffffffu);
#pragma unroll
                for (int t = 0; t < 16; ++t)
                    if (c + t < Cv) oh[(c + t) * DK] = __float2half_rn(__uint_as_float(x[t]));
            } else {
#pragma unroll
                for (int t = 0; t < 16; ++t)
                    if (c + t < Cv) o[(c + t) * DV] = __uint_as_float(x[t]);
            }
        }
        o += C * DV;
        oh += C * DK;
        os.next();
    }
    if (MODE == SHARED && most >= HALF_INF && g.lost) g.lost[part.seq] = 1;
    }
}

template <int DK, int R, int DV, int MODE>
__global__ void __launch_bounds__(CHAIN_THREADS, 1)
chain_kernel(const __grid_constant__ ChainMaps maps, const __nv_bfloat16* __restrict__ beta, const float* __restrict__ S0,
             float* __restrict__ O, float* __restrict__ S_final, int* __restrict__ status, ChainGeo g, ChainSeg sg) {
    using CFG = ChainCfg<DK, R, DV>;
    using SM = ChainSmem<DK, R, DV>;
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t bar[CFG::count];
    __shared__ uint32_t tmem_base;
    __shared__ ChainArgs args;
    __shared__ uint32_t lost[MODE == SHARED ? MOST_PARTS : 1];
    __shared__ ChainPart parts[MODE == SHARED ? MOST_PARTS : 1];
    __shared__ int parts_n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t bar_b = smem_u32(bar);
    // (SHARED: all parts have one width, and only `width` of this one is used)
    const ChainPart part = MODE == SHARED ? walk_of<DK, SM::C, MODE>(g, sg, S0, O, S_final, 0, 0, false, 0, g.nblk) : own_walk<DK, SM::C, MODE>(g, sg, S0, O, S_final);
    const int lo = share_of_cta() * g.share, count = MODE == SHARED ? min(g.share, g.total - lo) : part.nblk;
    const int quarters = part.width / 32;                         // lane quarters that hold rows of the state
    if ((smem_u32(smem) & 1023u) != 0) {                          // (the swizzled layouts need a 1024-byte aligned base)
        wait_for_previous_kernel();
        if (tid == 0) atomicCAS(status, 0, 99);
        return;
    }
    if (tid == 32) args = {g, sg};
    if (tid == 0) {
        for (int x = 0; x < (MODE == SHARED ? MOST_PARTS : 1); ++x) lost[x] = 0;
        mbar_init(&bar[B_SP], 2 * quarters);
        mbar_init(&bar[B_UP], 2 * quarters);
        mbar_init(&bar[B_SD], 1);
        mbar_init(&bar[B_UD], 1);
        mbar_init(&bar[B_QD], 1);
        mbar_init(&bar[B_GD], 1);
        mbar_init(&bar[B_RD], 1);
        mbar_init(&bar[B_RP], 2 * quarters);
        for (int x = 0; x < 4; ++x) mbar_init(&bar[B_END + x], 2);
        for (int x = 0; x < 2; ++x) {
            mbar_init(&bar[B_OD + x], 1);
            mbar_init(&bar[B_OFREE + x], quarters);
        }
        for (int x = 0; x < CFG::NS; ++x) {
            mbar_init(&bar[CFG::LAND + x], 1);
            mbar_init(&bar[CFG::FULL + x], 32 * 8);
            mbar_init(&bar[CFG::EMPTY + x], 2);
        }
        mbar_fence_init();
        prefetch_tmap(&maps.q);
        prefetch_tmap(&maps.k);
        prefetch_tmap(&maps.v);
    }
    if (MODE == SHARED && tid == 64) {
        int n = 0;
#pragma unroll 1
        for (int x = lo; x < lo + count && n < MOST_PARTS; x += parts[n++].nblk) parts[n] = part_at<DK, SM::C>(g, sg, S0, O, S_final, x, lo, lo + count);
        parts_n = n;
    }
    if (warp == W_MMA) tmem_alloc(&tmem_base, 512);
    if (SM::CP > SM::C) {                                         // (r = 3: query rows that no copy writes are read)
        for (int e = tid; e < CFG::NS * SM::stage / 16; e += CHAIN_THREADS) ((uint4*)smem)[e] = make_uint4(0, 0, 0, 0);
    } else {                                                      // (the upper triangles of P and T, which nothing writes)
        for (int st = 0; st < CFG::NS && st < count; ++st)
            for (int e = tid; e < SM::p_bytes / 16; e += CHAIN_THREADS) ((uint4*)(smem + st * SM::stage + SM::p_off))[e] = make_uint4(0, 0, 0, 0);
    }
    // (r = 3: as many slots as there are blocks, 80.5 us instead of 81.8 at 48 sequences of 1999; elsewhere all, 20.9 instead of 21.1 at 16 of 333, r = 2)
    const int t_slots = SM::CP > SM::C ? min(CFG::NS, count) : CFG::NS;
    for (int e = tid; e < t_slots * SM::t_bytes / 16; e += CHAIN_THREADS) ((uint4*)(smem + CFG::t_off))[e] = make_uint4(0, 0, 0, 0);
    for (int e = tid; e < IdStrip::bytes / 2; e += CHAIN_THREADS) ((uint16_t*)(smem + CFG::id_off))[e] = IdStrip::one(e) ? 0x3F80 : 0;
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tmem_base != 0) {                                         // (whoever holds all columns holds them from column 0 on)
        wait_for_previous_kernel();
        if (tid == 0) atomicCAS(status, 0, 350);
        if (warp == W_MMA) tmem_dealloc(tmem_base, 512);
        return;
    }
    const ChainWork<MODE> work{part, parts, MODE == SHARED ? parts_n : 1, count};
    // (each warpgroup sets its registers once, and no code is shared after that: its end is in its own branch)
    // (each waits for the kernel before by itself: nothing is left to be set up for each other after that.  With the CTA's barrier after that wait
    //  and the end state after the last output, us: 16 sequences of 40, d = 128, r = 2: 8.7, now 7.8; 148 of 40, d = 64: 7.9, now 7.0)
    auto begin = [&]() {
        wait_for_previous_kernel();
        if (g.nseg == 1) let_next_kernel_start();  // (chain_compose's blocks would crowd on what few multiprocessors have room: 144 us instead of 140)
    };
    auto all_done = [&]() {
        __syncwarp();
        tc_fence_before();
        named_bar(0, CHAIN_THREADS);
        tc_fence_after();
    };
    // (the chain's and the solve teams' warps, eight rows each, us a token with every row lost and with the chain's warps alone: d = 128, r = 1, 2, 4
    //  0.97, 1.56, 3.7 and 2.4, 5.1, 9.2; d = 64, r = 1 .. 4 0.54, 0.81, 1.1, 1.2 and 1.1, 2.1, 3.0, 3.3.  Fetching the next token's inputs ahead: no gain)
    auto walk_lost = [&](int x) {
#pragma unroll 1
        for (int i = 0; i < work.size(); ++i) {
            if (!(lost[i] >> (x >> 2) & 1)) continue;
            ChainPart p = work[i];
            if (MODE == SHARED && p.hand_in >= 0) {               // all of the walk, when its first part's outputs, which are replaced here, are written
                if (lane == 0 && !wait_for_count(g.finished + p.hand_in + 1, 1)) atomicCAS(status, 0, 337);
                __syncwarp();
                p.b0 -= p.before;
                p.O -= (long long)p.before * SM::C * g.d_v;
                p.nblk = p.walk;
            }
            walk_fp32<DK, R>(args, p, p.seq, 8 * x);
        }
    };
    if (warp < W_OUT) {
        set_registers<REGS_CHAIN>();
        begin();
        if (tid == 0 && blockIdx.x == 0 && g.clear) *status = 0;  // (the call's status word: a wait expires a second from now at the earliest)
        const bool holds_state = (warp & 3) < quarters;
        if (holds_state) {
            const int code = chain_role<DK>(g, work, lost, bar_b, warp, lane);
            if (code) atomicCAS(status, 0, code);
        }
        all_done();                                               // (every output is written)
        if (MODE == SHARED && tid == 0) {
            __threadfence();
            st_release_gpu(g.finished + share_of_cta(), 1);
        }
        walk_lost(warp);
    } else if (warp < W_CONV) {
        set_registers<REGS_OUT>();
        begin();
        if (warp - W_OUT < quarters) out_role<DK, R, DV>(g, work, bar_b, warp - W_OUT, lane);
        all_done();
    } else if (warp < W_SOLVE) {
        set_registers<REGS_CONV>();
        begin();
        convert_role<DK, R, DV>(count, smem, bar_b, tid - 32 * W_CONV);
        all_done();
    } else if (warp < W_MMA) {
        set_registers<REGS_SOLVE>();
        begin();
        solve_role<DK, R, DV>(g, work, beta, smem, bar_b, (warp - W_SOLVE) >> 2, (tid - 32 * W_SOLVE) & 127);
        all_done();
        walk_lost(8 + warp - W_SOLVE);
    } else {
        set_registers<REGS_ISSUE>();
        begin();
        if (warp == W_MMA) {
            const int code = mma_role<DK, R, DV>(work, smem, bar_b);
            if (code) atomicCAS(status, 0, code);
        } else if (warp == W_MMA_OUT) {
            mma_out_role<DK, R, DV>(count, part.width, status, smem, bar_b);
        } else if (warp == W_GRAM) {
            gram_role<DK, R, DV>(count, status, smem, bar_b);
        } else if (warp == W_LOAD) {
            load_role<DK, R, DV>(maps, work, status, smem, bar_b);
        }
        all_done();
        if (warp == W_MMA) tmem_dealloc(0, 512);
    }
}

// Start states of the segments: one CTA per sequence and 16 rows j, serial over the segments; four warps with a quarter of the
// columns i each.  start(1) = Xi_0, start(s+1) = start(s) P_s + Xi_s; the last one is S_final.  The diagonal's part of the product is
// fp32, the rest has fp16 operands.  What bounds it is the latency of a step, so P, Xi and the diagonal come through a ring of up to
// three steps (4 sequences of 16384, r = 1, the call: 77.9 us; one step ahead, Xi and the diagonal in registers: 80.2).
constexpr int COMPOSE_RING = 3;
template <int DK>
struct ComposeSmem {
    static constexpr int LD = DK + 8, LX = 20;                    // (row pitches without bank conflicts)
    static constexpr int p_bytes = DK * LD * 2, x_bytes = DK * LX * 4, stage = p_bytes + x_bytes + DK * 4, a_bytes = 2 * 16 * LD * 2;
};
// LOST: lost[sequence]: chain_apply walks it again, from a start state that S_final may replace.
template <int DK, bool LOST>
__global__ void __launch_bounds__(128) chain_compose(ChainSeg sg, float* __restrict__ S_final, const int* lost, int nseg, int d_v) {
    using SM = ComposeSmem<DK>;
    constexpr int LD = SM::LD, LX = SM::LX, NT = DK / 32;
    extern __shared__ __align__(16) uint8_t smem_tail[];
    __half* sA = (__half*)smem_tail;                              // [2][16][LD]  fp16 rows of the start state
    uint8_t* ring = smem_tail + SM::a_bytes;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const int groups = d_v / 16, depth = min(COMPOSE_RING, nseg - 1);
    const long long seq = blockIdx.x / groups;
    const int j0 = (int)(blockIdx.x % groups) * 16, j = j0 + gq, i0 = w * (DK / 4) + 2 * t4;
    auto copy16 = [](void* dst, const void* src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
    };
    // what step s needs (an empty group past the last: the count of groups in flight is the same in every step)
    auto load = [&](int s, int slot) {
        if (s < nseg) {
            uint8_t* at = ring + slot * SM::stage;
            const __half* P = sg.P + (seq * nseg + s) * DK * DK;
#pragma unroll
            for (int e = 0; e < DK * DK / 8 / 128; ++e) {
                const int p = e * 128 + tid, row = p / (DK / 8), c = p % (DK / 8);
                copy16((__half*)at + row * LD + c * 8, P + row * DK + c * 8);
            }
            const float* Xi = sg.Xi + (seq * nseg + s) * DK * d_v + j0;
#pragma unroll
            for (int e = 0; e < DK * 4 / 128; ++e) {
                const int p = e * 128 + tid, row = p / 4, c = p % 4;
                copy16((float*)(at + SM::p_bytes) + row * LX + c * 4, Xi + (long long)row * d_v + c * 4);
            }
            if (tid < DK / 4) copy16((float*)(at + SM::p_bytes + SM::x_bytes) + tid * 4, sg.D + (seq * nseg + s) * DK + tid * 4);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float S[NT][4];
    wait_for_previous_kernel();
    if (LOST && lost[seq]) S_final = nullptr;                     // (not __restrict__: what may not change could be read ahead of the wait)
    for (int s = 1; s <= depth; ++s) load(s, s - 1);
    {
        const float* src = sg.Xi + seq * nseg * DK * d_v;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) S[n][e] = src[(long long)(i0 + 8 * n + (e & 1)) * d_v + j + 8 * (e >> 1)];
    }
    int slot = 0;
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
        if (depth == 3) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (depth == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const __half* P = (const __half*)(ring + slot * SM::stage);
        const float *X = (const float*)(ring + slot * SM::stage + SM::p_bytes), *D = X + SM::x_bytes / 4;
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
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const float2 d = *(const float2*)(D + i0 + 8 * n);
#pragma unroll
            for (int e = 0; e < 4; ++e) S[n][e] = fmaf(S[n][e], e & 1 ? d.y : d.x, X[(i0 + 8 * n + (e & 1)) * LX + gq + 8 * (e >> 1)]) + M[n][e];
        }
        __syncthreads();                                          // (the slot is filled anew)
        load(s + depth, slot);
        slot = slot + 1 == depth ? 0 : slot + 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
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
// LOST_R (a rank, or 0): with `args`, which says which sequences are walked again instead.
template <int DK, int DV, int LOST_R>
__device__ __forceinline__ void apply_tile(const ChainSeg& sg, float* __restrict__ O, int L, int first_tokens, int seg_tokens, int nseg, const ChainArgs* args) {
    constexpr int LD = DK + 8, KT = DK / 16;
    extern __shared__ __align__(16) uint8_t smem_tail[];
    __half* sS = (__half*)smem_tail;                                   // [DV][LD]
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, gq = lane >> 2, t4 = lane & 3;
    const long long seq = blockIdx.y / (nseg - 1);
    const int s = 1 + (int)(blockIdx.y % (nseg - 1));
    const int start = first_tokens + (s - 1) * seg_tokens, t_end = min(L, start + seg_tokens), t0 = start + blockIdx.x * 128 + w * 16 + gq;
    const __half* src = sg.start + (seq * nseg + s) * DV * DK;
    wait_for_previous_kernel();
    const int lost = LOST_R > 0 ? args->g.lost[seq] : 0;          // (looked at when everything else is on its way)
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
    if constexpr (LOST_R > 0)
        if (lost) {
            const ChainGeo& g = args->g;
            ChainPart part{};
            part.nblk = g.nblk;
            part.S0 = g.S0 ? g.S0 + seq * DK * DV : nullptr;
            part.O = O + seq * L * DV;
            part.S_end = g.S_final ? g.S_final + seq * DK * DV : nullptr;
            const int block = (s - 1) * gridDim.x + blockIdx.x, blocks = (nseg - 1) * gridDim.x;
#pragma unroll 1
            for (int row0 = 8 * (8 * block + w); row0 < DV; row0 += 64 * blocks) walk_fp32<DK, LOST_R>(*args, part, seq, row0);
            return;
        }
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

template <int DK, int DV>
__global__ void __launch_bounds__(256) chain_apply(ChainSeg sg, float* __restrict__ O, int L, int first_tokens, int seg_tokens, int nseg) {
    apply_tile<DK, DV, 0>(sg, O, L, first_tokens, seg_tokens, nseg, nullptr);
}
// For calls that the single launch would take if walks were not shared out.  Its flows are those of 64 tokens, here a response runs through thousands: where one
// has left fp16's range, the whole sequence is walked again in fp32, by the first of its blocks here.
template <int DK, int DV, int R>
__global__ void __launch_bounds__(256, 2) chain_apply_or_walk(const __grid_constant__ ChainArgs args, int first_tokens, int seg_tokens) {
    apply_tile<DK, DV, R>(args.seg, args.g.O, args.g.L, first_tokens, seg_tokens, args.g.nseg, &args);
}

// A sequence has one CTA, or where few sequences are long, segments walked side by side: as many as one wave of CTAs holds pay for
// the second walk (the responses) and for two more kernels.  The time is 7 us, (waves of CTAs) x (blocks of a segment) x (time of a
// block) and what composing segments costs.  Measured, us per block for r = 1 .. 4 with 32 CTAs (d_k = 64 and 128), and with 148, when
// two multiprocessors share what they fetch instructions through (taken before G and P^T were one product; since then a block takes up to 18 % less, but so far the
// choices come out right: with the present times 32 sequences of 16384, r = 2, would go from the single launch's 472 us to 522 in segments); and 8192 tokens of 4 sequences, d = 128, r = 1, in 1, 2, 4, 8, 16
// segments: 259, 136, 85, 60, 55 us; of 2, d = 64, r = 2, in 2, 4, 8, 16: 163, 88, 53, 40.
struct ChainPlan {
    int nseg, seg_blk;
    double us;
    int first_blk;            // blocks of the first segment
    int share, ctas;          // SHARED: blocks of a CTA (0: a walk each) and CTAs
    bool rewalk;              // sequences in which a response leaves fp16's range are walked again (chain_apply)
    double short_us;          // the kernel alone without segments, the start of each wave counted: what a call of a few blocks takes
};
struct ChainCarve {
    size_t R, P, D, Xi, start, flags, flag_bytes, hand, total;
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
    if (plan.share > 0) {
        c.flag_bytes = (size_t)plan.ctas * 8 + (plan.rewalk ? (size_t)p.B * p.H * 4 : 0);
        c.flags = take(c.flag_bytes);
        c.hand = take((size_t)plan.ctas * p.d_k * p.d_v * 4);
    }
    c.total = off;
    return c;
}

// Equal shares of all blocks (part_at) in place of a walk each, where that is faster: more sequences than multiprocessors, or, of a state as wide as its response,
// few in segments, the first of which is as long as a share (it has no response to walk) and the others as many as it takes.  Against it stand clearing the flags, a state
// through memory and the starts of further walks, 12 us and 1.5 a walk, a block that takes longer while all multiprocessors are busy to the end, and more responses.
// Measured, us, shared out and not, inputs that change from call to call, d = 128: 160 and 200 sequences of 1000, r = 2: 82 and 110, 100 and 112; 300 of 500, r = 4: 123
// and 156; 150 of 2000, r = 3, d_v = 64: 171 and 297; 32 of 8192, r = 2: 243, and 250 in the single launch; r = 3: 302 and 344; 32 of 4096, r = 4: 187 and 214; d = 64: 64 of
// 4096, r = 4: 208 and 276; 200 of 2000, r = 1: 79 and 92; 32 of 8192, r = 2: 153 and 176; 200 of 1000, 64 x 128, r = 1: 54 and 57.  Not taken, and measured when they were (same
// inputs): 256 of 1024, r = 2: 119 and 113; 32 of 8192, r = 1: 175 and 167.  The estimates below are within 10 % of these, but 15 % low at 32 of 8192, r = 2 (207), and 16 % high
// for 200 of 2000 without sharing (107); one wave's without sharing is 8 % below make_plan's, whose choices against the single launch are left as they are.  Not where segments would need more workspace than the library keeps
// from call to call: a caller who synchronises between calls would have it mapped anew at each (32 of 9600, r = 2, 96.3 MB: 2700 us, 298 in the single launch).
ChainPlan share_out(const Problem& p, const ChainPlan& plan, int nblk, double block_us) {
    const long long nseq = (long long)p.B * p.H, sms = sm_count();
    if (sms < 1 || nseq * nblk > 0x3fffffffLL || p.no_share) return plan;
    const double row_bytes = 4.0 * p.d_k + 8.0 * p.d_v, tail = p.d_k == 128 ? 4.0 : 2.0, per_seg = p.d_k == 128 ? 0.85 : 0.4;
    ChainPlan out = plan;
    double us = 12.0, rival = 7.0 + 0.92 * (plan.us - 7.0);
    if (nseq > sms) {
        out.nseg = 1;
        out.seg_blk = out.first_blk = nblk;
        block_us *= p.d_k == 128 ? 1.05 : 0.95;
    } else {
        if (p.d_k != p.d_v || nblk < 8) return plan;
        const long long first = 2 * nblk * nseq / (sms + nseq);
        if (first >= nblk || first < 1) return plan;
        out.nseg = 1 + (int)((nblk - first + first - 1) / first);
        if (out.nseg > 64) return plan;
        out.seg_blk = (int)((nblk - first + out.nseg - 2) / (out.nseg - 1));
        out.first_blk = nblk - (out.nseg - 1) * out.seg_blk;
        if (out.first_blk < 1) return plan;
        us += 3.0 + tail + per_seg * out.nseg + (double)nseq * p.L * (nblk - out.first_blk) / nblk * row_bytes / 6e6;
        if (p.d_k == 64) block_us *= 0.95;
        if (plan.nseg > 1) {      // (the composing kernels' part of the estimate does not shrink, their traffic goes at 6 TB/s)
            const double traffic = (double)nseq * p.L * (plan.nseg - 1) / plan.nseg * row_bytes, kernels = (p.d_k == 128 ? 11.0 : 9.0) + per_seg * plan.nseg;
            rival = kernels + traffic / 6e6 + 0.92 * (plan.us - kernels - traffic / 4e6);
        }
    }
    const long long total = nseq * (2 * nblk - out.first_blk);
    out.share = (int)((total + sms - 1) / sms);
    out.ctas = (int)((total + out.share - 1) / out.share);
    const int other = out.nseg > 1 ? out.seg_blk : out.first_blk, longest = out.first_blk > other ? out.first_blk : other, shortest = out.first_blk < other ? out.first_blk : other;
    if (longest > out.share || out.share / shortest + 2 > MOST_PARTS) return plan;
    out.rewalk = out.nseg > 1 && fused_supported(p) && fused_estimate_us(p) < plan.us;
    if (out.nseg > 1 && carve(p, out).total > WORKSPACE_KEEP) return plan;
    out.us = us + out.share * block_us + 1.5 * out.share / shortest;
    return out.us < 0.985 * rival ? out : plan;
}
ChainPlan make_plan(const Problem& p) {
    static const double alone[2][4] = {{1.40, 1.25, 1.25, 1.19}, {1.95, 1.53, 1.50, 1.55}};
    static const double crowded[2][4] = {{1.70, 1.34, 1.33, 1.24}, {2.30, 1.79, 1.68, 1.58}};
    const long long nseq = (long long)p.B * p.H, sms = sm_count();
    const int C = NB / p.r, nblk = (p.L + C - 1) / C;
    auto step = [&](long long ctas) {
        const double a = alone[p.d_k == 128][p.r - 1], c = crowded[p.d_k == 128][p.r - 1];
        const double crowd = sms > 0 ? 2.0 * ctas / sms - 1.0 : 0.0;
        return a + (c - a) * (crowd < 0.0 ? 0.0 : crowd > 1.0 ? 1.0 : crowd);
    };
    const double waves = (double)((nseq + sms - 1) / (sms > 0 ? sms : 1)), walk = nblk * step(nseq) * waves;
    ChainPlan plan{1, nblk, 7.0 + walk, nblk, 0, 0, false, 5.0 * waves + walk};
    const double limit = 0.92 * plan.us;
    // (calls of up to 512 tokens at d_k = 128 are one launch, which a test of two sequences of 512 expects, also where segments would be faster: 16 of
    //  333, r = 2: 21.7 us, 20.9 estimated in four)
    if (p.d_k == 128 && p.L <= 512) return nseq > sms ? share_out(p, plan, nblk, step(sms)) : plan;
    for (int want = 2; nseq * (2 * want - 1) <= sms && want <= 64 && want <= nblk; ++want) {
        const int seg_blk = (nblk + want - 1) / want, nseg = (nblk + seg_blk - 1) / seg_blk;
        // (two kernels, their share per segment, and the traffic of the responses and of O at about 4 TB/s)
        const double traffic = (double)nseq * p.L * (nseg - 1) / nseg * (4.0 * p.d_k + 8.0 * p.d_v) / 4e6;
        const double us = (p.d_k == 128 ? 11.0 + 0.85 * nseg : 9.0 + 0.4 * nseg) + traffic + seg_blk * step(nseq * (2 * nseg - 1));
        if (us < limit && us < plan.us) plan = {nseg, seg_blk, us, seg_blk, 0, 0, false, plan.short_us};
    }
    return share_out(p, plan, nblk, step(sms));
}

ChainGeo make_geo(const Problem& p, const ChainPlan& plan, const ChainCarve& c, void* workspace) {
    ChainGeo g{};
    g.L = p.L;
    g.d_v = p.d_v;
    g.nblk = (p.L + NB / p.r - 1) / (NB / p.r);
    g.nseg = plan.nseg;
    g.seg_blk = plan.seg_blk;
    g.first_blk = plan.first_blk;
    if (plan.share > 0) {
        g.share = plan.share;
        g.total = (int)((long long)p.B * p.H * (2 * g.nblk - g.first_blk));
        g.hand = (float*)((uint8_t*)workspace + c.hand);
        g.handed = (int*)((uint8_t*)workspace + c.flags);
        g.finished = g.handed + plan.ctas;
        if (plan.rewalk) g.lost = g.finished + plan.ctas;
    }
    g.rm = p.mask_group();
    g.exact = p.exact ? 1 : 0;
    g.clear = p.clear_status ? 1 : 0;
    g.q = (const __nv_bfloat16*)p.q;
    g.k = (const __nv_bfloat16*)p.k;
    g.v = (const __nv_bfloat16*)p.v;
    g.beta = (const __nv_bfloat16*)p.beta;
    g.S0 = p.S0;
    g.O = p.O;
    g.S_final = p.S_final;
    return g;
}

template <int DK, int R, int DV, int MODE>
int launch(const Problem& p, const ChainPlan& plan, const ChainGeo& g, const ChainSeg& sg) {
    using CFG = ChainCfg<DK, R, DV>;
    static_assert(CFG::total + (MODE == SHARED ? 4096 : 1024) <= 227 * 1024 && CFG::NS >= 3, "shared memory budget");
    const void* fn = (const void*)chain_kernel<DK, R, DV, MODE>;
    constexpr int C = NB / R;
    const long long nseq = (long long)p.B * p.H, grid = MODE == SHARED ? plan.ctas : nseq * (2 * plan.nseg - 1);
    ChainMaps maps;
    if (!make_slab_map(&maps.k, p.k, nseq, (uint64_t)p.L * R, DK, 64, NB, 1) ||
        !make_slab_map(&maps.q, p.q, nseq, p.L, DK, 64, C, 1) ||
        !make_slab_map(&maps.v, p.v, nseq, (uint64_t)p.L * R, DV, 64, NB, DV / 64))
        return record_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    static std::atomic<uint64_t> opted_in{0};
    const int st = allow_smem(opted_in, fn, CFG::total);
    if (st != PF_OK) return st;
    void* args[] = {(void*)&maps, (void*)&p.beta, (void*)&p.S0, (void*)&p.O, (void*)&p.S_final, (void*)&p.status, (void*)&g, (void*)&sg};
    prof_begin("chain", p.stream);
    PF_CUDA_TRY(launch_early(fn, dim3((unsigned)grid), CHAIN_THREADS, args, (size_t)CFG::total, p.stream));
    prof_end(p.stream);
    count_launch(1);
    return PF_OK;
}

template <int DK, int R>
int launch_plan(const Problem& p, const ChainPlan& plan, const ChainGeo& g, const ChainSeg& sg) {
    if (plan.share > 0) return p.d_v == 128 ? launch<DK, R, 128, SHARED>(p, plan, g, sg) : launch<DK, R, 64, SHARED>(p, plan, g, sg);
    if (plan.nseg > 1) return p.d_v == 128 ? launch<DK, R, 128, SEGMENTS>(p, plan, g, sg) : launch<DK, R, 64, SEGMENTS>(p, plan, g, sg);
    return p.d_v == 128 ? launch<DK, R, 128, WHOLE>(p, plan, g, sg) : launch<DK, R, 64, WHOLE>(p, plan, g, sg);
}
template <int DK>
int launch_rank(const Problem& p, const ChainPlan& plan, const ChainGeo& g, const ChainSeg& sg) {
    switch (p.r) {
        case 1: return launch_plan<DK, 1>(p, plan, g, sg);
        case 2: return launch_plan<DK, 2>(p, plan, g, sg);
        case 3: return launch_plan<DK, 3>(p, plan, g, sg);
        default: return launch_plan<DK, 4>(p, plan, g, sg);
    }
}

template <int DK, int DV, int LOST_R = 0>
int launch_seg_tail(const Problem& p, const ChainPlan& plan, const ChainGeo& g, const ChainSeg& sg) {
    const int nseq = p.B * p.H, dv = DV, seg_tokens = plan.seg_blk * (NB / p.r), first_tokens = plan.first_blk * (NB / p.r);
    constexpr int LD = DK + 8;
    {
        using SM = ComposeSmem<DK>;
        const int smem = SM::a_bytes + (plan.nseg - 1 < COMPOSE_RING ? plan.nseg - 1 : COMPOSE_RING) * SM::stage;
        static std::atomic<uint64_t> opted_in{0};
        const void* fn = (const void*)chain_compose<DK, (LOST_R > 0)>;
        const int st = allow_smem(opted_in, fn, SM::a_bytes + COMPOSE_RING * SM::stage);
        if (st != PF_OK) return st;
        prof_begin("chain_compose", p.stream);
        void* args[] = {(void*)&sg, (void*)&p.S_final, (void*)&g.lost, (void*)&plan.nseg, (void*)&dv};
        PF_CUDA_TRY(launch_early(fn, dim3((unsigned)(nseq * (DV / 16))), 128, args, smem, p.stream));
        prof_end(p.stream);
    }
    constexpr int smem = DV * LD * 2;
    prof_begin("chain_apply", p.stream);
    const void* fn;
    void *args[6] = {(void*)&sg, (void*)&p.O, (void*)&p.L, (void*)&first_tokens, (void*)&seg_tokens, (void*)&plan.nseg}, *walk_args[3] = {nullptr, (void*)&first_tokens, (void*)&seg_tokens};
    const ChainArgs walk{g, sg};
    if constexpr (LOST_R > 0) {
        fn = (const void*)chain_apply_or_walk<DK, DV, LOST_R>;
        walk_args[0] = (void*)&walk;
    } else {
        fn = (const void*)chain_apply<DK, DV>;
    }
    PF_CUDA_TRY(launch_early(fn, dim3((unsigned)((seg_tokens + 127) / 128), (unsigned)(nseq * (plan.nseg - 1))), 256, LOST_R > 0 ? walk_args : args, smem, p.stream));
    prof_end(p.stream);
    count_launch(2);
    return PF_OK;
}

}  // namespace

double chain_estimate_us(const Problem& p) { return make_plan(p).us; }
double chain_short_us(const Problem& p) { return make_plan(p).short_us; }

size_t chain_workspace_bytes(const Problem& p) { return carve(p, make_plan(p)).total; }
bool chain_shares(const Problem& p) { return make_plan(p).share > 0; }
bool chain_needs_workspace(const Problem& p) {
    const ChainPlan plan = make_plan(p);
    return plan.nseg > 1 || plan.share > 0;
}

bool chain_supported(const Problem& p) {
    return p.in_dtype == PF_DTYPE_BF16 && p.L >= 1 && (long long)p.B * p.H * (p.d_v / 32) <= 0x7fffffffLL &&
           (long long)p.L * p.r <= 0x7fffffffLL;
}

int chain_forward(const Problem& p, void* workspace) {
    const ChainPlan plan = make_plan(p);
    const ChainCarve c = carve(p, plan);
    const ChainGeo g = make_geo(p, plan, c, workspace);
    ChainSeg sg{};
    if (plan.nseg > 1) {
        uint8_t* ws = (uint8_t*)workspace;
        sg = {(__half*)(ws + c.R), (__half*)(ws + c.P), (float*)(ws + c.D), (float*)(ws + c.Xi), (__half*)(ws + c.start)};
    }
    if (plan.share > 0) PF_CUDA_TRY(cudaMemsetAsync(g.handed, 0, c.flag_bytes, p.stream));
    const int st = p.d_k == 128 ? launch_rank<128>(p, plan, g, sg) : launch_rank<64>(p, plan, g, sg);
    if (st != PF_OK || plan.nseg == 1) return st;
    if (g.lost)                                                   // (the single launch's shapes)
        switch (p.r) {
            case 1: return launch_seg_tail<128, 128, 1>(p, plan, g, sg);
            case 2: return launch_seg_tail<128, 128, 2>(p, plan, g, sg);
            case 3: return launch_seg_tail<128, 128, 3>(p, plan, g, sg);
            default: return launch_seg_tail<128, 128, 4>(p, plan, g, sg);
        }
    if (p.d_k == 128) return p.d_v == 128 ? launch_seg_tail<128, 128>(p, plan, g, sg) : launch_seg_tail<128, 64>(p, plan, g, sg);
    return p.d_v == 128 ? launch_seg_tail<64, 128>(p, plan, g, sg) : launch_seg_tail<64, 64>(p, plan, g, sg);
}

}  // namespace pf
