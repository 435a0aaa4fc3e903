// recur: the recurrence itself, token by token, in fp32 with the state in registers (Section 1.1 readout, Section 1.3 /
// 3.1 update), for the calls whose time the chunk form cannot improve: every fp32 call, and bf16 calls of a few tokens.
//
// Per token the recurrence needs (4 r + 2) d_k d_v operations, less than half of what the chunk form needs on FFMA (no
// Gram product, no inverse, no W / Uh), and no intermediate ever leaves the SM: q, k, v, beta are read once per 32 columns
// of the state, O is written once.  What bounds it is the serial chain of one token (dot products, two shuffle stages, the
// update): 204 cycles at d_k = 64, r = 1 and 373 at d_k = 128, r = 2, of which the FFMA pipe is busy for 160.
// Measured (fp32): B*H = 32, L = 2048, d = 128, r = 2: 0.389 ms against 4.9 ms for the four chunk-form kernels in
// pf_simt.cu; one head, L = 256, d = 64, r = 1: 29 us walked as a whole, 19 in segments, against 209.
//
// A CTA takes one sequence and 32 columns j of the state S[j][i] (API layout X[i][j]); each of its four computing warps 8
// columns, without any exchange between warps.  Lane (ig, j) of a warp holds S[j][i] for a quarter of the rows i, so a dot
// product S k is finished by two shuffle stages; splitting a column over 8 or 16 lanes saves shared-memory loads but each
// further stage costs about 45 cycles of latency per token (measured: 0.56 and 0.57 ms instead of 0.40 at the first size
// above).  Taking several tokens per step (their dot products together, the coupling k_m . k_m' solved in registers)
// measured no faster: it is the number of instructions, not the shuffle latency, that such a step adds to.  Readouts S q are
// needed once per token and are not on the chain; four tokens of them are reduced together.
//
// A fifth warp keeps a ring of stages of up to 16 tokens filled with bulk copies; with the four computing warps loading
// for themselves the same kernel took 0.50 ms (issuing the copies cost them about 1200 cycles per stage).
//
// The factors of a group act on the same previous state (sum form: a group is a token's r factors; product form: every
// factor is a group of its own; GPT groups of RG factors make a token).
#include "pf_common.cuh"
#include "pf_tc_prims.cuh"

namespace pf {
namespace {

constexpr int RJ = 32;               // columns of S per CTA
constexpr int R_STAGES = 3;

// (a predicated store, not a branch: a branch would keep the compiler from moving anything across it)
__device__ __forceinline__ void store_if(float* p, float x, bool pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.f32 [%0], %1;\n\t}" ::"l"(p), "f"(x), "r"((unsigned)pred));
}

struct RecurGeo {
    int L, d_v;
    int ts;             // tokens per stage
    int clear;          // set the status word to 0
    int exact;          // PF_STEP_EXACT
    int nseg, seg_tok;  // segments per sequence (1: none) and tokens per segment (a multiple of ts)
};

// Segments (Section 3, "Scan"; Proposition 2.1: S_end = S_start P + Xi): few long sequences are cut into segments that are walked
// side by side, each from zero (S0 for the first), which gives its own part of O and Xi, and, but for the first, from the
// identity with v = 0, which gives P and the tokens' responses R_t = P_t q_t to the start state.  recur_compose then makes the
// start states, recur_apply adds start R_t to O.  All fp32.
struct RecurSeg {
    float* R;           // [nseq][L][d_k]
    float* P;           // [nseq][nseg][d_k i][d_k j]
    float* Xi;          // [nseq][nseg][d_k i][d_v j]
    float* start;       // [nseq][nseg][d_k i][d_v j]
};

// Two fp32 values in a register pair: one fma.rn.f32x2 does two FFMA's work in one issue slot.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pk2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 up2(f2 x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// four consecutive elements as two pairs
__device__ __forceinline__ void lds4(f2& x, f2& y, const float* p) {
    const ulonglong2 w = *(const ulonglong2*)p;
    x = w.x;
    y = w.y;
}
__device__ __forceinline__ void lds4(f2& x, f2& y, const __nv_bfloat16* p) {
    const uint2 w = *(const uint2*)p;
    x = pk2(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u));
    y = pk2(__uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }

// bytes of one stage of ts tokens: k rows, q rows, the CTA's columns of v, fp32 step sizes (padded to 16 bytes)
__host__ __device__ constexpr int recur_stage_bytes(int ts, int r, int d_k, int esize) {
    return ts * (r * d_k + d_k + r * RJ) * esize + (ts * r * 4 + 15) / 16 * 16;
}

// TB tokens per pass of the inner loop: 4, or 1 for calls of fewer than four tokens.  Tokens past the end of a pass are zero
// in shared memory, so that the pass has no branches and the compiler can put the loads, readouts and reductions of one
// token under the latency of another.
template <class Tin, int DK, int RG, int GPT, int TB, int IG>
__global__ void __launch_bounds__((IG + 1) * 32, 1)
recur_kernel(const Tin* __restrict__ q, const Tin* __restrict__ k, const Tin* __restrict__ v, const Tin* __restrict__ beta,
             const float* __restrict__ S0, float* __restrict__ O, float* __restrict__ S_final, int* __restrict__ status, RecurGeo g, RecurSeg sg) {
    constexpr int NI = DK / IG, r = RG * GPT;          // rows i of a column that a lane holds
    constexpr int JW = 32 / IG;                        // columns per warp (IG warps make up the CTA's 32 columns)
    constexpr bool AHEAD = RG * NI <= 64;              // keys are read one group ahead where registers allow it
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar_full[R_STAGES], bar_empty[R_STAGES];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the part this CTA walks: a sequence, or a segment of it, or a segment's response
    long long seq;
    int j0, tok0 = 0, Lp = g.L, width = g.d_v;
    bool response = false;
    const float* S_in = S0;
    float* S_out = S_final;
    float* O_out;
    {
        const int slices = g.d_v / RJ, x = (int)blockIdx.x;
        if (g.nseg == 1) {
            seq = x / slices;
            j0 = x % slices * RJ;
            O_out = O + seq * g.L * width;
            S_in = S0 ? S0 + seq * DK * width : nullptr;
            S_out = S_final ? S_final + seq * DK * width : nullptr;
        } else {
            constexpr int rs = DK / RJ;
            const int per_seq = g.nseg * slices + (g.nseg - 1) * rs, y = x % per_seq, z = y - g.nseg * slices;
            seq = x / per_seq;
            response = z >= 0;
            const int s = response ? 1 + z / rs : y / slices;
            j0 = (response ? z % rs : y % slices) * RJ;
            tok0 = s * g.seg_tok;
            Lp = min(g.seg_tok, g.L - tok0);
            width = response ? DK : g.d_v;
            O_out = (response ? sg.R : O) + (seq * g.L + tok0) * width;
            S_in = s == 0 && S0 ? S0 + seq * DK * width : nullptr;
            S_out = (response ? sg.P : sg.Xi) + (seq * g.nseg + s) * DK * width;
        }
    }
    const int L = Lp, d_v = g.d_v;
    const long long seq_tok = seq * g.L + tok0;        // first token of the part
    const int rows_s = g.ts * r;                       // rows per stage (at most 64)
    const int nb = (L + g.ts - 1) / g.ts;
    const int stage_bytes = recur_stage_bytes(g.ts, r, DK, (int)sizeof(Tin));
    auto s_k = [&](int st) { return (Tin*)(smem + st * stage_bytes); };
    auto s_q = [&](int st) { return s_k(st) + rows_s * DK; };
    auto s_v = [&](int st) { return s_q(st) + g.ts * DK; };
    auto s_b = [&](int st) { return (float*)(s_v(st) + rows_s * RJ); };

    if (tid == 0) {
        for (int x = 0; x < R_STAGES; ++x) {
            tc::mbar_init(&bar_full[x], 1);
            tc::mbar_init(&bar_empty[x], IG);
        }
        tc::mbar_fence_init();
    }
    wait_for_previous_kernel();
    if (g.nseg == 1) let_next_kernel_start();      // (recur_compose's blocks would crowd on what few multiprocessors have room: 75 us instead of 70)
    if (tid == 0 && blockIdx.x == 0 && g.clear) *status = 0;      // (the call's status word; a wait of this kernel expires a second later at the earliest)
    __syncthreads();

    if (warp == IG) {
        // ---- loader: bulk copies of the stages (k and q of a stage are contiguous, v is one copy per row), step sizes, and
        //      zeros for the tokens that the last pass has beyond the sequence
        for (int b = 0; b < nb; ++b) {
            const int st = b % R_STAGES, t0 = b * g.ts;
            const int nt = min(g.ts, L - t0), np = (nt + TB - 1) / TB * TB;
            if (b >= R_STAGES && !tc::mbar_wait_clk(&bar_empty[st], (uint32_t)(b / R_STAGES - 1) & 1, status, 301)) return;
            const long long tok = seq_tok + t0;
            if (lane == 0) {
                tc::mbar_expect_tx_only(&bar_full[st], (uint32_t)(nt * (r * DK + DK + (response ? 0 : r * RJ)) * sizeof(Tin)));
                tc::bulk_load(s_k(st), k + tok * r * DK, (uint32_t)(nt * r * DK * sizeof(Tin)), &bar_full[st]);
                tc::bulk_load(s_q(st), q + tok * DK, (uint32_t)(nt * DK * sizeof(Tin)), &bar_full[st]);
            }
            __syncwarp();
            if (response)
                for (int e = lane; e < nt * r * RJ; e += 32) s_v(st)[e] = Tin(0.f);
            else
                for (int row = lane; row < nt * r; row += 32)
                    tc::bulk_load(s_v(st) + row * RJ, v + (tok * r + row) * d_v + j0, (uint32_t)(RJ * sizeof(Tin)), &bar_full[st]);
            for (int row = lane; row < np * r; row += 32) s_b(st)[row] = row < nt * r ? to_f(beta[tok * r + row]) : 0.f;
            if (g.exact)                               // beta' = (1 - e^{-beta |k|^2}) / |k|^2
                for (int row = 0; row < nt * r; ++row) {
                    float s = 0.f;
                    for (int i = lane; i < DK; i += 32) {
                        const float x = to_f(k[(tok * r + row) * DK + i]);
                        s = fmaf(x, x, s);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
                    if (lane == (row & 31) && s > 0.f) s_b(st)[row] = -expm1f(-s_b(st)[row] * s) / s;
                }
            if (np > nt) {
                for (int e = nt * r * DK + lane; e < np * r * DK; e += 32) s_k(st)[e] = Tin(0.f);
                for (int e = nt * DK + lane; e < np * DK; e += 32) s_q(st)[e] = Tin(0.f);
                for (int e = nt * r * RJ + lane; e < np * r * RJ; e += 32) s_v(st)[e] = Tin(0.f);
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_full[st]);
        }
        return;
    }

    const int ig = lane / JW, jw = JW * warp + lane % JW;     // this lane's column within the CTA's 32
    // S[n] = rows i = 4 IG (n / 2) + 4 ig + 2 (n % 2), + 1 of the lane's column: neighbouring lanes read the same 16 bytes of a key
    f2 S[NI / 2];
    const long long sb = 4ll * ig * width + j0 + jw;
#pragma unroll
    for (int n = 0; n < NI; n += 2) {
        const int i = 4 * IG * (n >> 2) + (n & 3);
        const float* x = S_in + sb + (long long)i * width;
        S[n / 2] = S_in ? pk2(x[0], x[width]) : response ? pk2(i + 4 * ig == j0 + jw ? 1.f : 0.f, i + 4 * ig + 1 == j0 + jw ? 1.f : 0.f) : 0ull;
    }

    for (int b = 0; b < nb; ++b) {
        const int st = b % R_STAGES;
        const int nt = min(g.ts, L - b * g.ts);
        if (!tc::mbar_wait_clk(&bar_full[st], (uint32_t)(b / R_STAGES) & 1, status, 302)) return;
        // pointers to what is read next (one group past the stage's last at the end, inside the CTA's memory and unused)
        const Tin* kp = s_k(st) + 4 * ig;
        const Tin* qp = s_q(st) + 4 * ig;
        const Tin* vp = s_v(st) + jw;
        const float* bp = s_b(st);
        float* og = O_out + (long long)b * g.ts * width + j0 + jw;
        f2 kn[RG][NI / 2];
        float vn[RG], bn[RG];
        auto fetch_k = [&]() {
#pragma unroll
            for (int f = 0; f < RG; ++f)
#pragma unroll
                for (int c = 0; c < NI / 4; ++c) lds4(kn[f][2 * c], kn[f][2 * c + 1], kp + f * DK + 4 * IG * c);
            kp += RG * DK;
        };
        auto fetch_vb = [&]() {
#pragma unroll
            for (int f = 0; f < RG; ++f) {
                vn[f] = to_f(vp[f * RJ]);
                bn[f] = bp[f];
            }
            vp += RG * RJ;
            bp += RG;
        };
        if (AHEAD) fetch_k();
        fetch_vb();
#pragma unroll 1
        for (int t4 = 0; t4 < nt; t4 += TB) {
            float o[TB];                               // readouts, partial over the lanes of a column
#pragma unroll
            for (int tt = 0; tt < TB; ++tt) {
#pragma unroll
                for (int gi = 0; gi < GPT; ++gi) {
                    f2 kk[RG][NI / 2], uu[RG];
                    float d[RG], u[RG], ub[RG];
                    if (!AHEAD) fetch_k();
#pragma unroll
                    for (int f = 0; f < RG; ++f) {
                        f2 a0 = 0ull, a1 = 0ull;
#pragma unroll
                        for (int n = 0; n < NI / 2; n += 2) {
                            kk[f][n] = kn[f][n];
                            kk[f][n + 1] = kn[f][n + 1];
                            a0 = fma2(kk[f][n], S[n], a0);
                            a1 = fma2(kk[f][n + 1], S[n + 1], a1);
                        }
                        const float2 s2 = up2(add2(a0, a1));
                        d[f] = s2.x + s2.y;
                        u[f] = vn[f];
                        ub[f] = bn[f];
                    }
#pragma unroll
                    for (int m = JW; m < 32; m *= 2)
#pragma unroll
                        for (int f = 0; f < RG; ++f) d[f] += __shfl_xor_sync(FULL, d[f], m);
                    // (shuffles and shared-memory loads are served in order by one queue: the next group's loads go behind)
                    asm volatile("" ::: "memory");
                    if (AHEAD) fetch_k();
                    fetch_vb();
#pragma unroll
                    for (int f = 0; f < RG; ++f) {
                        u[f] = ub[f] * (u[f] - d[f]);
                        uu[f] = pk2(u[f], u[f]);
                    }
#pragma unroll
                    for (int n = 0; n < NI / 2; ++n)
#pragma unroll
                        for (int f = 0; f < RG; ++f) S[n] = fma2(uu[f], kk[f][n], S[n]);
                }
                f2 a0 = 0ull, a1 = 0ull;
#pragma unroll
                for (int c = 0; c < NI / 4; ++c) {
                    f2 x, y;
                    lds4(x, y, qp + 4 * IG * c);
                    a0 = fma2(x, S[2 * c], a0);
                    a1 = fma2(y, S[2 * c + 1], a1);
                }
                qp += DK;
                const float2 s2 = up2(add2(a0, a1));
                o[tt] = s2.x + s2.y;
            }
            // four tokens over the lanes of a column (lane bits 4 and 3 select the token), or one
            float y = o[0];
            if (TB == 4) {
                const bool b16 = lane & 16, b8 = lane & 8;
                const float s0 = b16 ? o[0] : o[2 % TB], s1 = b16 ? o[1 % TB] : o[3 % TB];
                const float x0 = (b16 ? o[2 % TB] : o[0]) + __shfl_xor_sync(FULL, s0, 16);
                const float x1 = (b16 ? o[3 % TB] : o[1 % TB]) + __shfl_xor_sync(FULL, s1, 16);
                y = (b8 ? x1 : x0) + __shfl_xor_sync(FULL, b8 ? x0 : x1, 8);
            }
#pragma unroll
            for (int m = JW; m < (TB == 4 ? 8 : 32); m *= 2) y += __shfl_xor_sync(FULL, y, m);
            const int tok = TB == 4 ? t4 + (lane >> 3) : t4;
            store_if(og + (long long)tok * width, y, tok < nt && (TB == 4 ? (lane & 7) < JW : lane < JW));
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_empty[st]);
    }
    if (S_out)
#pragma unroll
        for (int n = 0; n < NI; n += 2) {
            float* x = S_out + sb + (long long)(4 * IG * (n >> 2) + (n & 3)) * width;
            const float2 s2 = up2(S[n / 2]);
            x[0] = s2.x;
            x[width] = s2.y;
        }
}

// start(1) = Xi_0, start(s+1) = start(s) P_s + Xi_s, the last one is S_final: a CTA per sequence and ROWS rows j, serial over the
// segments.  A thread has four rows and one column i; P (stored [i][j']) comes to shared memory a step after it was requested,
// rows padded so that 32 threads reading 16 bytes of 32 rows meet no bank twice.  What bounds a step is shared memory: of a CTA's warps
// each reads its 32 rows of P once for 4 rows j.  So a CTA has 4 rows j, DK / 32 warps (the call, us, before with eight warps: one sequence of 256, d = 64,
// r = 1: 24.1 -> 18.8; of 2000: 48.4 -> 35.7; 16 of 1000, r = 2: 62.4 -> 60.8; one of 1000, d = 128, r = 2: 63.4 -> 59.3).  At d = 128, where P is
// four times as large and every CTA fetches its own copy, only while there is an SM for each (4 of 2000, r = 1: 86.7 -> 84.7; 8 of 1000 on 256 CTAs:
// 92.8 -> 94.1), and otherwise 8 rows, eight warps.
template <int DK, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) recur_compose(RecurSeg sg, float* __restrict__ S_final, int nseg, int d_v) {
    constexpr int CG = DK / 32, THREADS = 32 * WARPS, ROWS = 4 * (WARPS / CG), LD = DK + 4, NV = DK * DK / 4 / THREADS;
    extern __shared__ __align__(16) float smf[];
    float* Ps = smf;                    // [DK i][LD]
    float* cur = smf + DK * LD;         // [ROWS][DK]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int groups = d_v / ROWS, jl = 4 * (warp / CG), i = 32 * (warp % CG) + lane;
    const long long seq = blockIdx.x / groups;
    const int j = (int)(blockIdx.x % groups) * ROWS + jl;
    float4 pv[NV], xv;
    auto fetch_p = [&](int s) {
        const float4* p = (const float4*)(sg.P + (seq * nseg + s) * DK * DK);
#pragma unroll
        for (int u = 0; u < NV; ++u) pv[u] = p[u * THREADS + tid];
    };
    auto fetch_x = [&](int s) { return *(const float4*)(sg.Xi + ((seq * nseg + s) * DK + i) * d_v + j); };
    wait_for_previous_kernel();
    float4 acc = fetch_x(0);
    fetch_p(1);
    xv = fetch_x(1);
    for (int s = 1; s < nseg; ++s) {
        *(float4*)(sg.start + ((seq * nseg + s) * DK + i) * d_v + j) = acc;
        cur[(jl + 0) * DK + i] = acc.x;
        cur[(jl + 1) * DK + i] = acc.y;
        cur[(jl + 2) * DK + i] = acc.z;
        cur[(jl + 3) * DK + i] = acc.w;
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int e = (u * THREADS + tid) * 4;
            *(float4*)(Ps + (e / DK) * LD + e % DK) = pv[u];
        }
        acc = xv;
        __syncthreads();
        if (s + 1 < nseg) {
            fetch_p(s + 1);
            xv = fetch_x(s + 1);
        }
#pragma unroll 4
        for (int ip = 0; ip < DK; ip += 4) {
            const float4 p = *(const float4*)(Ps + i * LD + ip);
            const float4 a = *(const float4*)(cur + (jl + 0) * DK + ip), b = *(const float4*)(cur + (jl + 1) * DK + ip);
            const float4 c = *(const float4*)(cur + (jl + 2) * DK + ip), d = *(const float4*)(cur + (jl + 3) * DK + ip);
            acc.x = fmaf(a.x, p.x, fmaf(a.y, p.y, fmaf(a.z, p.z, fmaf(a.w, p.w, acc.x))));
            acc.y = fmaf(b.x, p.x, fmaf(b.y, p.y, fmaf(b.z, p.z, fmaf(b.w, p.w, acc.y))));
            acc.z = fmaf(c.x, p.x, fmaf(c.y, p.y, fmaf(c.z, p.z, fmaf(c.w, p.w, acc.z))));
            acc.w = fmaf(d.x, p.x, fmaf(d.y, p.y, fmaf(d.z, p.z, fmaf(d.w, p.w, acc.w))));
        }
        __syncthreads();
    }
    if (S_final) *(float4*)(S_final + (seq * DK + i) * d_v + j) = acc;
}

// O[t][j] += sum_i R[t][i] start[i][j] for the tokens of all segments but the first: grid (64-token tiles, nseq (nseg - 1)), thread
// (ty, tx) the tokens 4 ty .. 4 ty + 3 and the columns DV / 16 tx ...
template <int DK, int DV>
__global__ void __launch_bounds__(256) recur_apply(RecurSeg sg, float* __restrict__ O, int L, int seg_tok, int nseg) {
    constexpr int PER = DV / 16, TLD = 68;
    extern __shared__ __align__(16) float smf[];
    float* Ss = smf;                    // [DK i][DV j]
    float* Rs = smf + DK * DV;          // [DK i][TLD]  R transposed: the four tokens of a thread are one 16-byte load
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const long long seq = blockIdx.y / (nseg - 1);
    const int s = 1 + (int)(blockIdx.y % (nseg - 1)), t0 = s * seg_tok + blockIdx.x * 64;
    const int nt = min(64, min(L, (s + 1) * seg_tok) - t0);
    wait_for_previous_kernel();
    let_next_kernel_start();
    if (nt <= 0) return;
    const float4* st = (const float4*)(sg.start + (seq * nseg + s) * DK * DV);
#pragma unroll
    for (int e = 0; e < DK * DV / 4 / 256; ++e) ((float4*)Ss)[e * 256 + tid] = st[e * 256 + tid];
    const float* Rg = sg.R + (seq * L + t0) * DK;
    for (int e = tid; e < 64 * DK; e += 256) {
        const int t = e / DK, i = e % DK;
        Rs[i * TLD + t] = t < nt ? Rg[e] : 0.f;
    }
    float acc[4][PER];
    float* Og = O + (seq * L + t0 + 4 * ty) * DV + PER * tx;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < PER; c += 4) {
            const float4 o = 4 * ty + a < nt ? *(const float4*)(Og + a * DV + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[a][c] = o.x; acc[a][c + 1] = o.y; acc[a][c + 2] = o.z; acc[a][c + 3] = o.w;
        }
    __syncthreads();
#pragma unroll 4
    for (int i = 0; i < DK; ++i) {
        const float4 rv = *(const float4*)(Rs + i * TLD + 4 * ty);
#pragma unroll
        for (int c = 0; c < PER; c += 4) {
            const float4 b = *(const float4*)(Ss + i * DV + PER * tx + c);
            const float bb[4] = {b.x, b.y, b.z, b.w}, rr[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[a][c + u] = fmaf(rr[a], bb[u], acc[a][c + u]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
        if (4 * ty + a < nt)
#pragma unroll
            for (int c = 0; c < PER; c += 4) *(float4*)(Og + a * DV + c) = make_float4(acc[a][c], acc[a][c + 1], acc[a][c + 2], acc[a][c + 3]);
}

template <class Tin, int DK, int TB, int IG>
const void* recur_fn(int rg, int gpt) {
    switch (4 * (gpt - 1) + rg) {
        case 1: return (const void*)recur_kernel<Tin, DK, 1, 1, TB, IG>;
        case 2: return (const void*)recur_kernel<Tin, DK, 2, 1, TB, IG>;
        case 3: return (const void*)recur_kernel<Tin, DK, 3, 1, TB, IG>;
        case 4: return (const void*)recur_kernel<Tin, DK, 4, 1, TB, IG>;
        case 5: return (const void*)recur_kernel<Tin, DK, 1, 2, TB, IG>;
        case 9: return (const void*)recur_kernel<Tin, DK, 1, 3, TB, IG>;
        default: return (const void*)recur_kernel<Tin, DK, 1, 4, TB, IG>;
    }
}
template <class Tin>
const void* recur_fn(int d_k, int tb, int rg, int gpt) {
    if (d_k == 128) return tb == 4 ? recur_fn<Tin, 128, 4, 4>(rg, gpt) : recur_fn<Tin, 128, 1, 4>(rg, gpt);
    return tb == 4 ? recur_fn<Tin, 64, 4, 4>(rg, gpt) : recur_fn<Tin, 64, 1, 4>(rg, gpt);
}

// the chain of one token
double token_us(const Problem& p) {
    static const double cyc[2][4] = {{204, 259, 330, 401}, {275, 373, 480, 590}};      // d_k = 64 and 128, sum form
    const bool big = p.d_k == 128;
    return (p.mask_group() == p.r ? cyc[big][p.r - 1] : p.r * cyc[big][0] * 0.9) / 1900.0;
}

struct RecurPlan {
    int nseg, seg_tok;
};
size_t seg_bytes(const Problem& p, int nseg) {
    const size_t nseq = (size_t)p.B * p.H, slots = nseq * nseg;
    return align_up(nseq * p.L * p.d_k * 4, 256) + align_up(slots * p.d_k * p.d_k * 4, 256) + 2 * align_up(slots * p.d_k * p.d_v * 4, 256);
}
// Segments, where they make the call shorter (one fp32 head of 256 tokens: 19 us instead of 29): the walk of a token costs about the same while at most one CTA
// (d_k = 64: two, whose chains leave each other most of the issue slots) runs per SM; against it stand two more kernels, 1 to 2
// us of composing per segment, and the traffic and products of the responses.
RecurPlan make_plan(const Problem& p) {
    RecurPlan plan{1, p.L};
    if (p.L < 128 || p.wu_builder) return plan;
    const long long nseq = (long long)p.B * p.H, sms = sm_count();
    const bool big = p.d_k == 128;
    const double tok = token_us(p);
    const double walk = nseq * (p.d_v / RJ) > sms ? 0.0 : 4.0 + p.L * tok;      // (one wave: otherwise there is nothing to gain)
    const double extra = (big ? 17.0 : 12.0) + (double)nseq * p.L * (p.d_k * p.d_v / 12e6 + (8.0 * p.d_k + 8.0 * p.d_v) / 4e6);
    double best = 0.92 * walk;
    const long long most = (sms * (big ? 1 : 2) / nseq + p.d_k / RJ) / (p.d_v / RJ + p.d_k / RJ);
    for (int want = 2; want <= most && want <= 64; ++want) {
        const int seg_tok = (p.L + 16 * want - 1) / (16 * want) * 16, nseg = (p.L + seg_tok - 1) / seg_tok;
        const long long ctas = nseq * (nseg * (p.d_v / RJ) + (nseg - 1) * (p.d_k / RJ));
        const double us = extra + nseg * (big ? 1.9 : 0.7) + seg_tok * tok * (ctas > sms ? 1.2 : 1.0);
        // (a caller's workspace was sized for the chunk-form kernels of pf_simt.cu)
        if (nseg > 1 && us < best && (p.own_workspace || seg_bytes(p, nseg) + 256 <= simt_workspace_bytes(p))) {
            best = us;
            plan = {nseg, seg_tok};
        }
    }
    return plan;
}

template <int DK, int WARPS>
int launch_compose(const Problem& p, const RecurPlan& plan, const RecurSeg& sg, int nseq, int dv) {
    constexpr int rows = 4 * (WARPS / (DK / 32)), smem = (DK * (DK + 4) + rows * DK) * 4;
    static std::atomic<uint64_t> opted_in{0};
    const int st = allow_smem(opted_in, (const void*)recur_compose<DK, WARPS>, smem);
    if (st != PF_OK) return st;
    prof_begin("recur_compose", p.stream);
    void* args[] = {(void*)&sg, (void*)&p.S_final, (void*)&plan.nseg, (void*)&dv};
    PF_CUDA_TRY(launch_early((const void*)recur_compose<DK, WARPS>, dim3((unsigned)(nseq * (dv / rows))), 32 * WARPS, args, smem, p.stream));
    prof_end(p.stream);
    return PF_OK;
}
template <int DK, int DV>
int launch_seg_tail(const Problem& p, const RecurPlan& plan, const RecurSeg& sg) {
    const int nseq = p.B * p.H, dv = DV;
    const int st0 = DK == 64 || nseq * (DV / 4) <= sm_count() ? launch_compose<DK, DK / 32>(p, plan, sg, nseq, dv) : launch_compose<DK, 8>(p, plan, sg, nseq, dv);
    if (st0 != PF_OK) return st0;
    constexpr int smem = (DK * DV + DK * 68) * 4;
    static std::atomic<uint64_t> opted_in{0};
    const int st = allow_smem(opted_in, (const void*)recur_apply<DK, DV>, smem);
    if (st != PF_OK) return st;
    prof_begin("recur_apply", p.stream);
    void* args[] = {(void*)&sg, (void*)&p.O, (void*)&p.L, (void*)&plan.seg_tok, (void*)&plan.nseg};
    PF_CUDA_TRY(launch_early((const void*)recur_apply<DK, DV>, dim3((unsigned)((plan.seg_tok + 63) / 64), (unsigned)(nseq * (plan.nseg - 1))),
                             256, args, smem, p.stream));
    prof_end(p.stream);
    count_launch(2);
    return PF_OK;
}

}  // namespace

// The kernel's time for a call of a few tokens, without segments (measured up to 64 tokens and 512 sequences): the chain of one
// token, or where the CTAs are more than the SMs their instructions, which leave little to overlap.
double recur_short_us(const Problem& p) {
    const double ctas = (double)p.B * p.H * (p.d_v / RJ), sms = sm_count() > 0 ? sm_count() : 1;
    const double crowd = (p.d_k == 128 ? 0.9 : 0.72) * ctas / sms;
    return 3.3 + p.L * 1.1 * token_us(p) * (crowd > 1.0 ? crowd : 1.0);
}

size_t recur_workspace_bytes(const Problem& p) {
    const RecurPlan plan = make_plan(p);
    return plan.nseg > 1 ? seg_bytes(p, plan.nseg) + 256 : 0;
}

int recur_forward(const Problem& p, void* workspace) {
    RecurGeo g{};
    g.L = p.L; g.d_v = p.d_v; g.exact = p.exact; g.clear = p.clear_status;
    const int rg = p.mask_group();
    const int tb = p.L < 4 ? 1 : 4;
    g.ts = p.L >= 16 ? 16 : (p.L < 1 ? 1 : (p.L + tb - 1) / tb * tb);
    const bool f32 = p.in_dtype == PF_DTYPE_F32;
    const RecurPlan plan = workspace ? make_plan(p) : RecurPlan{1, p.L};
    g.nseg = plan.nseg;
    g.seg_tok = plan.seg_tok;
    RecurSeg sg{};
    if (plan.nseg > 1) {
        const size_t slots = (size_t)p.B * p.H * plan.nseg;
        uint8_t* ws = (uint8_t*)workspace + 256;          // (word 0 of a caller's workspace is the status word)
        auto take = [&](size_t bytes) {
            float* at = (float*)ws;
            ws += align_up(bytes, 256);
            return at;
        };
        sg.R = take((size_t)p.B * p.H * p.L * p.d_k * 4);
        sg.P = take(slots * p.d_k * p.d_k * 4);
        sg.Xi = take(slots * p.d_k * p.d_v * 4);
        sg.start = take(slots * p.d_k * p.d_v * 4);
    }
    const int nb = (p.L + g.ts - 1) / g.ts;
    const int smem = (nb < R_STAGES ? (nb < 1 ? 1 : nb) : R_STAGES) * recur_stage_bytes(g.ts, p.r, p.d_k, f32 ? 4 : 2) +
                     4 * 128 * 4;           // (one group of keys is read past the last stage)
    const void* fn = f32 ? recur_fn<float>(p.d_k, tb, rg, p.r / rg) : recur_fn<__nv_bfloat16>(p.d_k, tb, rg, p.r / rg);
    const long long grid = (long long)p.B * p.H * (plan.nseg * (p.d_v / RJ) + (plan.nseg - 1) * (p.d_k / RJ));
    if (grid > 0x7fffffffLL) return PF_ERR_UNSUPPORTED;
    // (opted in once per kernel, to what its longest stages need)
    static std::atomic<uint64_t> opted_in[2][2][2][16];
    if (smem > 48 * 1024) {
        const int st = allow_smem(opted_in[f32][p.d_k == 128][tb == 4][(rg - 1) * 4 + p.r - 1], fn,
                                  R_STAGES * recur_stage_bytes(16, p.r, p.d_k, f32 ? 4 : 2) + 4 * 128 * 4);
        if (st != PF_OK) return st;
    }
    void* args[] = {(void*)&p.q, (void*)&p.k, (void*)&p.v, (void*)&p.beta, (void*)&p.S0, (void*)&p.O, (void*)&p.S_final, (void*)&p.status, (void*)&g, (void*)&sg};
    prof_begin("recur", p.stream);
    PF_CUDA_TRY(launch_early(fn, dim3((unsigned)grid), 160, args, (size_t)smem, p.stream));
    prof_end(p.stream);
    count_launch(1);
    if (plan.nseg == 1) return PF_OK;
    if (p.d_k == 128) return p.d_v == 128 ? launch_seg_tail<128, 128>(p, plan, sg) : launch_seg_tail<128, 64>(p, plan, sg);
    return p.d_v == 128 ? launch_seg_tail<64, 128>(p, plan, sg) : launch_seg_tail<64, 64>(p, plan, sg);
}

}  // namespace pf
