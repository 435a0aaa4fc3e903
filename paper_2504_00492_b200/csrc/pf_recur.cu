// recur: the recurrence itself, token by token, in fp32 with the state in registers (Section 1.1 readout, Section 1.3 /
// 3.1 update), for the calls whose time the chunk form cannot improve: every fp32 call, and bf16 calls of a few tokens.
//
// Per token the recurrence needs (4 r + 2) d_k d_v operations, less than half of what the chunk form needs on FFMA (no
// Gram product, no inverse, no W / Uh), and no intermediate ever leaves the SM: q, k, v, beta are read once per 32 columns
// of the state, O is written once.  What bounds it is the serial chain of one token (dot products, two shuffle stages, the
// update): 204 cycles at d_k = 64, r = 1 and 373 at d_k = 128, r = 2, of which the FFMA pipe is busy for 160.
// Measured (fp32): B*H = 32, L = 2048, d = 128, r = 2: 0.397 ms against 4.9 ms for the four chunk-form kernels in
// pf_simt.cu; one head, L = 256, d = 64, r = 1: 32 us against 209.
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
             const float* __restrict__ S0, float* __restrict__ O, float* __restrict__ S_final, int* __restrict__ status, RecurGeo g) {
    constexpr int NI = DK / IG, r = RG * GPT;          // rows i of a column that a lane holds
    constexpr int JW = 32 / IG;                        // columns per warp (IG warps make up the CTA's 32 columns)
    constexpr bool AHEAD = RG * NI <= 64;              // keys are read one group ahead where registers allow it
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar_full[R_STAGES], bar_empty[R_STAGES];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slices = g.d_v / RJ;
    const long long seq = blockIdx.x / slices;
    const int j0 = (int)(blockIdx.x % slices) * RJ;
    const int L = g.L, d_v = g.d_v;
    const int rows_s = g.ts * r;                       // rows per stage (at most 64)
    const int nb = (L + g.ts - 1) / g.ts;
    const int stage_bytes = recur_stage_bytes(g.ts, r, DK, (int)sizeof(Tin));
    auto s_k = [&](int st) { return (Tin*)(smem + st * stage_bytes); };
    auto s_q = [&](int st) { return s_k(st) + rows_s * DK; };
    auto s_v = [&](int st) { return s_q(st) + g.ts * DK; };
    auto s_b = [&](int st) { return (float*)(s_v(st) + rows_s * RJ); };

    if (tid == 0) {
        if (blockIdx.x == 0 && g.clear) *status = 0;              // (the call's status word; a wait of this kernel expires a second later at the earliest)
        for (int x = 0; x < R_STAGES; ++x) {
            tc::mbar_init(&bar_full[x], 1);
            tc::mbar_init(&bar_empty[x], IG);
        }
        tc::mbar_fence_init();
    }
    __syncthreads();

    if (warp == IG) {
        // ---- loader: bulk copies of the stages (k and q of a stage are contiguous, v is one copy per row), step sizes, and
        //      zeros for the tokens that the last pass has beyond the sequence
        for (int b = 0; b < nb; ++b) {
            const int st = b % R_STAGES, t0 = b * g.ts;
            const int nt = min(g.ts, L - t0), np = (nt + TB - 1) / TB * TB;
            if (b >= R_STAGES && !tc::mbar_wait_clk(&bar_empty[st], (uint32_t)(b / R_STAGES - 1) & 1, status, 301)) return;
            const long long tok = seq * L + t0;
            if (lane == 0) {
                tc::mbar_expect_tx_only(&bar_full[st], (uint32_t)(nt * (r * DK + DK + r * RJ) * sizeof(Tin)));
                tc::bulk_load(s_k(st), k + tok * r * DK, (uint32_t)(nt * r * DK * sizeof(Tin)), &bar_full[st]);
                tc::bulk_load(s_q(st), q + tok * DK, (uint32_t)(nt * DK * sizeof(Tin)), &bar_full[st]);
            }
            __syncwarp();
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
    const long long sb = (seq * DK + 4 * ig) * d_v + j0 + jw;
#pragma unroll
    for (int n = 0; n < NI; n += 2) {
        const float* x = S0 + sb + (long long)(4 * IG * (n >> 2) + (n & 3)) * d_v;
        S[n / 2] = S0 ? pk2(x[0], x[d_v]) : 0ull;
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
        float* og = O + (seq * L + (long long)b * g.ts) * d_v + j0 + jw;
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
            store_if(og + (long long)tok * d_v, y, tok < nt && (TB == 4 ? (lane & 7) < JW : lane < JW));
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_empty[st]);
    }
    if (S_final)
#pragma unroll
        for (int n = 0; n < NI; n += 2) {
            float* x = S_final + sb + (long long)(4 * IG * (n >> 2) + (n & 3)) * d_v;
            const float2 s2 = up2(S[n / 2]);
            x[0] = s2.x;
            x[d_v] = s2.y;
        }
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

}  // namespace

int recur_forward(const Problem& p) {
    RecurGeo g{};
    g.L = p.L; g.d_v = p.d_v; g.exact = p.exact; g.clear = p.clear_status;
    const int rg = p.mask_group();
    const int tb = p.L < 4 ? 1 : 4;
    g.ts = p.L >= 16 ? 16 : (p.L < 1 ? 1 : (p.L + tb - 1) / tb * tb);
    const bool f32 = p.in_dtype == PF_DTYPE_F32;
    const int nb = (p.L + g.ts - 1) / g.ts;
    const int smem = (nb < R_STAGES ? (nb < 1 ? 1 : nb) : R_STAGES) * recur_stage_bytes(g.ts, p.r, p.d_k, f32 ? 4 : 2) +
                     4 * 128 * 4;           // (one group of keys is read past the last stage)
    const void* fn = f32 ? recur_fn<float>(p.d_k, tb, rg, p.r / rg) : recur_fn<__nv_bfloat16>(p.d_k, tb, rg, p.r / rg);
    const long long grid = (long long)p.B * p.H * (p.d_v / RJ);
    if (grid > 0x7fffffffLL) return PF_ERR_UNSUPPORTED;
    // (opted in once per kernel, to what its longest stages need)
    static std::atomic<uint64_t> opted_in[2][2][2][16];
    if (smem > 48 * 1024) {
        const int st = allow_smem(opted_in[f32][p.d_k == 128][tb == 4][(rg - 1) * 4 + p.r - 1], fn,
                                  R_STAGES * recur_stage_bytes(16, p.r, p.d_k, f32 ? 4 : 2) + 4 * 128 * 4);
        if (st != PF_OK) return st;
    }
    void* args[] = {(void*)&p.q, (void*)&p.k, (void*)&p.v, (void*)&p.beta, (void*)&p.S0, (void*)&p.O, (void*)&p.S_final, (void*)&p.status, (void*)&g};
    prof_begin("recur", p.stream);
    PF_CUDA_TRY(cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(160), args, (size_t)smem, p.stream));
    prof_end(p.stream);
    count_launch(1);
    return PF_OK;
}

}  // namespace pf
