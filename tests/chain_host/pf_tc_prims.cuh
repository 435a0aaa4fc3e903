// What csrc/pf_chain.cu needs of csrc/pf_tc_prims.cuh, for run.cpp: barriers are its own, data is not modelled (a product is
// complete when it is issued, a copy has landed when it is asked for, tensor memory holds zeros).
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "pf_common.cuh"

namespace pf {
inline void wait_for_previous_kernel() {}
inline void let_next_kernel_start() {}
namespace tc {
constexpr int WAIT_TRIES = 1 << 18;
constexpr long long WAIT_CYCLES = 2000000000ll;
inline uint32_t smem_u32(const void* p) { return (uint32_t)(uintptr_t)p; }
inline void mbar_init(uint64_t* bar, uint32_t count) { host::mbar_init(smem_u32(bar), (int)count); }
inline void mbar_fence_init() {}
inline void mbar_arrive_at(uint32_t bar) { host::mbar_arrive(bar); }
inline void mbar_expect_tx_at(uint32_t bar, uint32_t) { host::landed(bar); }
template <bool LAZY>
inline bool mbar_wait_tries(uint32_t bar, uint32_t parity, int tries = WAIT_TRIES) { return host::mbar_wait(bar, (int)parity, tries > 1); }
inline void named_bar(int id, int n) { host::named(id, n, true); }
inline bool named_bar_and(int id, int n, bool x) { host::named(id, n, true); return x; }
inline int ld_acquire_gpu(const int* p) { return *p; }
inline void st_release_gpu(int* p, int v) { *p = v; }
inline float ld_cg_f32(const float* p) { return *p; }
inline void fence_async_smem() {}
inline void tc_fence_before() {}
inline void tc_fence_after() {}
inline void prefetch_tmap(const CUtensorMap*) {}
inline void tma_load_4d(uint32_t, const CUtensorMap*, int, int, int, int, uint32_t) {}
inline void tmem_alloc(uint32_t* at, uint32_t) { *at = 0; }
inline void tmem_dealloc(uint32_t, uint32_t) {}
template <int N> inline void zeros(uint32_t (&r)[N]) { for (auto& x : r) x = 0; }
inline void tmem_ld32(uint32_t, uint32_t (&r)[32]) { zeros(r); }
inline void tmem_ld16(uint32_t, uint32_t (&r)[16]) { zeros(r); }
template <int N> inline void tmem_ld_frag(uint32_t, uint32_t (&r)[N / 2]) { zeros(r); }
inline void tmem_ld_wait() {}
template <int N> inline void tmem_st32(uint32_t, const uint32_t (&)[N]) {}
template <int N> inline void tmem_st16(uint32_t, const uint32_t (&)[N]) {}
template <int N> inline void tmem_st8(uint32_t, const uint32_t (&)[N]) {}
inline void tmem_st_wait() {}
inline uint64_t make_desc_ns(uint32_t, uint32_t, uint32_t) { return 0; }
constexpr uint32_t make_idesc(int, bool, bool, bool) { return 0; }
inline void mma_f16(uint32_t, uint64_t, uint64_t, uint32_t, bool) {}
inline void mma_f16_ta(uint32_t, uint32_t, uint64_t, uint32_t, bool) {}
inline bool elect_one() { return host::lane() == 0; }
enum { L_SWK = 0, L_SWMN = 1 };
template <int LAY, int ROWS> constexpr uint32_t kstep_off(int) { return 0; }
inline void mma_16816(float (&)[4], const uint32_t (&)[4], uint32_t, uint32_t) {}
inline void mma_acc(float (&c)[4], const uint32_t (&)[4], uint32_t, uint32_t, bool) { c[0] = c[1] = c[2] = c[3] = 0.f; }
inline void ldmatrix_x4(uint32_t (&r)[4], uint32_t) { zeros(r); }
inline void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t) { zeros(r); }
inline uint32_t pack_h2(float, float) { return 0; }
inline void frag_mul(float (&)[2][4], const uint32_t (&)[4], const uint32_t (&)[4]) {}
inline void frag_pack(uint32_t (&f)[4], const float (&)[2][4]) { zeros(f); }
}  // namespace tc
}  // namespace pf
