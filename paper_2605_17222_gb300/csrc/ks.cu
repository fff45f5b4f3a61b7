// Key-switching inner product (K4) and plaintext-diagonal multiply-accumulate
// (K6) kernels, sm_103a.
//
// Both kernels read their ring elements in the NTT domain with the hoisted
// automorphism fused in as an index gather: Algorithms 1-2 rotate the
// switching key, swk~_r = phi_{-r}(swk_r), and apply phi_r after the inner
// product; since phi_r is a pure permutation of NTT-domain words,
//     phi_r(x + <d, phi_{-r}(swk)>) = phi_r(x) + <phi_r(d), swk>
// holds word for word, so the standard key is streamed once, in order, and
// the digits are gathered.  In bit-reversed storage the gather maps every
// aligned run of 32 words onto one aligned run of 32 words (Eq. 8), so a
// warp's gathered load touches exactly the same 256 bytes as a plain load.
//
// Sums of products stay in carry-free accumulators of split operands (Sum40,
// Sum60, WsAcc) and are reduced once (PE modes CWPM-ACC / CM-ACC of Sec. V,
// done lazily).
#include "kernels.h"
#include "ks_products.cuh"
#include "mbar.cuh"

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace ckks {
namespace {

constexpr int THREADS = 256;

// ------------------------------------------------------------------ stored words
__device__ __forceinline__ u64 diag_at(const unsigned char* limb, u32 s, bool packed) {
    if (!packed) return ((const u64*)limb)[s];
    const unsigned char* b = limb + (size_t)(s / BLK) * (BLK * 5);
    const u32 l = s % BLK;
    return ((const u32*)b)[l] | (u64)b[BLK * 4 + l] << 32;
}

// ------------------------------------------------------------------ K4
// What a thread knows of its position, and the ends of a product.
struct KsPos {
    u32 t, s, gmod;
};
__device__ __forceinline__ KsPos ks_pos(const KsArgs& a, u32 run) {
    const u32 t = blockIdx.y;
    return {t, run * BLK + threadIdx.x, t < a.level ? t : a.L + (t - a.level)};
}
__device__ __forceinline__ u64 ks_x0(const KsArgs& a, const KsItem& E, const KsPos& p, u32 src, u64 q) {
    if (a.x0_mode == 1) return E.x0[((size_t)p.t << a.log_n) + src];
    if (a.x0_mode == 2 && p.t < a.level)
        return mul_shoup(E.x0[((size_t)p.t << a.log_n) + src], a.lift_c[p.gmod], a.lift_sh[p.gmod], q);
    return 0;
}
__device__ __forceinline__ void ks_store(const KsArgs& a, const KsItem& E, const KsPos& p, u64 v0, u64 v1, u64 q) {
    u64* o0 = E.out0 + p.t * a.o_limb + (p.s / BLK) * a.o_blk + p.s % BLK;
    u64* o1 = E.out1 + ((size_t)p.t << a.log_n) + p.s;
    v0 = canon8(v0, q), v1 = canon8(v1, q);
    if (a.accumulate) v0 = add_mod(v0, *o0, q), v1 = add_mod(v1, *o1, q);
    *o0 = v0;
    *o1 = v1;
}

// Staged K4.  The kernel streams keys and digits and computes little, so what
// bounds it is the bytes in flight: a CTA of BLK threads owns a run of BLK
// positions of limb t, one thread copies a product's digit runs and key block
// into a shared-memory stage (bulk copies, one mbarrier per stage), and the
// register file holds none of what is in flight.  With sum = 1 the CTA walks
// its products through two stages.  One product of the N = 2^16 level-24
// shape takes 47.6 us (250 MB, 5.3 TB/s); by loads into registers, four CTAs of
// 256 per SM, it took 62 us, and 56 with unpacked keys (305 MB).
// The wait is bounded (1 s).  A CTA whose wait gives up leaves together after
// it has waited, bounded, for its copies in flight, and sets *err.
template <int BETA>
__global__ void __launch_bounds__(BLK, 8) k_ks_ws(const __grid_constant__ KsArgs a, u32 stage) {
    constexpr u32 RB = BLK * 8;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) u64 full_bar[2];
    const u32 l = threadIdx.x;
    const u32 first = a.sum ? 0 : blockIdx.x % a.count, last = a.sum ? a.count : first + 1;
    const u32 run = a.sum ? blockIdx.x : blockIdx.x / a.count;
    const KsPos p = ks_pos(a, run);
    if (l == 0) {
        mbar_init(&full_bar[0], 1);
        mbar_init(&full_bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    const ModC m = a.mods[p.gmod];
    const bool packed = packed_q(m.q);
    const u32 kb = key_blk(packed, BETA, a.beta_max), hb = key_hi(a.beta_max);
    const size_t koff = m.koff + (size_t)run * key_blk(packed, a.beta_max, a.beta_max);
    auto issue = [&](u32 e) {  // thread 0: product e into stage (e - first) % 2
        const KsItem& E = a.e[e];
        unsigned char* st = smem + ((e - first) & 1) * stage;
        u64* bar = &full_bar[(e - first) & 1];
        const u32 srun = (E.gal ? auto_src(run * BLK, E.gal, a.log_n) : run * BLK) / BLK;
        mbar_expect_tx(bar, BETA * RB + kb);
        tma_load_1d(st + BETA * RB, E.key + koff, kb, bar);
        const u64* d = E.digits + p.t * a.dl.limb + srun * a.dl.blk;
        if (a.dl.dig == BLK) {
            tma_load_1d(st, d, BETA * RB, bar);
        } else {
#pragma unroll
            for (int b = 0; b < BETA; b++) tma_load_1d(st + b * RB, d + b * a.dl.dig, RB, bar);
        }
    };
    pdl_wait();
    if (l == 0) {
        issue(first);
        if (first + 1 < last) issue(first + 1);
    }
    u64 v0 = 0, v1 = 0;
    if (a.sum) {
        v0 = a.e[0].out0[((size_t)p.t << a.log_n) + p.s];
        v1 = a.e[0].out1[((size_t)p.t << a.log_n) + p.s];
    }
    __syncthreads();  // the barriers are set up
    for (u32 e = first; e < last; e++) {
        const KsItem& E = a.e[e];
        const u32 src = E.gal ? auto_src(p.s, E.gal, a.log_n) : p.s, it = e - first;
        v0 += ks_x0(a, E, p, src, m.q);  // below 6q
        const bool ok = mbar_wait_bounded(&full_bar[it & 1], (it >> 1) & 1);
        if (__syncthreads_or(!ok)) {
            if (l == 0) {
                for (u32 i = it; i < min(it + 2, last - first); i++) mbar_wait_bounded(&full_bar[i & 1], (i >> 1) & 1);
                atomicExch(a.err, 1u);
            }
            return;
        }
        const unsigned char* st = smem + (it & 1) * stage;
        const u64* dg = (const u64*)st + src % BLK;
        const unsigned char* K = st + BETA * RB;
        u64 d[BETA];
#pragma unroll
        for (int b = 0; b < BETA; b++) d[b] = dg[b * BLK];
        if (packed) {
            const u32 mu32 = (u32)m.mu_hi;
            const u32* hp = (const u32*)(K + l * hb);
            const uint2* kp = (const uint2*)(K + BLK * hb) + l;
            Sum40 s0, s1;
            u32 w = 0;
#pragma unroll
            for (int b = 0; b < BETA; b++) {
                if (!(b & 1)) w = hp[b / 2];
                const uint2 k = kp[b * BLK];
                u32 dl, dh;
                split20(d[b], dl, dh);
                s0.mac(dl, dh, k.x, (w >> (16 * (b & 1))) & 0xFFu);
                s1.mac(dl, dh, k.y, (w >> (16 * (b & 1) + 8)) & 0xFFu);
            }
            v0 = s0.value(v0, m.q, mu32);
            v1 = s1.value(v1, m.q, mu32);
        } else {
            const ulonglong2* kp = (const ulonglong2*)K + l;
            Sum60 s0, s1;
#pragma unroll
            for (int b = 0; b < BETA; b++) {
                const ulonglong2 k = kp[b * BLK];
                u32 dl, dh, kl, kh;
                split30(d[b], dl, dh);
                split30(k.x, kl, kh);
                s0.mac(dl, dh, kl, kh);
                split30(k.y, kl, kh);
                s1.mac(dl, dh, kl, kh);
            }
            v0 = s0.value(v0, m);
            v1 = s1.value(v1, m);
        }
        if (e + 2 < last) {
            __syncthreads();  // the stage has been read
            if (l == 0) {
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                issue(e + 2);
            }
        }
    }
    if (a.sum) {
        a.e[0].out0[((size_t)p.t << a.log_n) + p.s] = canon8(v0, m.q);
        a.e[0].out1[((size_t)p.t << a.log_n) + p.s] = canon8(v1, m.q);
    } else {
        ks_store(a, a.e[first], p, v0, v1, m.q);
    }
}

// Any number of digits, operands straight from global memory: more than eight
// digits, or unaligned ones.  Sixteen digits at N = 2^15, the seven products of the
// (1,8,4) split: 119 us.
__global__ void __launch_bounds__(BLK) k_ks_any(const __grid_constant__ KsArgs a) {
    const u32 first = a.sum ? 0 : blockIdx.x % a.count, last = a.sum ? a.count : first + 1;
    const u32 run = a.sum ? blockIdx.x : blockIdx.x / a.count;
    const KsPos p = ks_pos(a, run);
    const ModC m = a.mods[p.gmod];
    const bool packed = packed_q(m.q);
    const size_t koff = m.koff + (size_t)run * key_blk(packed, a.beta_max, a.beta_max);
    const size_t o = ((size_t)p.t << a.log_n) + p.s;
    pdl_wait();
    u64 v0 = 0, v1 = 0;
    if (a.sum) v0 = a.e[0].out0[o], v1 = a.e[0].out1[o];
    for (u32 e = first; e < last; e++) {
        const KsItem& E = a.e[e];
        const u32 src = E.gal ? auto_src(p.s, E.gal, a.log_n) : p.s;
        v0 += ks_x0(a, E, p, src, m.q);
        const u64* D = E.digits + p.t * a.dl.limb + (src / BLK) * a.dl.blk + src % BLK;
        if (packed) ks_products<true>(m, D, a.dl.dig, E.key + koff, threadIdx.x, a.beta, a.beta_max, v0, v1);
        else ks_products<false>(m, D, a.dl.dig, E.key + koff, threadIdx.x, a.beta, a.beta_max, v0, v1);
    }
    if (a.sum) a.e[0].out0[o] = canon8(v0, m.q), a.e[0].out1[o] = canon8(v1, m.q);
    else ks_store(a, a.e[first], p, v0, v1, m.q);
}

// ------------------------------------------------------------------ K6
// For one word s of limb t and K3 giant indices k (a chunk of the n3 outer
// rotations) this computes
//   U_{c,k}[s] = sum_{j < n2} sum_{i < n1} pair_c(i, j)[s] * f_{n1 n2 k + n1 j + i}[h_k(s)]
// where h_k is the gather of phi_{-n1 n2 k} (the pre-rotated diagonal
// f^ = phi_{-n1 n2 k}(f), Alg. 2 input) and
//   pair(i, 0) = (A_i, B_i)                                    (Alg. 2 lines 2-5)
//   pair(i, j) = phi_{n1 j}(A_i + <D_i, swk~_0>, <D_i, swk~_1>) (Alg. 2 lines 9-10)
// so Alg. 2 lines 8-14 (Phases 3 and 4 of Sec. IV) run without writing the
// n1*n2 rotated ciphertexts to HBM.  DH-BSGS is the case n2 = 1, the diagonal
// method n1 = 1, BSGS n2 = 1 over Q only.
//
// This plain form reads its operands straight from global memory; it runs what
// the staged kernel does not take: stages that do not fit (about forty digits,
// or up to eight of a key with well over a hundred), operands at an odd word,
// and bases of more than DM_MAX_LIMBS limbs.
template <int K3>
__global__ void __launch_bounds__(THREADS, 2) k_diag_mac(const __grid_constant__ DiagMacArgs a, u32 l0) {
    const u32 N = 1u << a.log_n;
    const u32 bidx = blockIdx.x % a.batch;
    const u32 s = (blockIdx.x / a.batch) * THREADS + threadIdx.x;
    const size_t ox = bidx * a.bs_x, ob = bidx * a.bs_b, ou = bidx * a.bs_u;
    const u32 t = a.ext <= (u32)DM_MAX_LIMBS ? a.limbs[l0 + blockIdx.y] : blockIdx.y;
    if (s >= N) return;
    const u32 k_first = blockIdx.z * K3;
    const u32 k_count = min((u32)K3, a.n3 - k_first);
    const u32 gmod = t < a.level ? t : a.L + (t - a.level);
    const ModC m = a.mods[gmod];
    const bool packed = packed_q(m.q);
    const size_t drow = m.doff + (t < a.level ? 0 : a.diag_p);
    const size_t koff = m.koff + (size_t)(s / BLK) * key_blk(packed, a.beta_max, a.beta_max);
    const size_t tN = (size_t)t * N;
    const u32 n1n2 = a.n1 * a.n2;
    const bool lift_limb = a.lift0 && t < a.level;
    const u64 lc = lift_limb ? a.lift_c[gmod] : 0, lsh = lift_limb ? a.lift_sh[gmod] : 0;

    const unsigned char* fb[K3];
    u32 fs[K3];
#pragma unroll
    for (int kk = 0; kk < K3; kk++) {
        const u32 kc = k_first + min((u32)kk, k_count - 1);  // lanes past the chunk mirror its last index
        const u32 g = a.gal_diag[kc];
        fb[kk] = a.diags + (size_t)(n1n2 * kc) * a.diag_stride + drow;
        fs[kk] = g ? auto_src(s, g, a.log_n) : s;
    }
    U128 acc0[K3], acc1[K3];
#pragma unroll
    for (int kk = 0; kk < K3; kk++) acc0[kk] = acc1[kk] = U128{0, 0};
    u32 terms = 0;
    pdl_wait();

    for (u32 j = 0; j < a.n2; j++) {
        const u32 src = j ? auto_src(s, a.gal_mid[j], a.log_n) : s;
        for (u32 i = 0; i < a.n1; i++) {
            const bool lifted = (i == 0) && a.lift0;
            const size_t didx = (size_t)(a.n1 * j + i) * a.diag_stride;
            u64 f[K3];
#pragma unroll
            for (int kk = 0; kk < K3; kk++) f[kk] = kk < (int)k_count ? diag_at(fb[kk] + didx, fs[kk], packed) : 0;
            const u64* X = a.X[i] + ox + ((size_t)t * (N / BLK) + src / BLK) * (a.slots * BLK) + src % BLK;
            u64 av = lifted && !lift_limb ? 0 : X[(a.slots - 1) * BLK], bv = 0;
            if (j == 0) {
                if (!lifted) bv = (a.B[i] + ob)[tN + s];
                else if (lift_limb) bv = mul_shoup(a.c1[bidx][tN + s], lc, lsh, m.q);
            } else {
                if (packed) ks_products<true>(m, X, BLK, a.keys[j] + koff, s % BLK, a.beta, a.beta_max, av, bv);
                else ks_products<false>(m, X, BLK, a.keys[j] + koff, s % BLK, a.beta, a.beta_max, av, bv);
            }
#pragma unroll
            for (int kk = 0; kk < K3; kk++) {
                if (kk < (int)k_count) {
                    mac128(acc0[kk], av, f[kk]);
                    mac128(acc1[kk], bv, f[kk]);
                }
            }
            if (++terms == FLUSH) {
                terms = 0;
#pragma unroll
                for (int kk = 0; kk < K3; kk++) {
                    acc0[kk] = U128{reduce128(acc0[kk], m), 0};
                    acc1[kk] = U128{reduce128(acc1[kk], m), 0};
                }
            }
        }
    }
#pragma unroll
    for (int kk = 0; kk < K3; kk++) {
        if (kk < (int)k_count) {
            a.U0[k_first + kk][ou + tN + s] = reduce128(acc0[kk], m);
            a.U1[k_first + kk][ou + tN + s] = reduce128(acc1[kk], m);
        }
    }
}

// Failure-detection self-test: one thread waits on an mbarrier that nothing
// will complete, with the same bounded wait the staged kernel uses (limit
// given in ns), and records the give-up in *err.
__global__ void k_wait_selftest(u32* err, u64 limit_ns) {
    __shared__ __align__(8) u64 bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    const u64 t0 = global_ns();
    bool ok = false;
    while (!(ok = mbar_try_wait(&bar, 0)))
        if (global_ns() - t0 > limit_ns) break;
    if (!ok) atomicExch(err, 1u);
}

}  // namespace

// ------------------------------------------------------------------ packing keys and diagonals
namespace {
__device__ __forceinline__ u64 residue(u64 x, const ModC& m) {
    x -= __umul64hi(x, m.mu_hi) * m.q;  // [0, 2q)
    return x >= m.q ? x - m.q : x;
}

// One block of a limb per CTA of BLK threads; z: the diagonal.
__global__ void __launch_bounds__(BLK) k_pack_diags(const PackArgs a) {
    const u32 N = 1u << a.log_n, l = threadIdx.x, t = blockIdx.y, g = t < a.level ? t : a.L + (t - a.level);
    const ModC m = a.mods[g];
    const bool packed = packed_q(m.q);
    const u64 x = residue(a.in[((size_t)blockIdx.z * (a.level + a.k) + t) * N + blockIdx.x * BLK + l], m);
    unsigned char* o = a.out + blockIdx.z * a.stride + m.doff + (t < a.level ? 0 : a.p_base) +
                       (size_t)blockIdx.x * diag_blk(packed);
    if (packed) {
        ((u32*)o)[l] = (u32)x;
        o[BLK * 4 + l] = (unsigned char)(x >> 32);
    } else {
        ((u64*)o)[l] = x;
    }
}

// in [beta_max][2][L + k][N] -> the key layout; z: the digit.
__global__ void __launch_bounds__(BLK) k_pack_key(const PackArgs a) {
    const u32 N = 1u << a.log_n, l = threadIdx.x, g = blockIdx.y, b = blockIdx.z;
    const ModC m = a.mods[g];
    const bool packed = packed_q(m.q);
    const size_t plane = (size_t)(a.L + a.k) * N, w = (size_t)g * N + blockIdx.x * BLK + l;
    const u64 x0 = residue(a.in[2 * b * plane + w], m), x1 = residue(a.in[(2 * b + 1) * plane + w], m);
    unsigned char* o = a.out + m.koff + (size_t)blockIdx.x * key_blk(packed, a.beta_max, a.beta_max);
    if (packed) {
        const u32 hb = key_hi(a.beta_max);
        *(uchar2*)(o + l * hb + 2 * b) = make_uchar2((unsigned char)(x0 >> 32), (unsigned char)(x1 >> 32));
        ((uint2*)(o + BLK * (hb + 8 * b)))[l] = make_uint2((u32)x0, (u32)x1);
    } else {
        ((ulonglong2*)(o + BLK * 16 * b))[l] = make_ulonglong2(x0, x1);
    }
}
}  // namespace

void launch_pack_diags(const PackArgs& a, u32 count, cudaStream_t st) {
    PackArgs p = a;
    const size_t in_step = (size_t)(a.level + a.k) << a.log_n;
    for (u32 d0 = 0; d0 < count; d0 += 32768) {  // grid.z is 16 bits
        p.in = a.in + d0 * in_step;
        p.out = a.out + d0 * a.stride;
        k_pack_diags<<<dim3((1u << a.log_n) / BLK, a.level + a.k, std::min(32768u, count - d0)), BLK, 0, st>>>(p);
        count_launch();
    }
}

void launch_pack_key(const PackArgs& a, cudaStream_t st) {
    k_pack_key<<<dim3((1u << a.log_n) / BLK, a.L + a.k, a.beta_max), BLK, 0, st>>>(a);
    count_launch();
}

void launch_wait_selftest(u32* err, u64 limit_ns, cudaStream_t st) {
    k_wait_selftest<<<1, 32, 0, st>>>(err, limit_ns);
    count_launch();
}

template <int BETA>
static void run_ks_ws(const KsArgs& a, cudaStream_t st) {
    // two stages where a CTA walks several products, the limb with the larger stage
    const u32 stage = BETA * BLK * 8 + std::max(key_blk(true, BETA, a.beta_max), key_blk(false, BETA, a.beta_max));
    const u32 sm = a.sum && a.count > 1 ? 2 * stage : stage;
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t bit = 1ull << (dev & 63);
    if (!(done.load(std::memory_order_acquire) & bit) &&
        cudaFuncSetAttribute(k_ks_ws<BETA>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024) == cudaSuccess)
        done.fetch_or(bit, std::memory_order_release);
    const dim3 grid((1u << a.log_n) / BLK * (a.sum ? 1 : a.count), a.ext);
    launch(false, k_ks_ws<BETA>, grid, BLK, sm, st, a, stage);
}

void launch_ks(const KsArgs& a, cudaStream_t st) {
    ProfScope ps(K_KS_INNER, st, 2.0 * a.beta * a.count * a.ext * (1u << a.log_n));
    // Bulk copies read 16-byte aligned digits (a caller's may be at any word);
    // the stages fit 96 KB for up to eight digits of a key with up to 64.
    bool staged = a.beta_max <= 64;
    for (u32 e = 0; e < a.count; e++) staged = staged && ((uintptr_t)a.e[e].digits & 15) == 0;
    switch (staged ? a.beta : 0) {
        case 1: run_ks_ws<1>(a, st); break;
        case 2: run_ks_ws<2>(a, st); break;
        case 3: run_ks_ws<3>(a, st); break;
        case 4: run_ks_ws<4>(a, st); break;
        case 5: run_ks_ws<5>(a, st); break;
        case 6: run_ks_ws<6>(a, st); break;
        case 7: run_ks_ws<7>(a, st); break;
        case 8: run_ks_ws<8>(a, st); break;
        default: launch(false, k_ks_any, dim3((1u << a.log_n) / BLK * (a.sum ? 1 : a.count), a.ext), BLK, 0, st, a);
    }
    count_launch();
}

void launch_diag_mac(const DiagMacArgs& a, cudaStream_t st) {
    const u32 N = 1u << a.log_n;
    u32 k3 = 1;
    while (k3 < a.n3 && k3 < (u32)DM_MAX_K3) k3 *= 2;
    // a tile with fewer outer indices per CTA (more CTAs along z, each redoing the middle layer)
    if (a.tile_k3 && a.tile_k3 < k3 && !(a.tile_k3 & (a.tile_k3 - 1))) k3 = a.tile_k3;
    const dim3 grid(((N + THREADS - 1) / THREADS) * a.batch, a.ext, (a.n3 + k3 - 1) / k3);
    // multiply-accumulates: two per diagonal product (c0, c1), and the middle
    // layer's 2 beta per step with j > 0, once per block of k3 outer indices
    const double n1n2 = (double)a.n1 * a.n2, beta_mid = a.n2 > 1 ? a.beta : 0;
    const double macs = (double)N * a.batch * a.ext *
                        (2.0 * n1n2 * a.n3 + 2.0 * beta_mid * grid.z * (n1n2 - a.n1));
    ProfScope ps(K_DIAG_MAC, st, macs);
    // Bulk copies read 16-byte aligned runs; a wrapped ciphertext may lie at any word.
    bool aligned = true;
    for (u32 b = 0; b < a.batch; b++) aligned = aligned && ((uintptr_t)a.c1[b] & 15) == 0;
    for (u32 i = 0; i < a.n1; i++) aligned = aligned && (((uintptr_t)a.X[i] | (uintptr_t)a.B[i]) & 15) == 0;
    auto run = [&](auto k3c, auto packedc, bool join) {
        constexpr int K3 = decltype(k3c)::value;
        constexpr bool PACKED = decltype(packedc)::value;
        const u32 l0 = PACKED ? 0 : a.n_packed, n = PACKED ? a.n_packed : a.ext - a.n_packed;
        if (!n) return;
        if (!aligned || !launch_ws<K3, PACKED>(a, join, st))
            launch(false, k_diag_mac<K3>, dim3(grid.x, n, grid.z), THREADS, 0, st, a, l0);
        count_launch();
    };
    auto both = [&](auto k3c) {
        if (a.ext > (u32)DM_MAX_LIMBS) {
            launch(false, k_diag_mac<decltype(k3c)::value>, grid, THREADS, 0, st, a, 0u);
            count_launch();
            return;
        }
        run(k3c, std::false_type{}, false);
        run(k3c, std::true_type{}, a.n_packed < a.ext);
    };
    switch (k3) {
        case 1: both(std::integral_constant<int, 1>{}); break;
        case 2: both(std::integral_constant<int, 2>{}); break;
        case 4: both(std::integral_constant<int, 4>{}); break;
        default: both(std::integral_constant<int, 8>{}); break;
    }
}

}  // namespace ckks
