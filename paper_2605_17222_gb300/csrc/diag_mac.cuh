// The staged diagonal multiply-accumulate kernel (K6), instantiated per number
// of outer indices and class of limbs in diag_mac_<K3>_{packed,wide}.cu so that
// the instances compile in parallel.
#pragma once
#include "kernels.h"
#include "ks_products.cuh"
#include "mbar.cuh"

#include <algorithm>
#include <atomic>

namespace ckks {
namespace {

// ------------------------------------------------------------------ K6, warp-specialised
// The same computation with the copies issued by a warp of their own.  In
// bit-reversed storage every automorphism maps an aligned run of BLK words
// onto one aligned run (Eq. 8).  A CTA owns one run of BLK positions of limb
// t: four compute warps (one position a thread) and one producer warp.  Every
// operand of a step -- K3 diagonal blocks, the group of digit runs and the A
// run, the switching-key block (A and B runs at j = 0) -- arrives in a
// shared-memory stage by bulk copies, and the compute warps apply the in-run
// permutation.  Copies are issued by one thread one after another, so their
// number per step counts (K3 + 2; with a copy per digit, K3 + beta + 2, the
// copies alone took 1.36 ms of the 23 packed limbs at the (1,64,4) split).
// The ring's stages are ordered by two mbarriers per stage, with no CTA-wide
// barrier in the loop:
//   full[s]  : the producer's expect_tx; the stage's copies complete it.
//   empty[s] : one arrival per compute warp once the warp has read the stage;
//              the producer waits on it before it refills the stage.
// The ring takes as many stages as its share of shared memory holds (up to
// WS_MAX_STAGES; the packed limbs' stages are a quarter smaller, so they get
// more).
//
// At the N = 2^16 (1,64,4) split, 10.3 GB of keys and diagonals: 1.74 ms (2.45
// before: unpacked, 17 copies per step issued from the lanes of a warp,
// 96-bit carry chains).  The copies alone take 1.13 ms for the 23 packed limbs
// (6.7 TB/s), the arithmetic alone 1.2; the multiplier pipe is about 70% busy.
//
// Every wait is bounded (compute: wait_ns, default 1 s; producer: 1 s) and
// also gives up as soon as the CTA's abort flag is raised.  A warp whose wait
// gives up raises the flag and leaves its loop (all its lanes together); the
// producer stops issuing.  Each thread then reaches one final named barrier
// exactly once; after it, if the flag is up, the producer waits (1 s limit)
// for the last copies it issued into each stage -- a stage is only refilled
// after every warp consumed it, so at most one phase of each full barrier is
// pending -- sets *err, and the CTA writes no output.
constexpr u32 WS_THREADS = BLK + 32;
constexpr u32 WS_MAX_STAGES = 6;
// BETA of the instance for more than eight digits: a loop over groups of four
// digits from the stage, two CTAs per SM, or one if two stages need it.  Sixteen
// digits at N = 2^15, the (1,8,4) split: 229 us, and 286 at (2,4,8); the plain
// kernel takes 623 and 793 with branches between a group's loads.
constexpr int WS_ANY = 9;

// Sums of v * f, v a middle-layer word and f a diagonal word, per class of
// limb (chosen once per CTA).  TERMS products fit between two reductions.
enum WsClass { C40 = 0, C55 = 1, C60 = 2 };  // packed 40-bit; other moduli up to 55 bits; wider

// C40: v < 3q, f < q < 2^40, in 32-bit halves: L = sum v0 f0 (its carries go
// to H), M = sum v0 f1 + v1 f0 (below 2^44 a term), H = sum v1 f1 (below
// 2^17.6).  L and M are register pairs of their own, so that each product is
// one multiply-add: four a product and five registers, against seven and
// three for mac96, whose middle products straddle its register pairs.
template <int CLS>
struct WsAcc {
    static constexpr u32 TERMS = 16384;
    u64 L, M;
    u32 H;
    __device__ __forceinline__ void set(u64 x) { L = x, M = 0, H = 0; }
    __device__ __forceinline__ void mac(u64 v, u64 f) {
        asm("{\n\t.reg .u32 l0, l1, x0, x1, y0, y1;\n\t"
            "mov.b64 {l0, l1}, %0;\n\t"
            "mov.b64 {x0, x1}, %3;\n\t"
            "mov.b64 {y0, y1}, %4;\n\t"
            "mad.lo.cc.u32 l0, x0, y0, l0;\n\t"
            "madc.hi.cc.u32 l1, x0, y0, l1;\n\t"
            "madc.lo.u32 %2, x1, y1, %2;\n\t"
            "mad.wide.u32 %1, x0, y1, %1;\n\t"
            "mad.wide.u32 %1, x1, y0, %1;\n\t"
            "mov.b64 %0, {l0, l1};\n\t}"
            : "+l"(L), "+l"(M), "+r"(H)
            : "l"(v), "l"(f));
    }
    // the sum mod q: T = M + 2^32 H fits 64 bits; then L + 2^32 t (t < 3q) in
    // two steps of 62 and 54 bits
    __device__ __forceinline__ u64 value(const ModC& m) const {
        const u32 mu32 = (u32)m.mu_hi;
        const u64 u = (L >> 32) + reduce64_40(M + ((u64)H << 32), m.q, mu32);  // below 2^42
        const u64 r = reduce64_40(u << 20 | (u32)L >> 12, m.q, mu32);
        return canon8(reduce64_40(r << 12 | ((u32)L & 0xFFFu), m.q, mu32), m.q);
    }
};

// C55: v < 5q, f < q < 2^55.  As C40 with a 64-bit H; M's terms are below 2^57.7.
template <>
struct WsAcc<C55> {
    static constexpr u32 TERMS = 64;
    u64 L, M, H;
    __device__ __forceinline__ void set(u64 x) { L = x, M = 0, H = 0; }
    __device__ __forceinline__ void mac(u64 v, u64 f) {
        asm("{\n\t.reg .u32 l0, l1, h0, h1, x0, x1, y0, y1;\n\t"
            "mov.b64 {l0, l1}, %0;\n\t"
            "mov.b64 {h0, h1}, %2;\n\t"
            "mov.b64 {x0, x1}, %3;\n\t"
            "mov.b64 {y0, y1}, %4;\n\t"
            "mad.lo.cc.u32 l0, x0, y0, l0;\n\t"
            "madc.hi.cc.u32 l1, x0, y0, l1;\n\t"
            "madc.lo.cc.u32 h0, x1, y1, h0;\n\t"
            "madc.hi.u32 h1, x1, y1, h1;\n\t"
            "mad.wide.u32 %1, x0, y1, %1;\n\t"
            "mad.wide.u32 %1, x1, y0, %1;\n\t"
            "mov.b64 %0, {l0, l1};\n\t"
            "mov.b64 %2, {h0, h1};\n\t}"
            : "+l"(L), "+l"(M), "+l"(H)
            : "l"(v), "l"(f));
    }
    __device__ __forceinline__ u64 value(const ModC& m) const {
        U128 x{L, H + (M >> 32)};
        add128(x, M << 32);
        return reduce128(x, m);
    }
};

// C60: v < 5q, f < q < 2^60: 128-bit sums.
template <>
struct WsAcc<C60> {
    static constexpr u32 TERMS = FLUSH;
    U128 v;
    __device__ __forceinline__ void set(u64 x) { v = U128{x, 0}; }
    __device__ __forceinline__ void mac(u64 x, u64 f) { mac128(v, x, f); }
    __device__ __forceinline__ u64 value(const ModC& m) const { return reduce128(v, m); }
};

// What the compute threads of k_diag_mac_ws share.
struct WsCtx {
    const DiagMacArgs& a;
    const unsigned char* smem;
    u64* full_bar;
    u64* empty_bar;
    volatile u32* abort;
    const u32* jtab;  // per middle index: source run | gather constants (see the kernel)
    u32 s, l, k_first, k_count, ns, stage, off_a;
    size_t o;  // output word
    bool lift_limb;
    u64 lc, lsh;
    ModC m;
};

// The compute threads' step loop of k_diag_mac_ws (see there) and the output.
// A step is one serial chain per warp, and registers allow three or four warps
// per scheduler, so its latency is what counts: the loop body has no branch
// (BETA is exact, outer indices past k_count compute on stale words that are
// never stored), so that the middle layer's shared-memory loads are issued
// together.  The diagonal words are read after its products, whose registers
// they then take ((1,64,4) 1.78 -> 1.74 ms, Set-B 0.62 -> 0.58), but for wide limbs
// with one digit and eight outer indices, where two CTAs per SM leave registers
// for both: Set-A (16,16,16) 0.920 ms early, 0.963 late; (4,16,8) 146 us, 152; Set-B
// at level 8, (1,32,8) 372, 387.  With four they are even (88 and 88 us, 221 and
// 221), with one or two early is the slower (Set-A (4,16,2) 70 us, 68 late;
// (1,64,1) 67, 66; Set-B (1,32,2) 166, 160; (1,32,1) 147, 143).
template <int K3, int BETA, int CLS>
__device__ __forceinline__ void ws_compute(const WsCtx& c) {
    constexpr u32 FULLM = 0xffffffffu;
    constexpr u32 FB = CLS == C40 ? BLK * 5 : BLK * 8;  // diagonal block
    constexpr bool EARLY_F = BETA == 1 && K3 >= 8;      // wide limbs: diagonal words before the products (above)
    const DiagMacArgs& a = c.a;
    const u32 l = c.l, n1 = a.n1, n1n2 = a.n1 * a.n2;
    const ModC m = c.m;
    const u64 q = m.q;
    const u32 mu32 = (u32)m.mu_hi;  // floor(2^64 / q) (C40)
    const u32 lb = __brev(l) >> 25;  // brv_7(l)
    const u32 hb = key_hi(a.beta_max);
    const u32 off_key = c.off_a + BLK * 8;
    u32 pd[K3];  // in-run positions of the diagonal gathers
#pragma unroll
    for (int kk = 0; kk < K3; kk++) {
        const u32 g = a.gal_diag[c.k_first + min((u32)kk, c.k_count - 1)];
        pd[kk] = (g ? auto_src(c.s, g, a.log_n) : c.s) % BLK;
    }
    WsAcc<CLS> acc0[K3], acc1[K3];
#pragma unroll
    for (int kk = 0; kk < K3; kk++) acc0[kk].set(0), acc1[kk].set(0);
    const u64 wait_ns = a.wait_ns ? a.wait_ns : DM_WAIT_NS;
    u32 terms = 0, sidx = 0, phase = 0;
    bool ok = true;
    // the warp decides together, so that its lanes stay converged
    auto wait = [&] {
        ok = __all_sync(FULLM, mbar_wait_abortable(&c.full_bar[sidx], phase, wait_ns, c.abort));
        if (!ok) *c.abort = 1u;
        return ok;
    };
    u64 f[K3];  // the step's diagonal words
    auto load_f = [&](const unsigned char* st) {
#pragma unroll
        for (int kk = 0; kk < K3; kk++) {
            const unsigned char* fp = st + kk * FB;
            if constexpr (CLS == C40) f[kk] = ((const u32*)fp)[pd[kk]] | (u64)fp[BLK * 4 + pd[kk]] << 32;
            else f[kk] = ((const u64*)fp)[pd[kk]];
        }
    };
    auto release = [&] {
        __syncwarp();
        if ((l & 31) == 0) mbar_arrive(&c.empty_bar[sidx]);
        if (++sidx == c.ns) sidx = 0, phase ^= 1;
    };
    auto outer = [&](u64 av, u64 bv) {
#pragma unroll
        for (int kk = 0; kk < K3; kk++) {
            acc0[kk].mac(av, f[kk]);
            acc1[kk].mac(bv, f[kk]);
        }
        if (++terms == WsAcc<CLS>::TERMS) {
            terms = 0;
#pragma unroll
            for (int kk = 0; kk < K3; kk++) {
                acc0[kk].set(acc0[kk].value(m));
                acc1[kk].set(acc1[kk].value(m));
            }
        }
    };
    // j = 0: the pairs (A_i, B_i)
    for (u32 i = 0; i < n1 && ok; i++) {
        if (!wait()) break;
        const unsigned char* st = c.smem + sidx * c.stage;
        const bool lifted = i == 0 && a.lift0, zero = lifted && !c.lift_limb;
        const u64 av = zero ? 0 : ((const u64*)(st + c.off_a))[l];  // the first one comes lifted
        u64 bv = zero ? 0 : ((const u64*)(st + off_key))[l];
        load_f(st);
        release();
        if (lifted) bv = mul_shoup(bv, c.lc, c.lsh, q);
        outer(av, bv);
    }
    if constexpr (BETA > 0) {
        u32 i = 0, j = 1;
        for (u32 it = n1; it < n1n2 && ok; it++) {
            // in-run source of phi_{n1 j}: brv_7(C + g brv_7(l)), C and g mod 128 from the table
            const u32 e = c.jtab[j];
            const u32 pm = __brev((e >> 16) + (e >> 24) * lb) >> 25;
            const bool zero = i == 0 && a.lift0 && !c.lift_limb;
            if (++i == n1) i = 0, j++;
            if (!wait()) break;
            const unsigned char* st = c.smem + sidx * c.stage;
            const u64 x = zero ? 0 : ((const u64*)(st + c.off_a))[pm];
            const u64* dg = (const u64*)(st + K3 * FB) + pm;
            if constexpr (BETA == WS_ANY) {
                u64 av = x, bv = 0;
                ks_products<CLS == C40>(m, dg, BLK, st + off_key, l, a.beta, a.beta_max, av, bv);
                load_f(st);
                release();
                outer(av, bv);
                continue;
            }
            u64 d[BETA], av, bv;
#pragma unroll
            for (int b = 0; b < BETA; b++) d[b] = dg[b * BLK];
            if constexpr (CLS == C40) {
                const u32* hp = (const u32*)(st + off_key + l * hb);
                const uint2* kp = (const uint2*)(st + off_key + BLK * hb) + l;
                u32 w[(BETA + 1) / 2];
                uint2 k[BETA];
#pragma unroll
                for (int b = 0; b < BETA; b++) {
                    k[b] = kp[b * BLK];
                    if (!(b & 1)) w[b / 2] = hp[b / 2];
                }
                Sum40 s0, s1;
#pragma unroll
                for (int b = 0; b < BETA; b++) {
                    u32 dl, dh;
                    split20(d[b], dl, dh);
                    s0.mac(dl, dh, k[b].x, (w[b / 2] >> (16 * (b & 1))) & 0xFFu);
                    s1.mac(dl, dh, k[b].y, (w[b / 2] >> (16 * (b & 1) + 8)) & 0xFFu);
                }
                load_f(st);
                release();
                av = s0.value(x, q, mu32);
                bv = s1.value(0, q, mu32);
            } else {
                const ulonglong2* kp = (const ulonglong2*)(st + off_key) + l;
                ulonglong2 k[BETA];
#pragma unroll
                for (int b = 0; b < BETA; b++) k[b] = kp[b * BLK];
                if constexpr (EARLY_F) {
                    load_f(st);
                    release();
                }
                Sum60 s0, s1;
#pragma unroll
                for (int b = 0; b < BETA; b++) {
                    u32 dl, dh, kl, kh;
                    split30(d[b], dl, dh);
                    split30(k[b].x, kl, kh);
                    s0.mac(dl, dh, kl, kh);
                    split30(k[b].y, kl, kh);
                    s1.mac(dl, dh, kl, kh);
                }
                if constexpr (!EARLY_F) {
                    load_f(st);
                    release();
                }
                av = s0.value(x, m);
                bv = s1.value(0, m);
            }
            outer(av, bv);
        }
    }
    nbar_sync(1, WS_THREADS);  // every thread of the CTA reaches this once; then one decision for all
    if (*c.abort) return;
#pragma unroll
    for (int kk = 0; kk < K3; kk++) {
        if (kk < (int)c.k_count) {
            a.U0[c.k_first + kk][c.o] = acc0[kk].value(m);
            a.U1[c.k_first + kk][c.o] = acc1[kk].value(m);
        }
    }
}

// The source run of phi_{n1 j} over run `run` (see the j table below).
__device__ __forceinline__ u32 mid_run(u32 run, u32 g, u32 lr, u32 N) {
    const u32 E = ((g * (2 * (__brev(run) >> (32 - lr)) + 1) - 1) >> 1) & (N - 1);
    return __brev(E & ((1u << lr) - 1)) >> (32 - lr);
}

// Bytes of one stage: K3 diagonal blocks | beta digit runs | A run | key block (B run at j = 0).
__host__ __device__ inline u32 ws_stage(bool packed, u32 k3, u32 beta, u32 beta_max) {
    const u32 kb = beta ? key_blk(packed, beta, beta_max) : 0;
    return k3 * diag_blk(packed) + (beta + 1) * BLK * 8 + (kb > BLK * 8 ? kb : BLK * 8);
}

// Packed and wide limbs are two launches: each class has the registers and the
// CTAs per SM that suit its body (K3 = 4: 96 registers and four CTAs, or 128
// and three), and neither keeps the other's code (one kernel for both: 1.86 ms
// at (1,64,4), Set-A 1.09; split: 1.78 and 1.03).  The wide limbs go first and
// the packed ones are launched early behind them (they read nothing that the
// first launch writes); `join` makes the last CTA wait, at its end, for the
// launch before, so that a kernel that waits for this one has both.
// ring: bytes of dynamic shared memory for the stages; the j table follows.
template <int K3, int BETA, int MINB, bool PACKED>
__global__ void __launch_bounds__(WS_THREADS, MINB) k_diag_mac_ws(const __grid_constant__ DiagMacArgs a, u32 ring,
                                                                 bool join) {
    constexpr u32 RB = BLK * 8;  // bytes of a run of words
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) u64 full_bar[WS_MAX_STAGES];
    __shared__ __align__(8) u64 empty_bar[WS_MAX_STAGES];
    __shared__ u32 abort_flag;
    const u32 N = 1u << a.log_n;
    const u32 l = threadIdx.x;
    const u32 bidx = blockIdx.x % a.batch;
    const u32 run = blockIdx.x / a.batch;
    const size_t ou = bidx * a.bs_u;
    const u32 t = a.limbs[PACKED ? blockIdx.y : a.n_packed + blockIdx.y];
    const u32 k_first = blockIdx.z * K3;
    const u32 k_count = min((u32)K3, a.n3 - k_first);
    const u32 gmod = t < a.level ? t : a.L + (t - a.level);
    const ModC m = a.mods[gmod];
    constexpr bool packed = PACKED;
    const size_t tN = (size_t)t * N;
    const u32 n1 = a.n1, n2 = a.n2, n1n2 = n1 * n2;
    const u32 beta = BETA == WS_ANY ? a.beta : BETA;  // a.beta, or 0 without a middle layer
    const u32 fb = diag_blk(packed);
    const u32 kb = beta ? key_blk(packed, beta, a.beta_max) : 0;
    const u32 off_dig = K3 * fb, off_a = off_dig + beta * RB, off_key = off_a + RB;
    const u32 stage = ws_stage(packed, K3, beta, a.beta_max);
    const u32 ns = min(WS_MAX_STAGES, ring / stage);
    const bool lift_limb = a.lift0 && t < a.level;
    // Per middle index j, the gather of phi_{n1 j} over this run: word l of the
    // run reads word brv_7(C + g brv_7(l) mod 128) of run srun, where with
    // R = brv(run), E = (g (2R + 1) - 1) / 2 mod N: C is E's top 7 bits and
    // srun the bit reversal of the rest (Eq. 7 split at the run boundary).
    u32* jtab = (u32*)(smem + ring);
    const u32 lr = a.log_n - 7;
    for (u32 jj = l; jj < n2; jj += WS_THREADS) {
        const u32 g = jj ? a.gal_mid[jj] : 1u;
        const u32 R = __brev(run) >> (32 - lr);
        const u32 E = ((g * (2 * R + 1) - 1) >> 1) & (N - 1);
        jtab[jj] = mid_run(run, g, lr, N) | ((E >> lr) << 16) | ((g & 127u) << 24);
    }
    if (l == 0) {
        for (u32 b = 0; b < ns; b++) {
            mbar_init(&full_bar[b], 1);
            mbar_init(&empty_bar[b], BLK / 32);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (!join) pdl_wait();
    else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    volatile u32* abort = &abort_flag;

    if (l >= BLK) {
        // ------------------------------------------------------------ producer warp
        // Copies are issued by one thread, one after another.  A bulk copy takes
        // its operands from uniform registers: spread over the lanes of a warp,
        // copies are issued one lane at a time by a loop that moves each lane's
        // operands there, and in a loop that one thread runs every operand is
        // moved; only where the whole warp runs the loop and an elected lane
        // issues are the addresses uniform to begin with.  That is what the wide
        // limbs do, whose stages were bound by it (Set-A, ten copies a step: 1.03
        // -> 0.93 ms, Set-B 0.65 -> 0.63).  The packed limbs at N = 2^16, bound
        // by arithmetic, lost time to it (1.78 -> 1.90 ms) and keep one thread.
        u32 issued = 0;
        const bool leader = PACKED ? l == BLK : elect_one();
        if (!PACKED || leader) {
            const unsigned char* fsrc[K3];  // the next step's diagonal blocks
#pragma unroll
            for (int kk = 0; kk < K3; kk++) {
                const u32 kc = k_first + min((u32)kk, k_count - 1), g = a.gal_diag[kc];
                const u32 hrun = (g ? auto_src(run * BLK, g, a.log_n) : run * BLK) / BLK;
                fsrc[kk] = a.diags + (size_t)(n1n2 * kc) * a.diag_stride + m.doff + (t < a.level ? 0 : a.diag_p) +
                           (size_t)hrun * fb;
            }
            const size_t koff = m.koff + (size_t)run * key_blk(packed, a.beta_max, a.beta_max);
            const u32 group = a.slots * BLK;  // words from one block's group of slots to the next
            const size_t ox = bidx * a.bs_x + (size_t)t * (N / BLK) * group;
            u32 sidx = 0, phase = 1, i = 0, j = 0, srun = run;
            for (u32 it = 0; it < n1n2; it++) {
                // every compute warp has read step it - ns, or giving up
                if (it >= ns) {
                    bool ok = mbar_wait_abortable(&empty_bar[sidx], phase, DM_WAIT_NS, abort);
                    if (!PACKED) ok = __all_sync(0xffffffffu, ok);
                    if (!ok) {
                        *abort = 1u;
                        break;
                    }
                }
                issued = it + 1;
                if (it != a.starve_step) {  // test hook: this step is never issued
                    const bool copy_a = i > 0 || !a.lift0 || lift_limb;
                    unsigned char* st = smem + sidx * stage;
                    u64* bar = &full_bar[sidx];
                    const u32 xb = (beta + (copy_a ? 1 : 0)) * RB;  // digits and A
                    const u64* X = a.X[i] + ox + (size_t)(PACKED ? jtab[j] & 0xFFFFu : srun) * group;
                    const u64* B = (i || !a.lift0 ? a.B[i] + bidx * a.bs_b : a.c1[bidx]) + tN + (size_t)run * BLK;
                    const unsigned char* K = a.keys[j] + koff;
                    if (PACKED || leader) {
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                        mbar_expect_tx(bar, k_count * fb + (j ? xb + kb : (copy_a ? 2 * RB : 0)));
#pragma unroll
                        for (int kk = 0; kk < K3; kk++)
                            if (kk < (int)k_count) tma_load_1d(st + kk * fb, fsrc[kk], fb, bar);
                        if (j) {
                            tma_load_1d(st + off_dig, X, xb, bar);
                            tma_load_1d(st + off_key, K, kb, bar);
                        } else if (copy_a) {
                            tma_load_1d(st + off_a, X + group - BLK, RB, bar);
                            tma_load_1d(st + off_key, B, RB, bar);
                        }
                    }
                }
#pragma unroll
                for (int kk = 0; kk < K3; kk++) fsrc[kk] += a.diag_stride;
                if (++sidx == ns) sidx = 0, phase ^= 1;
                if (++i == n1) {
                    i = 0;
                    if (++j < n2 && !PACKED) srun = mid_run(run, a.gal_mid[j], lr, N);
                }
            }
        }
        __syncwarp();
        nbar_sync(1, WS_THREADS);  // every thread of the CTA reaches this once
        if (join && blockIdx.x + 1 == gridDim.x && blockIdx.y + 1 == gridDim.y && blockIdx.z + 1 == gridDim.z) pdl_wait();
        if (*abort && leader) {
            // drain: the last phase issued into each stage (the earlier ones completed and were consumed)
            for (u32 it = issued > ns ? issued - ns : 0; it < issued; it++)
                if (it != a.starve_step) mbar_wait_bounded(&full_bar[it % ns], (it / ns) & 1);
            atomicExch(a.err, 1u);
        }
        return;
    }

    // ---------------------------------------------------------------- compute threads
    const u32 s = run * BLK + l;
    const u64 lc = lift_limb ? a.lift_c[gmod] : 0, lsh = lift_limb ? a.lift_sh[gmod] : 0;
    const WsCtx c{a, smem, full_bar, empty_bar, abort, jtab, s, l, k_first, k_count, ns, stage, off_a,
                  ou + tN + s, lift_limb, lc, lsh, m};
    if constexpr (PACKED) {
        ws_compute<K3, BETA, C40>(c);
    } else {
        if (m.bits <= 55) ws_compute<K3, BETA, C55>(c);
        else ws_compute<K3, BETA, C60>(c);
    }
}

// Launches k_diag_mac_ws on one class of limbs, with the ring that MINB CTAs
// per SM leave room for; false if two stages do not fit, so that the plain
// kernel runs.  The dynamic shared-memory limit is a per-device function
// attribute: set once per device (threads may race to set it; the call is
// idempotent).  A device that refuses it falls back too, and the error the
// refusal left is cleared so that a later status check does not see it.
constexpr u32 SM_SMEM = 227 * 1024;

template <int K3, int BETA, int MINB, bool PACKED>
bool try_ws(const DiagMacArgs& a, bool join, cudaStream_t st) {
    const u32 beta = BETA == WS_ANY ? a.beta : BETA;
    const u32 N = 1u << a.log_n;
    // one CTA's share, less the 1 KB that the system takes per CTA and the static
    // barriers: of MINB CTAs, or of fewer where two stages need it, for a long j
    // table or a key block with the high bytes of many more digits.  Eight digits,
    // wide, (1,400,2) at N = 2^12 with three CTAs: 358 us, 887 by the plain kernel;
    // packed, of 36, (1,16,4) at 2^14: 74 and 95; of 128, (1,8,4) at 2^12 with two:
    // 23.2 and 25.3.  One CTA is slower than the plain kernel (of 160: 28.5 and
    // 25.0), but past eight digits, whose every stage is large, it is not (see WS_ANY)
    const u32 tab = (4 * a.n2 + 15) & ~15u;
    constexpr int MIN_CTAS = BETA == WS_ANY ? 1 : 2;
    u32 ring = 0;
    for (int ctas = MINB; ctas >= MIN_CTAS; ctas--) {
        const u32 share = SM_SMEM / ctas - 1024 - 256;
        if (tab >= share) continue;
        ring = (share - tab) & ~127u;
        if (ring >= 2 * ws_stage(PACKED, K3, beta, a.beta_max)) break;
        ring = 0;
    }
    if (!ring) return false;
    static std::atomic<uint64_t> attr_set{0}, attr_bad{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return false;
    }
    const uint64_t bit = 1ull << dev;
    if (attr_bad.load(std::memory_order_relaxed) & bit) return false;
    if (!(attr_set.load(std::memory_order_acquire) & bit)) {
        if (cudaFuncSetAttribute(k_diag_mac_ws<K3, BETA, MINB, PACKED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(SM_SMEM / MIN_CTAS - 1024 - 256)) != cudaSuccess) {
            cudaGetLastError();
            attr_bad.fetch_or(bit, std::memory_order_relaxed);
            return false;
        }
        attr_set.fetch_or(bit, std::memory_order_release);
    }
    const dim3 grid((N / BLK) * a.batch, PACKED ? a.n_packed : a.ext - a.n_packed, (a.n3 + K3 - 1) / K3);
    launch(join, k_diag_mac_ws<K3, BETA, MINB, PACKED>, grid, WS_THREADS, ring + tab, st, a, ring, join);
    return true;
}

}  // namespace

// CTAs per SM.  More CTAs are more warps and more independent rings, as long as
// the body keeps its registers.  Four outer indices at N = 2^16 (1,64,4), packed:
// 1.87 ms with four CTAs, 2.17 with five; eight at N = 2^15 (1,12,8): 154 us with
// three, 169 with two.  The wide limbs' body takes more: 54-bit moduli, eight
// outer indices, 0.67 ms with two, 0.78 with three; at N = 2^16 (four) 1.87 with
// three for them and 1.89 with four.
template <int K3, bool PACKED>
bool launch_ws(const DiagMacArgs& a, bool join, cudaStream_t st) {
    constexpr int MINB = K3 >= 8 ? (PACKED ? 3 : 2) : K3 == 4 && !PACKED ? 3 : 4;
    switch (a.n2 == 1 ? 0 : a.beta) {
        case 0: return try_ws<K3, 0, MINB, PACKED>(a, join, st);
        case 1: return try_ws<K3, 1, MINB, PACKED>(a, join, st);
        case 2: return try_ws<K3, 2, MINB, PACKED>(a, join, st);
        case 3: return try_ws<K3, 3, MINB, PACKED>(a, join, st);
        case 4: return try_ws<K3, 4, MINB, PACKED>(a, join, st);
        case 5: return try_ws<K3, 5, MINB, PACKED>(a, join, st);
        case 6: return try_ws<K3, 6, MINB, PACKED>(a, join, st);
        case 7: return try_ws<K3, 7, MINB, PACKED>(a, join, st);
        case 8: return try_ws<K3, 8, MINB, PACKED>(a, join, st);
        default: return try_ws<K3, WS_ANY, 2, PACKED>(a, join, st);
    }
}

}  // namespace ckks
