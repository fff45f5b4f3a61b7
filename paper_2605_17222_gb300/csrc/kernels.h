// Kernel launch interface shared by the .cu files of the library (internal).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "modarith.cuh"

namespace ckks {

// ------------------------------------------------------------------ launches
// With `early`, a kernel is launched with programmatic stream serialisation:
// its launch, its parameters and what it loads from the context's constant
// tables overlap the end of the kernel before it, and pdl_wait() holds it
// before it touches memory that an earlier kernel wrote (or that it
// overwrites).  pdl_wait() returns when the kernel before it is complete and
// its writes are visible; every CTA of an evaluation's kernels calls it, so all
// earlier ones are complete too.  The exception is the packed diagonal kernel
// behind a wide one: it starts early, and only its last CTA waits, at its end
// (diag_mac.cuh).  That is sound because the wide launch is never early (what
// both read was complete when it started) and that CTA keeps the packed grid
// from completing before the wide one.  Who launches early was measured kernel by
// kernel: the second pass of each transform and the gathers always (N = 2^14
// BSGS 1.92 -> 1.70 ms, N = 2^16 level 9 708 -> 689 us); the inverse row pass
// in small grids (1.70 -> 1.61); the forward column pass, the key products and
// the diagonal kernel not, whose early CTAs only share SMs with the kernel
// before (everything early: Set-A 1.48 ms against 1.38).
constexpr u32 SMS = 152;  // of a GB300
template <typename... P, typename... A>
inline void launch(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);  // an error stays for the caller's status check
}
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------------------------ layout of keys and diagonals
// Switching keys and diagonals are what an LT streams from HBM, so the library
// stores them at 5 bytes a word where the modulus allows it (2^32 < q < 2^40:
// 23 of the 28 limbs of the N = 2^16 workload, 31% fewer bytes) and at 8 bytes
// otherwise.  A limb is stored in blocks of BLK = 128 consecutive words, the
// unit that every automorphism maps onto one block (Eq. 8), so that one bulk
// copy fetches a block:
//   diagonals : packed  [128 x u32 low words][128 x u8 high bytes], 640 bytes
//               wide    [128 x u64], 1024 bytes
//   keys      : packed  [128 x key_hi bytes: the high bytes of (component 0, component 1) per digit]
//                       [beta_max][128 x (u32, u32) low words]
//               wide    [beta_max][128 x (u64, u64)]
// A level with beta < beta_max digits reads a prefix of a key block.
constexpr u32 BLK = 128;
__host__ __device__ inline bool packed_q(u64 q) { return q > (1ull << 32) && q < (1ull << 40); }
__host__ __device__ inline u32 diag_blk(bool packed) { return packed ? BLK * 5 : BLK * 8; }
__host__ __device__ inline u32 key_hi(u32 beta_max) { return (2 * beta_max + 3) & ~3u; }  // bytes per position
// bytes of the first beta digits of a key block (beta = beta_max: of the block)
__host__ __device__ inline u32 key_blk(bool packed, u32 beta, u32 beta_max) {
    return packed ? BLK * (key_hi(beta_max) + 8 * beta) : BLK * 16 * beta;
}
// Words [rows][N] -> packed or wide limbs, reduced on the way, so that any word
// of the residue class is taken.
struct PackArgs {
    const u64* in;
    unsigned char* out;
    const ModC* mods;
    u32 level, L, k, beta_max, log_n;  // diagonals: Q limbs stored; keys: beta_max
    u64 p_base, stride;                // diagonals: offset of the P limbs, bytes per diagonal
};
void launch_pack_diags(const PackArgs& a, u32 count, cudaStream_t st);
void launch_pack_key(const PackArgs& a, cudaStream_t st);

// Per-context device tables every NTT kernel reads.
struct NttTables {
    const ModC* mods;          // [n_mod] {q, mu}
    const ulonglong2* psi;     // [n_mod][N] (psi^brv(i), Shoup companion)
    const ulonglong2* ipsi;    // [n_mod][N] (psi^-brv(i), Shoup companion)
    u32 log_n;
};

// One limb of a forward NTT.
//   pass 1 load : nsrc == 0 -> src[x];
//                 nsrc  > 0 -> sum_j src[j*N + x] * bcst[j] mod q   (basis conversion, Eq. 3)
//                 (bits 0-15: the source count; bit 16: every source word is
//                 below 2^40, which with a packed_q target allows 40-bit sums)
//   pass 2 store: subx == nullptr -> dst[x] = X;
//                 otherwise dst[x] = (subx[x] - X) * c mod q          (ModDown tail, Eq. 4)
// Pass 1 writes dst; pass 2 runs in place on dst.  subx is a plain limb.
// FwdJob::nsrc bit 17: a copy job, dst[x] = src[x -> x^gal] with gal in c
// (0: plain copy) and no transform, for the limbs a Decompose passes through
// unchanged; it rides in the same launch as the transforms.
// Bit 18 (with bit 17): a scaling job instead, dst[x] = src[x] * c mod q
// (c_sh its Shoup companion), e.g. the lift P c0 of Alg. 2 line 2.
// Bits 19..31: the blocks of BLK words from one of dst's blocks to the next
// (0: 1, a plain limb), for limbs that are slots of grouped blocks (DigLayout).
constexpr u32 FWD_COPY = 1u << 17;
constexpr u32 FWD_SCALE = 1u << 18;
constexpr u32 FWD_STEP = 19;
struct FwdJob {
    const u64* src;
    u64* dst;
    const u64* bcst;
    const u64* subx;
    u64 c, c_sh;
    u32 mod;
    u32 nsrc;
};

// One limb of an inverse NTT: pass A reads src (gathered through x -> x^gal
// when gal != 0) and writes tmp; pass B reads tmp and writes dst scaled by c
// (c includes N^-1).  tmp may alias dst; src may alias tmp only when gal == 0.
struct InvJob {
    const u64* src;
    u64* tmp;
    u64* dst;
    u64 c, c_sh;
    u32 mod;
    u32 gal;
};

// An inverse transform with a basis conversion taken off on the way out:
// dst[x] = X[x] * c - (sum_i csrc[i*N + x] * bcst[i]) * c2 mod q, i < nsrc,
// X the unscaled inverse.  A ModDown that feeds a Decompose (Alg. 2 lines 6-7
// and 15-16) needs the coefficients of (x - conv) P^-1, and
// INTT(x - NTT(conv)) = INTT(x) - conv.
struct InvConvJob : InvJob {
    const u64* csrc;
    const u64* bcst;
    u64 c2, c2_sh;
    u32 nsrc;
    u32 pad;
};
// The inverse transforms of `sub` after those of `first`, whose outputs are the
// sub jobs' csrc; their row passes are one launch.
void launch_inv_conv(const NttTables& T, const InvJob* first, int nfirst, const InvConvJob* sub, int nsub, cudaStream_t st);

void launch_fwd_ntt(const NttTables& T, const FwdJob* jobs, int njobs, cudaStream_t st);
void launch_inv_ntt(const NttTables& T, const InvJob* jobs, int njobs, cudaStream_t st);

// out[l][s] = in[l][src_g(s)] for n_limbs limbs (NTT-domain automorphism, Eq. 7).
void launch_automorphism(const u64* in, u64* out, u32 n_limbs, u32 gal, u32 log_n, cudaStream_t st);

// out[s] = a[src_gal(s)] + b[s] mod q, per limb.
struct AddJob {
    const u64* a;
    const u64* b;
    u64* out;
    u32 mod;
    u32 gal;
};
void launch_add_gather(const ModC* mods, const AddJob* jobs, int njobs, u32 log_n, cudaStream_t st);

// The giant steps' sum of BSGS: acc0[t][s] += sum_k a_k[t][src_{g_k}(s)] + b0_k[t][s] and
// acc1[t][s] += sum_k b1_k[t][s] mod q_t, over `level` Q limbs, k < count.
constexpr int SUM_MAX = 64;
struct SumArgs {
    const u64 *a[SUM_MAX], *b0[SUM_MAX], *b1[SUM_MAX];
    u32 gal[SUM_MAX];
    u64 *acc0, *acc1;
    const ModC* mods;
    u32 count, level, log_n;
};
void launch_sum_gather(const SumArgs& a, cudaStream_t st);

// Where word x of digit b of limb t lies: t limb + (x / BLK) blk + b dig + x % BLK.
// Plain digits [beta][ext][N], or grouped [ext][N/BLK][slots][BLK]: the slots
// of one block side by side, so that the diagonal kernel fetches every digit
// of a run (and the A run, the last slot) with one bulk copy.
struct DigLayout {
    u64 limb, blk, dig;
};
inline DigLayout plain_digits(u32 ext, u32 log_n) { return {1ull << log_n, BLK, (u64)ext << log_n}; }
inline DigLayout grouped_digits(u32 slots, u32 log_n) { return {(u64)slots << log_n, (u64)slots * BLK, BLK}; }

// Switching-key inner products with hoisted automorphism (K4): for product e
//   P_{e,c} = phi_g(x0_e) (c = 0 only) + <phi_g(d_e), swk_{e,c}>
// x0_mode 0: no x0; 1: an extended polynomial; 2: a Q polynomial lifted to P x0.
// sum = 0: out_{e,c} = P_{e,c}, added to what out holds if accumulate (one
// launch for many independent products; neighbours in the grid take the same
// run of positions, so entries that share a key read it once).
// sum = 1: out_{0,c} += sum_e P_{e,c}, the outer key-switch layer of Algorithm
// 2 (lines 17-18) for every giant index at once.
constexpr int KS_MAX = 32;  // 1.5 KB of kernel parameters: every launch copies them
struct KsItem {
    const u64* digits;         // dl
    const unsigned char* key;  // layout above
    const u64* x0;
    u64* out0;                 // o_limb, o_blk: its limb and block strides
    u64* out1;                 // plain
    u32 gal;
    u32 pad;
};
struct KsArgs {
    KsItem e[KS_MAX];
    const ModC* mods;  // context moduli (index = global modulus id)
    const u64* lift_c; // [L+k] [P]_{q_j} (0 for P moduli) and Shoup companions
    const u64* lift_sh;
    u32* err;          // set to nonzero when a bounded device wait gives up
    DigLayout dl;
    u64 o_limb, o_blk;
    u32 count, sum, x0_mode, accumulate, level, ext, L, beta, beta_max, log_n;
};
void launch_ks(const KsArgs& a, cudaStream_t st);

// Multi-output plaintext-diagonal multiply-accumulate with the middle
// (hoisted) key-switch layer fused in (K6).  See ks.cu.
constexpr int DM_MAX_N1 = 64;
constexpr int DM_MAX_N2 = 1024;
constexpr int DM_MAX_K3 = 8;   // giant indices per thread (grid.z covers the rest)
constexpr int DM_MAX_N3 = 64;
constexpr int DM_MAX_LIMBS = 256;
constexpr int DM_MAX_B = 16;   // ciphertexts per batched launch
struct DiagMacArgs {
    const ModC* mods;
    const u64* lift_c;
    const u64* lift_sh;
    const unsigned char* diags;  // [n_diag] of diag_stride bytes, the P limbs at diag_p
    u64 diag_stride, diag_p;
    const u64* X[DM_MAX_N1];         // per baby index: its digits and A_i, [ext][N/BLK][slots][BLK], A_i the last slot
    const u64* B[DM_MAX_N1];         // B_i [ext][N] (i = 0 with lift0: c1 below)
    const unsigned char* keys[DM_MAX_N2];  // middle-layer keys, index j (j >= 1)
    u32 gal_mid[DM_MAX_N2];          // x -> x^gal for rotation n1*j*stride
    u64* U0[DM_MAX_N3];
    u64* U1[DM_MAX_N3];
    u32 gal_diag[DM_MAX_N3];         // rotation -(n1*n2*k*stride), 0 = none
    u32 level, ext, L, k_p, beta, beta_max, log_n;
    u32 n1, n2, n3;
    u32 slots;                       // beta + 1, or 1 without a middle layer (n2 = 1)
    // 1: (A_0, B_0) is the lifted input P (c0, c1) (Alg. 2 line 2), zero on
    // the P limbs; X[0] holds P c0 on the Q limbs, c1 is lifted here
    u32 lift0;
    u32* err;                        // set to nonzero when a bounded device wait gives up
    // Failure-detection test hook of the staged kernel: the step loop's
    // waits give up after wait_ns (0: the default of one second), and step
    // starve_step (~0u: none) is never issued, so that its wait runs out.
    // The drain of copies in flight always keeps the default limit.
    u64 wait_ns;
    u32 starve_step;
    // Tile (0 = default): outer indices per CTA, a power of two below the
    // next power of two >= n3, at most 8.  Results do not depend on it.
    u32 tile_k3;
    // the limbs t < ext: the packed_q ones, then the wide ones (a basis of more
    // than DM_MAX_LIMBS runs the plain kernel over every limb)
    u32 n_packed;
    unsigned char limbs[DM_MAX_LIMBS];
    // Batch of ciphertexts sharing the diagonals and keys: ciphertext b uses
    // X[i] + b*bs_x, B[i] + b*bs_b, c1[b] and U0/U1[k] + b*bs_u.  CTAs of the
    // same (limb, run) for different b are adjacent in the grid, so the
    // diagonal and key words they share are read from HBM once.
    u32 batch;
    u64 bs_x, bs_b, bs_u;
    const u64* c1[DM_MAX_B];
};
void launch_diag_mac(const DiagMacArgs& a, cudaStream_t st);
// Its staged kernel on the packed or the wide limbs, K3 (1, 2, 4 or 8) outer
// indices per CTA, or false if a shape does not fit (diag_mac.cuh).
template <int K3, bool PACKED>
bool launch_ws(const DiagMacArgs& a, bool join, cudaStream_t st);
void launch_wait_selftest(u32* err, u64 limit_ns, cudaStream_t st);

uint64_t launches();
void count_launch(int n = 1);

// Kernel classes for live timing (ckks_profile_*).
enum KClass { K_DIAG_MAC = 0, K_KS_INNER, K_FWD_COLS, K_FWD_ROWS, K_INV_ROWS, K_INV_COLS, K_AUTO, K_ADD, K_NCLASS };
extern const char* const kclass_names[K_NCLASS];
bool prof_on(int cls);
// Brackets one launch with events when its class is enabled, and adds the
// launch's algorithmic integer work (128-bit multiply-accumulates, NTT
// butterflies) to the class's totals.
struct ProfScope {
    int cls;
    cudaStream_t st;
    void* ev;
    ProfScope(int c, cudaStream_t s, double macs = 0, double butterflies = 0);
    ~ProfScope();
};
int prof_class(const char* name);
void prof_enable(int cls, bool on);
bool prof_read(int cls, double* ms, uint64_t* n);
bool prof_work(int cls, double* macs, double* butterflies);
void prof_reset();

// Register-only rate probes of the library's own 128-bit multiply-accumulate
// and forward NTT butterfly over `blocks` CTAs (best of two timed runs after a
// warm-up); synchronous, on a stream of its own.
cudaError_t probe_int_rates(u32 blocks, double* macs_per_s, double* butterflies_per_s);

}  // namespace ckks
