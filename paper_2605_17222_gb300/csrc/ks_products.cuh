// Key-switching products of one position over any number of digits.
#pragma once
#include "kernels.h"

namespace ckks {

// v_c += sum_b d_b k_{b,c}, b < beta, for position l of a key block K (digits
// dstep words apart; global or shared memory), the result in [0, 3q) (PACKED)
// or [0, 5q).  Four digits between two reductions; the loads of a group have no
// branch between them (a digit past the last re-reads it and counts as zero),
// so that they are issued together.
template <bool PACKED>
__device__ __forceinline__ void ks_products(const ModC& m, const u64* D, size_t dstep, const unsigned char* K, u32 l,
                                            u32 beta, u32 beta_max, u64& v0, u64& v1) {
    constexpr u32 G = 4;
    const u32 hb = key_hi(beta_max);
    for (u32 b0 = 0; b0 < beta; b0 += G) {
        u64 d[G];
        u32 c[G];
#pragma unroll
        for (u32 j = 0; j < G; j++) {
            c[j] = min(b0 + j, beta - 1);
            d[j] = D[c[j] * dstep];
        }
        if constexpr (PACKED) {
            const uint2* lp = (const uint2*)(K + BLK * hb) + l;
            const unsigned short* hp = (const unsigned short*)(K + l * hb);
            uint2 k[G];
            u32 h[G];
#pragma unroll
            for (u32 j = 0; j < G; j++) k[j] = lp[c[j] * BLK], h[j] = hp[c[j]];
            Sum40 s0, s1;
#pragma unroll
            for (u32 j = 0; j < G; j++) {
                u32 dl, dh;
                split20(b0 + j < beta ? d[j] : 0, dl, dh);
                s0.mac(dl, dh, k[j].x, h[j] & 0xFFu);
                s1.mac(dl, dh, k[j].y, h[j] >> 8);
            }
            v0 = s0.value(v0, m.q, (u32)m.mu_hi);
            v1 = s1.value(v1, m.q, (u32)m.mu_hi);
        } else {
            const ulonglong2* kp = (const ulonglong2*)K + l;
            ulonglong2 k[G];
#pragma unroll
            for (u32 j = 0; j < G; j++) k[j] = kp[c[j] * BLK];
            Sum60 s0, s1;
#pragma unroll
            for (u32 j = 0; j < G; j++) {
                u32 dl, dh, kl, kh;
                split30(b0 + j < beta ? d[j] : 0, dl, dh);
                split30(k[j].x, kl, kh);
                s0.mac(dl, dh, kl, kh);
                split30(k[j].y, kl, kh);
                s1.mac(dl, dh, kl, kh);
            }
            v0 = s0.value(v0, m);
            v1 = s1.value(v1, m);
        }
    }
}

}  // namespace ckks
