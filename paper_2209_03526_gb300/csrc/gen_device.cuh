// gen_device.cuh -- DPF / DCF Gen of one key pair on the device, for the batched key
// generation kernels.  The construction is the host's (BGI16 tree DPF, Boyle et al. DCF;
// H_K(s) = AES_K(s) xor s under the fixed keys, control bit = bit 0 of byte 0 of a child
// seed, Convert = bytes 4..7 of a seed / bytes 0..3 of a value block, input bits MSB
// first).  The correction words go to a Sink, which decides the key layout:
//   sink.level(lv, scw[4], tl, tr, vcw)   level lv = 0..n-1 (vcw only for DCF)
//   sink.final(cw)                        CW_{n+1}
#pragma once

#include <cstdint>

#include "device_fss.cuh"

namespace ogm {

// b - a for a of the pair's party 0 and b of its party 1, from this lane's own value
__device__ __forceinline__ uint32_t party_diff(uint32_t own, uint32_t party) {
    const uint32_t d = __shfl_xor_sync(0xFFFFFFFFu, own, 1) - own;
    return party ? 0u - d : d;
}

// Gen of f^=_{alpha,beta} (DCF = false) or g^<_{alpha,beta} (DCF = true) over Z_{2^32} on a
// pair of lanes: the even lane expands party 0's seeds (root s), the odd lane party 1's, and
// the lose children, control bits and value words meet by shuffles and ballots.  The whole
// warp takes part.  The shared-memory lookups bound it (616 per lane and DCF level).  A thread
// per pair had eight AES bodies in a row, 16 warps per SM and twice the work in its smallest
// unit; with both sides unrolled the lane pairs are slower than that (1.91 ms below), the code
// being larger than the instruction cache.  50,000 elements' fresh tokens 1.71 -> 1.62 ms,
// 1,000 elements 0.28 -> 0.12 ms, 1,000 DCF pairs 0.16 -> 0.07 ms.
template <bool DCF, class Sink>
__device__ __forceinline__ void gen_pair(const SmemTab& T, const AesParams& A, int n, uint32_t alpha, uint32_t beta,
                                         uint32_t party, uint32_t s[4], Sink& sink) {
    const uint32_t other = (threadIdx.x & 31u) ^ 1u;
    uint32_t t = party, valpha = 0u;
#pragma unroll 1
    for (int lv = 1; lv <= n; lv++) {
        const uint32_t a = (alpha >> (n - lv)) & 1u;
        uint32_t scw[4], keep[4], tc[2], dv[2];            // tc, dv: lose, keep
#pragma unroll 1
        for (int side = 0; side < 2; side++) {
            const uint32_t m = 0u - (side ? a : a ^ 1u);
            uint32_t c[4], v = 0u;
            aes_sel(T, A.rk_st, A.d_st, m, s, c);
            if (DCF) v = aes_sel_w0(T, A.rk_v, A.d_v, m, s) ^ s[0];
#pragma unroll
            for (int w = 0; w < 4; w++) c[w] ^= s[w];
            if (side == 0) {
                tc[0] = c[0] & 1u;
                c[0] &= ~1u;
#pragma unroll
                for (int w = 0; w < 4; w++) scw[w] = c[w] ^ __shfl_xor_sync(0xFFFFFFFFu, c[w], 1);
                if (DCF) dv[0] = party_diff(v, party);
            } else {
                tc[1] = c[0] & 1u;
                c[0] &= ~1u;
#pragma unroll
                for (int w = 0; w < 4; w++) keep[w] = c[w];
                if (DCF) dv[1] = party_diff(v, party);
            }
        }
        // control-bit words of the lose and the keep side: the sides' bits differ only in a
        const uint32_t t_lose = tc[0] ^ ((__ballot_sync(0xFFFFFFFFu, tc[0]) >> other) & 1u);
        const uint32_t t_keep = tc[1] ^ ((__ballot_sync(0xFFFFFFFFu, tc[1]) >> other) & 1u) ^ 1u;
        uint32_t vcw = 0u;
        if (DCF) {
            const bool neg = (t ^ party ^ 1u) != 0;        // party 1's bit: the two differ on alpha's path
            vcw = dv[0] - valpha;
            if (neg) vcw = 0u - vcw;
            if (a) vcw += neg ? 0u - beta : beta;          // lose side is L: inputs below alpha
            valpha = valpha - dv[1] + (neg ? 0u - vcw : vcw);
        }
        sink.level(lv - 1, scw, a ? t_lose : t_keep, a ? t_keep : t_lose, vcw);
        const uint32_t m = 0u - t;
#pragma unroll
        for (int w = 0; w < 4; w++) s[w] = keep[w] ^ (scw[w] & m);
        t = tc[1] ^ (t & t_keep);
    }
    const uint32_t d = party_diff(s[1], party);
    uint32_t cw = DCF ? d - valpha : beta + d;
    if (t ^ party ^ 1u) cw = 0u - cw;
    sink.final(cw);
}

}  // namespace ogm
