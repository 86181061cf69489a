// Check-node pass that loads its operands straight into registers, for codes
// whose rows all have an exact shape (flooding with accumulated posteriors).
//
// A warp owns 32 SLOTS consecutive checks of one base row and frame, lane l the
// checks l, l + 32, ...; every load, store and reduction of a warp is then one
// contiguous 128-byte run. Pairs of a lane's checks are evaluated in packed
// FP32x2 arithmetic, bit for bit as in the staged pass (check_pass.cuh), and
// the next pair's operands are loaded before a pair computes. Warps share
// nothing but one flag, so no warp waits at a barrier for a serial copy set-up,
// and there is no shared-memory round trip. Bounded by the latency of its loads
// and by instruction issue: 16 frames of n = 10^6, FP32, took 102.7 us a pass
// staged and take 89.5 us, FP16 90.9 and 83.7 (replayed alone). Without the
// loads ahead 8 checks per lane took 103 us, and 256-thread blocks 100.6.
// Registers: 72 (7 blocks of 128 threads), where the FP32 form with 8 checks per
// lane spills 148 bytes a thread. 64 spill 748; 80, the first without a spill,
// leave too few warps: 85.8, 86.9 and 93.1 us an iteration of 16 frames at 64, 72
// and 80, and 30.7, 26.7 and 26.2 of 5 frames.
#pragma once

#include "decode_common.cuh"

namespace {

template <typename M>
__device__ __forceinline__ M ld_msg(const M *p) { return __ldcg(p); }
template <>
__device__ __forceinline__ int8_t ld_msg<int8_t>(const int8_t *p) {
    return (int8_t)__ldcg(reinterpret_cast<const signed char *>(p));
}

// Operands of two checks (32 apart) of one lane.
template <int NH, int ND, typename M>
struct PairOps {
    float2 lv[NH > 0 ? NH : 1], ph[ND > 0 ? ND : 1];
    M ma[NH > 0 ? NH : 1], mb[NH > 0 ? NH : 1];
    uint32_t da[ND > 0 ? ND : 1], db[ND > 0 ? ND : 1];
};

// The checks wb .. wb + 32 SLOTS - 1 of row r (first entry rp), frame f; returns
// whether one of the lane's checks fails the stop test of iteration t - 1.
template <int NH, int ND, int MODE, typename M, int SLOTS, bool SOFT>
__device__ __forceinline__ bool cd_row(const Table &T, const Work &W, int f, int r, int rp, int t, const int *oa,
                                       const int *ob, int wb) {
    static_assert(SLOTS % 2 == 0, "checks are evaluated in pairs");
    constexpr int D = NH + ND;
    constexpr int NHa = NH > 0 ? NH : 1;
    constexpr int NDa = ND > 0 ? ND : 1;
    constexpr bool kUpdate = MODE != kTestOnly;
    constexpr bool kReadMsg = MODE == kSteady || MODE == kSteadyTest;
    constexpr bool kTest = MODE == kSteadyTest || MODE == kTestOnly;
    constexpr bool kSyn = !syn_folded(ND);
    const int Z = T.Z;
    const int lane = threadIdx.x & 31;
    const int i0 = wb + lane;
    const float *pL[NHa], *pP[NDa];
    int32_t *pA[NHa];
    M *pM[NHa];
    const uint32_t *pB[NDa];
    uint32_t *pC[NDa];
#pragma unroll
    for (int k = 0; k < NH; k++) {
        pL[k] = W.L + ((size_t)f * W.col_f + (uint32_t)(oa[k] + i0));
        pA[k] = W.acc + ((size_t)f * W.col_f + (uint32_t)(oa[k] + i0));
        pM[k] = static_cast<M *>(W.msg) + ((size_t)f * W.msg_f + (uint32_t)(ob[k] + i0));
    }
#pragma unroll
    for (int k = 0; k < ND; k++) {
        pP[k] = W.phiq + ((size_t)f * W.d1_f + (uint32_t)(oa[NH + k] + i0));
        const uint32_t o = (uint32_t)(ob[NH + k] + (wb >> 5));
        pB[k] = W.bits + ((size_t)(((t - 1) & 1) * W.n_frames + f) * W.bit_f + o);
        pC[k] = W.bits + ((size_t)((t & 1) * W.n_frames + f) * W.bit_f + o);
    }
    const int cb = r * Z + i0;
    const uint32_t *sy = W.syn + ((size_t)f * W.words_m + (cb >> 5));
    const int ssh = 31 - (cb & 31);
    const int dsh = 31 - lane;
    uint32_t badw = 0;
    using Ops = PairOps<NH, ND, M>;
    auto load = [&](Ops &o, int c) {
#pragma unroll
        for (int k = 0; k < NH; k++) o.lv[k] = make_float2(pL[k][c * 32], pL[k][c * 32 + 32]);
        if constexpr (kReadMsg) {
#pragma unroll
            for (int k = 0; k < NH; k++) {
                o.ma[k] = ld_msg<M>(pM[k] + c * 32);
                o.mb[k] = ld_msg<M>(pM[k] + c * 32 + 32);
            }
        }
        if constexpr (kUpdate) {
#pragma unroll
            for (int k = 0; k < ND; k++) o.ph[k] = make_float2(__ldcg(pP[k] + c * 32), __ldcg(pP[k] + c * 32 + 32));
        }
        if constexpr (kTest) {
#pragma unroll
            for (int k = 0; k < ND; k++) {
                o.da[k] = pB[k][c];
                o.db[k] = pB[k][c + 1];
            }
        }
    };
    Ops buf[2];
    load(buf[0], 0);
#pragma unroll
    for (int c = 0; c < SLOTS; c += 2) {
        if (wb + c * 32 >= Z) break;  // warp-uniform
        const bool va = i0 + c * 32 < Z, vb = i0 + c * 32 + 32 < Z;
        // the next pair's operands are on their way while this one computes
        // (beyond Z they come from the next row or the array's padding)
        const Ops &o = buf[(c >> 1) & 1];
        if (c + 2 < SLOTS) load(buf[((c >> 1) + 1) & 1], c + 2);
        const uint32_t sa = kSyn && va ? __ldg(sy + c) << ssh : 0u, sb = kSyn && vb ? __ldg(sy + c + 1) << ssh : 0u;
        if constexpr (kTest) {
            uint32_t pa = sa, pb = sb;
#pragma unroll
            for (int k = 0; k < NH; k++) {
                pa ^= fbits(o.lv[k].x);
                pb ^= fbits(o.lv[k].y);
            }
#pragma unroll
            for (int k = 0; k < ND; k++) {
                pa ^= o.da[k] << dsh;
                pb ^= o.db[k] << dsh;
            }
            if (va) badw |= pa;
            if (vb) badw |= pb;
        }
        if constexpr (kUpdate) {
            float2 phi[D];
            uint32_t sga[D], sgb[D];
            uint32_t sta = sa, stb = sb;
#pragma unroll
            for (int k = 0; k < NH; k++) {
                float2 d = o.lv[k];
                if constexpr (kReadMsg) {
                    const float2 m = make_float2(Codec<M>::dec(o.ma[k], W), Codec<M>::dec(o.mb[k], W));
                    d = __ffma2_rn(m, f2(-1.0f), d);  // lv - m, one rounding
                }
                phi[k] = psi2_clamped(d, W.phi_lo, W.phi_hi);
                sga[k] = fbits(d.x);
                sgb[k] = fbits(d.y);
                sta ^= sga[k];
                stb ^= sgb[k];
            }
#pragma unroll
            for (int k = 0; k < ND; k++) {
                phi[NH + k] = make_float2(fabsf(o.ph[k].x), fabsf(o.ph[k].y));
                sga[NH + k] = fbits(o.ph[k].x);
                sgb[NH + k] = fbits(o.ph[k].y);
                sta ^= sga[NH + k];
                stb ^= sgb[NH + k];
            }
            float2 pre[D], suf[D];
            pre[0] = phi[0];
#pragma unroll
            for (int k = 1; k < D; k++) pre[k] = __fadd2_rn(pre[k - 1], phi[k]);
            suf[D - 1] = phi[D - 1];
#pragma unroll
            for (int k = D - 2; k >= 0; k--) suf[k] = __fadd2_rn(suf[k + 1], phi[k]);
#pragma unroll
            for (int k = 0; k < D; k++) {
                const float2 s2 = k == 0 ? suf[1] : k == D - 1 ? pre[D - 2] : __fadd2_rn(pre[k - 1], suf[k + 1]);
                if (k < NH) {
                    const uint32_t ska = (sta ^ sga[k]) & kSign, skb = (stb ^ sgb[k]) & kSign;
                    const float2 mag = psi2(make_float2(fmaxf(s2.x, W.xmin_h), fmaxf(s2.y, W.xmin_h)));
                    const M ea = Codec<M>::enc(__uint_as_float(fbits(mag.x) ^ ska), W);
                    const M eb = Codec<M>::enc(__uint_as_float(fbits(mag.y) ^ skb), W);
                    st_if(pM[k] + c * 32, ea, va);
                    st_if(pM[k] + c * 32 + 32, eb, vb);
                    red_add_if(pA[k] + c * 32, acc_value(ea, W), va);
                    red_add_if(pA[k] + c * 32 + 32, acc_value(eb, W), vb);
                } else {
                    const float2 ex = make_float2(fmaxf(s2.x, W.xmin), fmaxf(s2.y, W.xmin));
                    const uint32_t ba = ex.x < phi[k].x ? sta ^ sga[k] : sga[k];
                    const uint32_t bb = ex.y < phi[k].y ? stb ^ sgb[k] : sgb[k];
                    const uint32_t wa = __ballot_sync(0xffffffffu, va && (int)ba < 0);
                    const uint32_t wv = __ballot_sync(0xffffffffu, vb && (int)bb < 0);
                    st_if(pC[k - NH] + c, wa, lane == 0);
                    st_if(pC[k - NH] + c + 1, wv, lane == 0 && vb);
                    if constexpr (SOFT) {
                        const uint32_t ska = (sta ^ sga[k]) & kSign, skb = (stb ^ sgb[k]) & kSign;
                        if (va) soft_deg1(T, W, f, r, t, rp + k, i0 + c * 32, ex.x, ska);
                        if (vb) soft_deg1(T, W, f, r, t, rp + k, i0 + c * 32 + 32, ex.y, skb);
                    }
                }
            }
        }
    }
    return (int)badw < 0;
}

template <int MODE, typename M, int SLOTS, bool SOFT>
__device__ __forceinline__ bool cd_dispatch(const Table &T, const Work &W, int f, int4 head, int t, const int *oa,
                                            const int *ob, int wb) {
    const int r = head.x, rp = head.y;
    switch (head.z * 4 + head.w) {
        case 1 * 4 + 1: return cd_row<1, 1, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 2 * 4 + 0: return cd_row<2, 0, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 2 * 4 + 1: return cd_row<2, 1, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 3 * 4 + 0: return cd_row<3, 0, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 3 * 4 + 1: return cd_row<3, 1, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 4 * 4 + 0: return cd_row<4, 0, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        case 4 * 4 + 1: return cd_row<4, 1, MODE, M, SLOTS, SOFT>(T, W, f, r, rp, t, oa, ob, wb);
        default: return false;
    }
}

// Flooding check pass of iteration t: grid (tiles of blockDim.x SLOTS checks,
// base row in shape order, frame).
template <typename M, int SLOTS, bool SOFT>
__global__ void __launch_bounds__(qc::kCnDirectThreads, kCdMinBlocks)
    cn_direct_kernel(const __grid_constant__ Table T, const __grid_constant__ Work W) {
    // One store of the frame's failure per block: far from convergence every
    // warp has a failed check, and a store from each queued up in the L2 at
    // the one word (n = 10^6, 16 frames: 185 us a pass against 105 us).
    __shared__ int s_failed;
    // The posterior pass may be scheduled once the last block runs, unless other
    // chains run beside this one: its waiting blocks would keep theirs off the
    // SMs (see cn_tma_kernel, whose blocks are larger and gain nothing by it).
    if (!W.side) pdl_launch_dependents();
    if (threadIdx.x == 0) s_failed = 0;
    __syncthreads();
    pdl_wait();  // after a programmatic edge: the previous posterior pass is complete
    const int f = blockIdx.z;
    const qc::RowDesc *dp = T.row_desc_ord + blockIdx.y;
    const int4 head = __ldg(reinterpret_cast<const int4 *>(dp));  // r, rp, nh, nd
    int oa[qc::kDescEnts], ob[qc::kDescEnts];
    load_offsets(dp, oa, ob);
    const int t = W.t[f];
    const bool running = W.active[f] != 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
        W.ct[f] = running ? t : 0;  // for the posterior pass, which counts t on
    const int wb = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (32 * SLOTS);
    if (!running || wb >= T.Z) return;  // warp-uniform
    const int mode = t > W.max_iter ? kTestOnly : t == 1 ? kFirst : (t - 1 >= W.et_start) ? kSteadyTest : kSteady;
    bool bad;
    switch (mode) {
        case kFirst: bad = cd_dispatch<kFirst, M, SLOTS, SOFT>(T, W, f, head, t, oa, ob, wb); break;
        case kSteady: bad = cd_dispatch<kSteady, M, SLOTS, SOFT>(T, W, f, head, t, oa, ob, wb); break;
        case kSteadyTest: bad = cd_dispatch<kSteadyTest, M, SLOTS, SOFT>(T, W, f, head, t, oa, ob, wb); break;
        default: bad = cd_dispatch<kTestOnly, M, SLOTS, SOFT>(T, W, f, head, t, oa, ob, wb); break;
    }
    if (mode == kSteadyTest || mode == kTestOnly) {
        if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0 && atomicExch(&s_failed, 1) == 0)
            W.fail[(size_t)f * W.fail_f] = t;
    }
}

// slots: checks per lane, 2 or 8 (soft output: 2).
template <typename M>
void *cn_direct_select(int slots, bool soft) {
    if (soft) return (void *)cn_direct_kernel<M, 2, true>;
    if (slots == 8) return (void *)cn_direct_kernel<M, 8, false>;
    return (void *)cn_direct_kernel<M, 2, false>;
}
}  // namespace
