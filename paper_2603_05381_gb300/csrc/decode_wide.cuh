#pragma once
// Streaming tier of the BP4M decoder in FP32 arithmetic: shots with more unsatisfied detectors
// than the shared-memory tiers hold, their message matrices in a scratch slot in global memory
// (one per block, or one per thread-block cluster in the cluster form).  FP32, IEEE half or
// bfloat16 messages.  (FP64: decode_stream.cuh.)
//
// Slot (LD = 32 CH columns):
//   Lg[r][k]     prior l_rk in log2 units, -inf for k >= s
//   Mt[b][r][k]  message M[k][r] arriving at row r (b = iteration parity); diagonal 0, or with
//                16-bit storage r_r, which decodes to 0 (see decode_smem.cuh)
//   and with 16-bit storage room between the two, so that either buffer and the room hold the
//   FP32 posteriors of a decision (FP32 storage: the other buffer alone)
// A row's own outputs M[r][k] are column r of Mt: nothing else is kept of them.
//
// Update.  A warp updates two rows at a time, 16 lanes each; lane t of a row holds the columns
// 32 c + 2t and 32 c + 2t + 1, so that two columns share one 64-bit shared-memory access and one
// packed FP32x2 operation, and two rows share one reduction.  The sums are those of 32 lanes
// holding one column of each 32 and added by halves (16, 8, 4, 2, 1 apart), in that order.  Rows
// of Lg and Mt are copied ahead into shared memory (cp.async) while the warp works on the rows
// before them; outputs are staged for the 2 W rows of a block's batch and written transposed,
// four rows a thread.
//
// Bound: the rows' way from L2 and DRAM (12 bytes an FP32 update, 8 with 16-bit messages) and the
// barriers of the batches; instruction issue is active in 27 to 39% of the cycles.  One row a warp with all
// posteriors judged in every iteration measured (us a shot, circuit at p = 0.005, FP32 / FP16)
// 7.1 / - at d = 15, 14.0 / 13.8 at 17, 29.6 / 27.0 at 19, 62.3 / 55.2 at 21, 235 / - at 25;
// this form 5.0, 11.5 / 9.1, 21.4 / 16.2, 43.9 / 34.5, 163.
//
// Decisions.  An iteration has converged only if every row keeps exactly one variable, so a row
// that does not settles it: two warps of a block look at one row each, beside the update, and the
// rows are judged (all posteriors) only when no watched row violates, in the last iteration and
// wherever a candidate is needed.  Judging every posterior in every iteration took 17 warp
// instructions of 45 per 32 updates, and an own-output matrix to be written and read.
//
// Cluster form (CL > 1): the CL blocks of a cluster share one shot and one slot.  Block q
// updates the batches q, q + CL, ...; messages cross blocks only through the slot (read past
// L1); per-row state goes into every block's copy through distributed shared memory, after
// which every block runs the row-global steps (matching rounds, candidate weights) on identical
// data, so that every branch and loop bound is the same in all blocks and every cluster barrier
// is reached by all of them.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <type_traits>

#include "decode_smem.cuh"
#include "device.cuh"

namespace bp4m {
namespace {

namespace cg = cooperative_groups;

// Bytes of a slot: priors and two message matrices, and with 16-bit messages the room beside them.
template <typename MS>
constexpr size_t wide_slot_bytes(int ld) {
    return (size_t)ld * ld * (sizeof(MS) == 2 ? 10 : 12);
}

// Blocks per SM at CH columns per lane: two where each still has batches of sixteen rows, so that
// one block's memory latency and barriers run beside the other's arithmetic (448 columns in FP32:
// 22.8 -> 21.4 us a d = 19 shot; 640 columns, with batches of twelve rows: 43.9 -> 49.6 us, so one;
// 16-bit messages at 448 and 512 columns: 16.2 -> 17.2 us, so one).
constexpr int wide_blocks(int ch, int msg_bytes) { return ch <= (msg_bytes == 4 ? 16 : 12) ? 2 : 1; }

// ALONE: one block per SM with the warps of two, for launches of no more shots than SMs.  Blocks of half
// the warps would leave half of an SM idle, or meet two to an SM while other SMs hold the batch's smaller
// classes.  FP32, halves -> alone (us, BP4M at T = 12 / BP4MF at T = 10): 152 shots of 192 columns
// 243 / 633 -> 230 / 580, of 320 674 / 1866 -> 584 / 1419, of 448 1320 / 4996 -> 1152 / 3166, of 512 1672 / 6440 ->
// 1460 / 4598; one shot of 448 columns 848 / 2685 -> 729 / 1976.
template <int CH, typename MS, int CL = 1, bool ALONE = false>
struct WideShape {
    static constexpr int LD = 32 * CH;
    static constexpr bool HALF = sizeof(MS) == 2;
    // output stage pitch in elements: row pairs of a column pair in distinct banks
    static constexpr int SP = LD + 2;
    static constexpr int blocks = CL == 1 && !ALONE ? wide_blocks(CH, (int)sizeof(MS)) : 1;
    // prefetched message rows: 16-bit rows apart by half the banks
    static constexpr int PX = HALF ? LD + 32 : LD;
    static constexpr size_t per_warp = 2 * ((size_t)LD * 4 + (size_t)(PX + SP) * sizeof(MS));
    static constexpr size_t fixed = (size_t)LD * (8 + 4 + 4 + 2 + 2 + 8 + (HALF ? 8 : 0)) + 256;
    static constexpr size_t watch_bytes = (size_t)2 * LD * (4 + sizeof(MS));  // the watched rows' priors and messages
    static constexpr size_t budget = (blocks == 2 ? 113 : 227) * 1024 - 1024;
    static constexpr int fit(size_t extra) { return (int)((budget - fixed - extra) / per_warp) / 2 * 2; }
    // Warps per block (even): as many as fit, and in the cluster form the count that leaves the
    // least to the busiest block (the batches of 2 W rows go round the blocks; with the largest
    // batches a 395-defect shot left two of forty rows to some of eight blocks and one to others:
    // 9% slower than sixteen-row batches).
    static constexpr int cap = blocks == 2 ? 16 : CH <= 16 ? 24 : 20;
    static constexpr int most = fit(0) < cap ? fit(0) : cap;
    static constexpr int warps() {
        if (CL == 1) return most;
        int best = most, rows = 1 << 30;
        for (int w = 4; w <= most; w += 2) {
            const int batches = (LD + 2 * w - 1) / (2 * w);
            const int r = (batches + CL - 1) / CL * (2 * w + 6);  // a batch costs about six rows more
            if (r <= rows) {
                rows = r;
                best = w;
            }
        }
        return best;
    }
    static constexpr int W = warps();
    static constexpr bool WBUF = fit(watch_bytes) >= W;       // room for the watched rows
    static constexpr int RB = 2 * W;                          // rows per batch (multiple of 4)
    static constexpr size_t smem = per_warp * W + fixed + (WBUF ? watch_bytes : 0);
    static constexpr size_t slot_bytes = wide_slot_bytes<MS>(LD);
};

template <int CH, typename MS, int CL, bool ALONE = false>
__global__ void __launch_bounds__(WideShape<CH, MS, CL, ALONE>::W * 32, WideShape<CH, MS, CL, ALONE>::blocks) decode_wide_kernel(const DecodeArgs a) {
    using SH = WideShape<CH, MS, CL, ALONE>;
    using IO = MsgIO<MS, float>;
    constexpr bool HALF = SH::HALF;
    constexpr int LD = SH::LD, SP = SH::SP, PX = SH::PX, W = SH::W, RB = SH::RB, NTH = W * 32;
    static_assert(W >= 4 && W % 2 == 0, "two watching warps, batches of a multiple of four rows");
    extern __shared__ __align__(16) unsigned char smem[];
    // per warp: two prior rows, two message rows; then the stage
    float* const pl0 = reinterpret_cast<float*>(smem);
    MS* const px0 = reinterpret_cast<MS*>(smem + (size_t)W * 2 * LD * 4);
    MS* const stage = px0 + (size_t)W * 2 * PX;
    double* const rowacc = reinterpret_cast<double*>(smem + SH::per_warp * W);
    int* const dets = reinterpret_cast<int*>(rowacc + LD);
    int* const choice = dets + LD;
    float* const dgv = reinterpret_cast<float*>(choice + LD);   // [2][LD]: M[r][r] by iteration parity
    float* const nref = dgv + 2 * LD;                           // 16-bit: [2][LD], -r_k of the messages of Mt[b]
    short* const bestp = reinterpret_cast<short*>(nref + (HALF ? 2 * LD : 0));
    short* const order = bestp + LD;
    float* const rowf = reinterpret_cast<float*>(rowacc);        // static partition: the maximum of each row's block
    unsigned* const wown = reinterpret_cast<unsigned*>(rowacc);  // [2][LD]: watched rows' own outputs
    // the watched rows' priors [2][LD] and messages [2][LD], where there is room
    float* const wl = reinterpret_cast<float*>(smem + SH::per_warp * W + SH::fixed);
    MS* const wx = reinterpret_cast<MS*>(wl + 2 * LD);
    __shared__ unsigned openw[CH];          // forced convergence: unmatched rows
    __shared__ int sh_item2[2], sh_s, sh_best_par, sh_best_forced, sh_improve, sh_use_best, sh_bad[2];
    __shared__ int sh_votes[2][CL];
    __shared__ double sh_best_w;

    const int crank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
    auto csync = [&]() {
        if constexpr (CL > 1)
            cg::this_cluster().sync();
        else
            __syncthreads();
    };
    auto bcast = [&](auto* p, auto v) {
        if constexpr (CL > 1) {
            cg::cluster_group cl = cg::this_cluster();
#pragma unroll
            for (int q = 0; q < CL; ++q) *cl.map_shared_rank(p, q) = v;
        } else {
            *p = v;
        }
    };
    unsigned char* const slot = reinterpret_cast<unsigned char*>(a.gscratch) + (size_t)(blockIdx.x / CL) * SH::slot_bytes;
    float* const Lg = reinterpret_cast<float*>(slot);
    constexpr size_t MAT = (size_t)LD * LD;
    MS* const Mt0 = reinterpret_cast<MS*>(slot + MAT * 4);
    constexpr size_t MOFF = HALF ? 2 * MAT : MAT;  // element offset of Mt[1]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int hf = lane >> 4, t16 = lane & 15;     // the lane's row of the warp's two, its column pair
    const int64_t count = a.count ? (int64_t)*a.count : a.count_val;
    const float ainv = (float)(1.0 / a.alpha);
    const bool full = (a.decoder == 1) || !a.early_exit;
    float* const trl = reinterpret_cast<float*>(a.tr_lambda);
    const float ninf = Num<float>::ninf();
    unsigned long long acc_it = 0, acc_msg = 0, acc_def = 0, acc_shots = 0, acc_fc = 0, acc_fcr = 0;

    // every block of the cluster runs before any block writes into another's shared memory
    if constexpr (CL > 1) csync();
    for (int fetch = 0;; ++fetch) {
        // the cluster's next shot, taken by block 0 and written into every block (two
        // buffers by fetch parity: a block may still be reading the previous one)
        const int fb = CL > 1 ? (fetch & 1) : 0;
        if (crank == 0 && tid == 0) bcast(&sh_item2[fb], atomicAdd(a.next, 1));
        csync();
        const int item = sh_item2[fb];
        if (item >= count) break;
        const ItemCtx ic = resolve_item(a, a.list ? (int64_t)a.list[item] : (int64_t)item);
        const int64_t shot = ic.shot;
        const int n = ic.tb.n_det;
        if (warp == 0) {
            const int s0 = compact_defects(ic.synd + (size_t)shot * ic.tb.n_words, ic.tb.n_words, dets, LD, lane);
            if (lane == 0) sh_s = s0;
        }
        __syncthreads();
        const int s = sh_s;
        if (s > LD || s < 2) {
            if (crank == 0 && tid == 0 && a.ctr) atomicAdd(a.ctr + C_ERRORS, 1ull);
            continue;
        }
        const bool tr_on = CL == 1 && (trl != nullptr || a.tr_partner != nullptr) && s <= a.s_cap;
        for (int r = crank * W + warp; r < s; r += W * CL) {
            const float* trow = ic.tb.L32 + (size_t)dets[r] * n;
#pragma unroll 4
            for (int k = lane; k < LD; k += 32) {
                Lg[(size_t)r * LD + k] = k < s ? __ldg(trow + dets[k]) * (float)kLog2e : ninf;
                Mt0[(size_t)r * LD + k] = MS(0.f);
                Mt0[MOFF + (size_t)r * LD + k] = MS(0.f);
            }
        }
        for (int r = tid; r < LD; r += NTH) {
            bestp[r] = -1;
            dgv[r] = dgv[LD + r] = 0.f;
            if constexpr (HALF) nref[r] = nref[LD + r] = 0.f;
        }
        if (tid == 0) {
            sh_best_w = Num<double>::pinf();
            sh_best_par = 0;
            sh_best_forced = 0;
            sh_use_best = 0;
            sh_bad[0] = sh_bad[1] = -1;
        }
        // every block's rows of the slot are initialised before any block writes into them
        csync();

        int cur = 0, t = 0, par_v = 0;  // par_v: parity of the cluster votes
        // rows this block judges: groups of eight, q = crank, crank + CL, ...
        const int ngrp = (s + 7) / 8;
        // the rows that the last two warps watch (-1: none of this block's rows)
        int watch = -1;
        {
            const int wq = warp - (W - 2);
            const int mine = (ngrp - crank + CL - 1) / CL;  // groups of this block
            if (wq >= 0 && mine > 0) watch = min(((mine * (2 * wq + 1) / 4) * CL + crank) * 8, s - 1);
        }
        bool any_conv = false, forced_ran = false;
        int out_par = 0, out_forced = 0, out_from_best = 0;
        // the update t + 1 has been made and lambda^t has to be judged
        bool ahead = false;

        // message from `from` to `to` in the current buffer
        auto msg = [&](int to, int from) -> float {
            const MS* p = Mt0 + (cur ? MOFF : 0) + (size_t)to * LD + from;
            if constexpr (HALF) {
                const unsigned short v = CL > 1 ? __ldcg(reinterpret_cast<const unsigned short*>(p))
                                                : *reinterpret_cast<const unsigned short*>(p);
                return IO::unpack((unsigned)v).x + nref[cur * LD + from];
            } else {
                return CL > 1 ? __ldcg(p) : *p;
            }
        };
        auto prior = [&](int r, int k) -> float {
            const float* p = Lg + (size_t)r * LD + k;
            return CL > 1 ? __ldcg(p) : *p;
        };
        // the decision's posteriors: the other message buffer (and the room beside it)
        auto lam_mat = [&]() -> float* {
            return HALF ? (cur ? reinterpret_cast<float*>(Mt0) : reinterpret_cast<float*>(Mt0 + MAT))
                        : reinterpret_cast<float*>(Mt0 + (cur ? 0 : MOFF));
        };
        // Posteriors of this block's rows: kept counts (returns whether each row keeps exactly one;
        // the kept column goes to every block's choice[]); with `store` they are written to
        // lam_mat(), with `blocks` the static partition's block of a row (its columns k >= r) gives its
        // maximum to rowf[] and the column (ties: the smaller) to order[] of every block.  Eight rows
        // a warp, sixteen columns at a time, four a lane: the rows are read in 64-byte pieces and the
        // columns (the own outputs) in whole 32-byte sectors.
        // (BP4MF with the static partition, T = 10, FP32, us for 304 shots of one width, storing the posteriors,
        // scanning them again and comparing the maxima in FP64 -> so: 3800 -> 2024 at 320 columns,
        // 17130 -> 8858 at 640, 50899 -> 27241 at 1024.)
        auto judge = [&](bool store, auto blocks) -> int {
            int ok = 1;
            float* const lam_g = lam_mat();
            const MS* const mc = Mt0 + (cur ? MOFF : 0);
            const float* const nr = nref + cur * LD;
            for (int q = crank + CL * warp; q < ngrp; q += CL * W) {
                const int r = q * 8 + (lane & 7);
                int cnt = 0, kl = -1, bk = 0x7fffffff;
                float bl = ninf;
                if (r < s) {
                    const float dgr = dgv[cur * LD + r];
                    const float nrr = HALF ? nr[r] : 0.f;
                    const float* const lrow = Lg + (size_t)r * LD;
                    const MS* const xrow = mc + (size_t)r * LD;
                    constexpr int U = HALF && decltype(blocks)::value ? 1 : 2;
#pragma unroll U
                    for (int k = 4 * (lane >> 3); k < s; k += 16) {
                        const float4* const lp = reinterpret_cast<const float4*>(lrow + k);
                        const float4 l = CL > 1 ? __ldcg(lp) : *lp;
                        float4 x;
                        float own[4];
                        if constexpr (HALF) {
                            const uint2* const xp = reinterpret_cast<const uint2*>(xrow + k);
                            const uint2 v = CL > 1 ? __ldcg(xp) : *xp;
                            const float4 nk = *reinterpret_cast<const float4*>(nr + k);
                            const float2 lo = __fadd2_rn(IO::unpack(v.x), make_float2(nk.x, nk.y));
                            const float2 hi = __fadd2_rn(IO::unpack(v.y), make_float2(nk.z, nk.w));
                            x = make_float4(lo.x, lo.y, hi.x, hi.y);
                        } else {
                            const float4* const xp = reinterpret_cast<const float4*>(xrow + k);
                            x = CL > 1 ? __ldcg(xp) : *xp;
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const MS* const op = mc + (size_t)min(k + e, s - 1) * LD + r;
                            if constexpr (HALF) {
                                const unsigned short v = CL > 1 ? __ldcg(reinterpret_cast<const unsigned short*>(op))
                                                                : *reinterpret_cast<const unsigned short*>(op);
                                own[e] = IO::unpack((unsigned)v).x + nrr;
                            } else {
                                own[e] = CL > 1 ? __ldcg(op) : *op;
                            }
                        }
                        float4 lam = make_float4(l.x + (own[0] + x.x), l.y + (own[1] + x.y), l.z + (own[2] + x.z),
                                                 l.w + (own[3] + x.w));
                        if ((r & ~3) == k) {
                            // the boundary variable
                            if ((r & 3) == 0) lam.x = l.x + dgr;
                            if ((r & 3) == 1) lam.y = l.y + dgr;
                            if ((r & 3) == 2) lam.z = l.z + dgr;
                            if ((r & 3) == 3) lam.w = l.w + dgr;
                        }
                        cnt += (lam.x > 0.f) + (lam.y > 0.f) + (lam.z > 0.f) + (lam.w > 0.f);
                        kl = lam.w > 0.f ? k + 3 : lam.z > 0.f ? k + 2 : lam.y > 0.f ? k + 1 : lam.x > 0.f ? k : kl;
                        if (store) *reinterpret_cast<float4*>(lam_g + (size_t)r * LD + k) = lam;
                        if constexpr (blocks.value) {
                            const float v[4] = {lam.x, lam.y, lam.z, lam.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (k + e >= r && k + e < s && (bk == 0x7fffffff || v[e] > bl)) {
                                    bl = v[e];
                                    bk = k + e;
                                }
                        }
                    }
                }
                if constexpr (blocks.value) {
#pragma unroll
                    for (int off = 8; off < 32; off <<= 1) {
                        const float ol = __shfl_xor_sync(kFull, bl, off);
                        const int ok2 = __shfl_xor_sync(kFull, bk, off);
                        if (ok2 != 0x7fffffff && (bk == 0x7fffffff || ol > bl || (ol == bl && ok2 < bk))) {
                            bl = ol;
                            bk = ok2;
                        }
                    }
                    if (lane < 8 && r < s) {
                        bcast(&rowf[r], bl);
                        bcast(&order[r], (short)bk);
                    }
                }
#pragma unroll
                for (int off = 8; off < 32; off <<= 1) {
                    cnt += __shfl_xor_sync(kFull, cnt, off);
                    kl = max(kl, __shfl_xor_sync(kFull, kl, off));
                }
                if (r < s) {
                    if (lane < 8) bcast(&choice[r], kl >= 0 ? kl : 0x7fffffff);
                    if (cnt != 1) {
                        ok = 0;
                        // a violating row to watch (any will do)
                        if (lane < 8) atomicMax(&sh_bad[(q / CL) & 1], r);
                    }
                }
            }
            return ok;
        };
        // all blocks' votes: 1 if every one is 1
        auto vote_all = [&](int ok) -> int {
            const int cta = __syncthreads_and(ok);
            if constexpr (CL > 1) {
                par_v ^= 1;
                if (tid == 0) bcast(&sh_votes[par_v][crank], cta);
                csync();
                int v = 1;
#pragma unroll
                for (int q = 0; q < CL; ++q) v &= sh_votes[par_v][q];
                return v;
            }
            return cta;
        };
        for (;;) {
            const bool first = t > 0 && !ahead && (tr_on || t == a.T || a.decoder == 1);
            if (ahead || first) {
                // ---- decisions of lambda^t = l + (M[r][k] + M[k][r])
                // the static partition needs no posteriors beyond its blocks' maxima
                const int conv = vote_all(first && a.forced_static ? judge(tr_on && trl, std::true_type()) : judge(first, std::false_type()));
                if (!conv && warp >= W - 2) {
                    const int b = sh_bad[warp & 1] >= 0 ? sh_bad[warp & 1] : sh_bad[(warp & 1) ^ 1];
                    if (b >= 0) watch = b;
                }
                const float* const lam_g = lam_mat();
                auto lam_at = [&](int r, int k) -> float {
                    return CL > 1 ? __ldcg(lam_g + (size_t)r * LD + k) : lam_g[(size_t)r * LD + k];
                };
                if (tr_on && trl) {
                    __syncthreads();
                    for (int r = warp; r < s; r += W)
                        for (int k = lane; k < s; k += 32)
                            trl[((size_t)shot * a.s_cap + r) * a.s_cap + k] = lam_at(r, k) * (float)kLn2;
                }
                bool have_cand = false, cand_forced = false;
                if (conv) {
                    any_conv = true;
                    have_cand = true;
                } else if (a.decoder == 1 || t == a.T) {
                    // ---- forced convergence on lambda^t
                    forced_ran = true;
                    for (int c = tid; c < CH; c += NTH) openw[c] = s >= 32 * (c + 1) ? kFull : s <= 32 * c ? 0u : (1u << (s & 31)) - 1u;
                    csync();  // (also: every block's posteriors precede the reads below)
                    if (a.forced_static) {
                        // the paper's static partition: row r's block is v_rk, k >= r; its
                        // maximum (ties: smaller k) represents factor r; representatives are
                        // ranked by posterior (ties: smaller r) and processed in that order
                        for (int r = tid; r < s; r += NTH) choice[r] = order[r];
                        __syncthreads();
                        for (int r = tid; r < s; r += NTH) {
                            const float v = rowf[r];
                            int rank = 0;
                            for (int j = 0; j < s; j += 4) {
                                const float4 u = *reinterpret_cast<const float4*>(rowf + j);
                                rank += (u.x > v || (u.x == v && j < r)) ? 1 : 0;
                                rank += j + 1 < s && (u.y > v || (u.y == v && j + 1 < r)) ? 1 : 0;
                                rank += j + 2 < s && (u.z > v || (u.z == v && j + 2 < r)) ? 1 : 0;
                                rank += j + 3 < s && (u.w > v || (u.w == v && j + 3 < r)) ? 1 : 0;
                            }
                            order[rank] = (short)r;
                        }
                        __syncthreads();
                        if (tid == 0) {
                            // a factor whose representative's other factor is taken goes to the
                            // boundary (a case the paper does not treat)
                            for (int q = 0; q < s; ++q) {
                                const int rr = order[q];
                                if (!((openw[rr >> 5] >> (rr & 31)) & 1u)) continue;
                                const int k = choice[rr];
                                openw[rr >> 5] &= ~(1u << (rr & 31));
                                if (k == rr || !((openw[k >> 5] >> (k & 31)) & 1u)) {
                                    choice[rr] = rr;
                                } else {
                                    openw[k >> 5] &= ~(1u << (k & 31));
                                    choice[k] = rr;
                                }
                            }
                            if (crank == 0) acc_fcr += 1;
                        }
                        __syncthreads();
                    }
                    // greedy matching by rounds of locally dominant choices; a row whose choice is
                    // still unmatched keeps it (the best of a set that has only shrunk around it)
                    for (int round = 0; round < s && !a.forced_static; ++round) {
                        for (int r = crank * W + warp; r < s; r += W * CL) {
                            if (!((openw[r >> 5] >> (r & 31)) & 1u)) continue;  // uniform per warp
                            if (round > 0) {
                                const int pk = choice[r];
                                if ((openw[pk >> 5] >> (pk & 31)) & 1u) continue;
                            }
                            float bl = ninf;
                            int bk = 0x7fffffff;
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int k = lane + 32 * c;
                                if ((openw[c] >> lane) & 1u) {
                                    const float lam = lam_at(r, k);
                                    if (bk == 0x7fffffff || lam > bl) {
                                        bl = lam;
                                        bk = k;
                                    }
                                }
                            }
#pragma unroll
                            for (int off = 16; off; off >>= 1) {
                                const float ol = __shfl_xor_sync(kFull, bl, off);
                                const int okk = __shfl_xor_sync(kFull, bk, off);
                                if (okk != 0x7fffffff && (bk == 0x7fffffff || ol > bl || (ol == bl && okk < bk))) {
                                    bl = ol;
                                    bk = okk;
                                }
                            }
                            __syncwarp();
                            if (lane == 0) bcast(&choice[r], bk != 0x7fffffff ? bk : r);
                        }
                        csync();
                        int left = 0;
                        for (int r = tid; r < s; r += NTH) {
                            rowacc[r] = 0.0;
                            if (!((openw[r >> 5] >> (r & 31)) & 1u)) continue;
                            const int pk = choice[r];
                            const bool newm = (pk == r) || (choice[pk] == r);
                            rowacc[r] = newm ? 1.0 : 0.0;
                            left += !newm;
                        }
                        __syncthreads();
                        for (int r = tid; r < s; r += NTH)
                            if (rowacc[r] != 0.0) atomicAnd(&openw[r >> 5], ~(1u << (r & 31)));
                        if (tid == 0 && crank == 0) acc_fcr += 1;
                        const int left_all = __syncthreads_count(left);
                        // cluster form: the next round's choices overwrite every block's copy
                        if constexpr (CL > 1) csync();
                        if (left_all == 0) break;
                    }
                    if (tid == 0 && crank == 0) acc_fc += 1;
                    have_cand = true;
                    cand_forced = true;
                }
                if (have_cand) {
                    int pc = 0;
                    for (int r = tid; r < s; r += NTH) {
                        const int k = choice[r];
                        double w = 0.0;
                        if (k >= r) {
                            const size_t off = (size_t)dets[r] * n + dets[k];
                            pc ^= ic.tb.P[off];
                            if (full) w = ic.tb.W64[off];
                        }
                        rowacc[r] = w;
                    }
                    const int par = __syncthreads_count(pc) & 1;
                    bool finish = false;
                    if (!full) {
                        out_par = par;
                        out_forced = cand_forced;
                        finish = true;
                    } else {
                        if (tid == 0) {
                            double w = 0.0;
                            for (int r = 0; r < s; ++r) w += rowacc[r];
                            sh_improve = 0;
                            sh_use_best = 0;
                            if (a.decoder == 1 || !cand_forced) {
                                if (w < sh_best_w) {
                                    sh_best_w = w;
                                    sh_best_par = par;
                                    sh_best_forced = cand_forced;
                                    sh_improve = 1;
                                }
                            } else {
                                sh_use_best = sh_best_w <= w;
                            }
                        }
                        __syncthreads();
                        if (sh_improve)
                            for (int r = tid; r < s; r += NTH) bestp[r] = (short)choice[r];
                        if (t == a.T || (a.decoder == 0 && cand_forced)) {
                            finish = true;
                            if (a.decoder == 0 && cand_forced && !sh_use_best) {
                                out_par = par;
                                out_forced = 1;
                            } else {
                                out_par = sh_best_par;
                                out_forced = sh_best_forced;
                                out_from_best = 1;
                            }
                        }
                        __syncthreads();
                    }
                    if (finish) break;
                }
                if (ahead) {
                    ahead = false;
                    cur ^= 1;
                    ++t;
                    csync();
                    continue;
                }
                // the update overwrites the posteriors and the decision's scratch
                csync();
                if constexpr (HALF) {
                    // the FP32 posteriors went over columns past s of the next messages, which are
                    // read but never written
                    for (int r = crank * W + warp; r < s; r += W * CL)
                        for (int k = s + lane; k < LD; k += 32) Mt0[(cur ? 0 : MOFF) + (size_t)r * LD + k] = MS(0.f);
                }
            }
            if (tid == 0) sh_bad[0] = sh_bad[1] = -1;
            // ---- update pass: M' for every row, batch by batch
            const MS* const Mc = Mt0 + (cur ? MOFF : 0);
            MS* const Mn = Mt0 + (cur ? 0 : MOFF);
            const float* const nrc = nref + cur * LD;
            const int nxt = cur ^ 1;
            const int nbatch = (s + RB - 1) / RB;
            const int rl = 2 * warp + hf;  // this half warp's row in a batch
            float* const pl = pl0 + (size_t)rl * LD;
            MS* const px = px0 + (size_t)rl * PX;
            auto prefetch = [&](int r) {
                if (r < s) {
                    const unsigned char* const sl = reinterpret_cast<const unsigned char*>(Lg + (size_t)r * LD);
                    const unsigned char* const sx = reinterpret_cast<const unsigned char*>(Mc + (size_t)r * LD);
                    constexpr int VL = LD * 4 / 16, VM = LD * (int)sizeof(MS) / 16;
#pragma unroll
                    for (int v = 0; v < VL; v += 16)
                        if (VL % 16 == 0 || v + t16 < VL)
                            cp_async16(reinterpret_cast<unsigned char*>(pl) + 16 * (v + t16), sl + 16 * (v + t16));
#pragma unroll
                    for (int v = 0; v < VM; v += 16)
                        if (VM % 16 == 0 || v + t16 < VM)
                            cp_async16(reinterpret_cast<unsigned char*>(px) + 16 * (v + t16), sx + 16 * (v + t16));
                }
                cp_async_commit();
            };
            const bool vote = t > 0 && !first;
            const bool watching = vote && warp >= W - 2 && watch >= 0;
            // the watched row's own outputs, a column of Mc, as 4-byte words
            auto own_word = [&](int k) -> const unsigned char* {
                return reinterpret_cast<const unsigned char*>(Mc) + ((((size_t)k * LD + watch) * sizeof(MS)) & ~(size_t)3);
            };
            if (watching) {
                if constexpr (CL == 1)
                    for (int k = lane; k < s; k += 32) cp_async4(wown + (warp & 1) * LD + k, own_word(k));
                if constexpr (SH::WBUF) {
                    for (int v = lane; v < LD / 4; v += 32)
                        cp_async16(wl + (warp & 1) * LD + 4 * v, Lg + (size_t)watch * LD + 4 * v);
                    for (int v = lane; v < LD * (int)sizeof(MS) / 16; v += 32)
                        cp_async16(reinterpret_cast<unsigned char*>(wx + (warp & 1) * LD) + 16 * v,
                                   reinterpret_cast<const unsigned char*>(Mc + (size_t)watch * LD) + 16 * v);
                }
            }
            prefetch(crank * RB + rl);
            if (CL > 1 && watching) {
#pragma unroll 8
                for (int k = lane; k < s; k += 32)
                    wown[(warp & 1) * LD + k] = __ldcg(reinterpret_cast<const unsigned*>(own_word(k)));
            }
            const float2 ainv2 = make_float2(ainv, ainv), neg1 = make_float2(-1.f, -1.f);
            for (int b = crank; b < nbatch; b += CL) {
                const int r = b * RB + rl;
                MS* const srow = stage + (size_t)rl * SP;
                cp_async_wait_all();
                __syncwarp();
                // Q = l + M[k][r]/alpha, its maximum and second maximum
                float2 q[CH];
                float m1 = ninf, m2 = ninf;
#pragma unroll
                for (int c = 0; c < CH; c += 2) {
                    float2 p[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int k = 32 * (c + e) + 2 * t16;
                        const float2 l = *reinterpret_cast<const float2*>(pl + k);
                        float2 x;
                        if constexpr (HALF)
                            x = __fadd2_rn(IO::ld2(px + k), *reinterpret_cast<const float2*>(nrc + k));
                        else
                            x = *reinterpret_cast<const float2*>(px + k);
                        p[e] = __ffma2_rn(x, ainv2, l);
                        q[c + e] = p[e];
                    }
                    const float h0 = fmaxf(p[0].x, p[0].y), l0 = fminf(p[0].x, p[0].y);
                    const float h1 = fmaxf(p[1].x, p[1].y), l1 = fminf(p[1].x, p[1].y);
                    const float hi = fmaxf(h0, h1), lo = max3f(l0, l1, fminf(h0, h1));
                    m2 = max3f(m2, lo, fminf(m1, hi));
                    m1 = fmaxf(m1, hi);
                }
                // the last read of this row's prefetch buffers: the next row may replace them
                __syncwarp();
                prefetch(r + RB * CL);
#pragma unroll
                for (int off = 8; off; off >>= 1) {
                    const float o1 = __shfl_xor_sync(kFull, m1, off), o2 = __shfl_xor_sync(kFull, m2, off);
                    m2 = max3f(m2, o2, fminf(m1, o1));
                    m1 = fmaxf(m1, o1);
                }
                // exponentials and their sum; the column above m2 (decode_smem.cuh)
                const float2 m22 = make_float2(m2, m2);
                float2 s2 = make_float2(0.f, 0.f);
                unsigned topx = 0, topy = 0;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const float2 dq = __ffma2_rn(q[c], neg1, m22);
                    const float2 u = make_float2(B2<float>::ex2(-dq.x), B2<float>::ex2(-dq.y));
                    q[c] = u;
                    s2 = __fadd2_rn(s2, make_float2(sat1(u.x), sat1(u.y)));
                    topx = __funnelshift_l(__float_as_uint(dq.x), topx, 1);
                    topy = __funnelshift_l(__float_as_uint(dq.y), topy, 1);
                }
#pragma unroll
                for (int off = 8; off; off >>= 1)
                    s2 = __fadd2_rn(s2, make_float2(__shfl_xor_sync(kFull, s2.x, off), __shfl_xor_sync(kFull, s2.y, off)));
                const float S = s2.x + s2.y;
                if (r < s) {
                    const float cf = B2<float>::ex2(m2 - m1);
                    const float Aa = __fmaf_rn(cf, S - 1.f, 1.f);
                    float rf = 0.f, dref = 0.f;
                    if constexpr (HALF) {
                        rf = IO::unpack(IO::pack(m1, 0.f)).x;
                        dref = rf - m1;
                    }
                    const float2 ncf = make_float2(-cf, -cf), A2 = make_float2(Aa, Aa);
                    const float2 nm1 = HALF ? make_float2(dref, dref) : make_float2(-m1, -m1);
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const float2 y = __ffma2_rn(ncf, q[c], A2);
                        const float2 out = __ffma2_rn(make_float2(B2<float>::lg2(y.x), B2<float>::lg2(y.y)), neg1, nm1);
                        const int k = 32 * c + 2 * t16;
                        if constexpr (HALF)
                            *reinterpret_cast<unsigned*>(srow + k) = IO::pack(out.x, out.y);
                        else
                            *reinterpret_cast<float2*>(srow + k) = out;
                    }
                    if (topx | topy) {
                        const unsigned top = topx ? topx : topy;
                        const int am = 32 * (CH - 32 + __clz((int)top)) + 2 * t16 + (topx ? 0 : 1);
                        const float lgS = B2<float>::lg2(S - 1.f);
                        if constexpr (HALF)
                            IO::st(srow + am, __fmaf_rn(lgS, -1.f, rf - m2));
                        else
                            srow[am] = -m2 - lgS;
                    }
                    if (((r & 31) >> 1) == t16) {
                        // the diagonal: the message to the boundary variable is kept apart
                        float dv = IO::ld(srow + r);
                        if constexpr (HALF) dv = dv + (-rf);
                        bcast(&dgv[nxt * LD + r], dv);
                        if constexpr (HALF) {
                            IO::st(srow + r, rf);
                            bcast(&nref[nxt * LD + r], -rf);
                        } else {
                            srow[r] = 0.f;
                        }
                    }
                }
                __syncthreads();
                // transposed write of the batch: two columns of four rows per thread
                const int r0 = b * RB;
                const int rows = min(RB, s - r0);
                constexpr int W4 = RB / 4;
                for (int e = tid; e < ((s + 1) >> 1) * W4; e += NTH) {
                    const int kk = e / W4, w = (e - kk * W4) * 4;
                    if (w >= rows) continue;
                    const MS* const sp = stage + (size_t)w * SP + 2 * kk;
                    MS* const d0 = Mn + (size_t)(2 * kk) * LD + r0 + w;
                    if constexpr (HALF) {
                        unsigned v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = w + j < rows ? *reinterpret_cast<const unsigned*>(sp + j * SP) : 0u;
                        *reinterpret_cast<uint2*>(d0) =
                            make_uint2(__byte_perm(v[0], v[1], 0x5410), __byte_perm(v[2], v[3], 0x5410));
                        *reinterpret_cast<uint2*>(d0 + LD) =
                            make_uint2(__byte_perm(v[0], v[1], 0x7632), __byte_perm(v[2], v[3], 0x7632));
                    } else {
                        float2 v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            v[j] = w + j < rows ? *reinterpret_cast<const float2*>(sp + j * SP) : make_float2(0.f, 0.f);
                        *reinterpret_cast<float4*>(d0) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
                        *reinterpret_cast<float4*>(d0 + LD) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
                    }
                }
                // the next batch may overwrite the stage only after this write
                if (b + CL < nbatch) __syncthreads();
            }
            cp_async_wait_all();
            int ok = 0;  // stays 0 without a vote: no judgement
            if (vote) {
                ok = 1;
                if (watching) {
                    __syncwarp();
                    const int r = watch;
                    int cnt = 0;
#pragma unroll 4
                    for (int k = lane; k < s; k += 32) {
                        float own;
                        if constexpr (HALF) {
                            const unsigned v = wown[(warp & 1) * LD + k];
                            const float2 u = IO::unpack(v);
                            own = ((r & 1) ? u.y : u.x) + nrc[r];
                        } else {
                            own = __uint_as_float(wown[(warp & 1) * LD + k]);
                        }
                        float l, x;
                        if constexpr (SH::WBUF) {
                            l = wl[(warp & 1) * LD + k];
                            x = IO::ld(wx + (warp & 1) * LD + k);
                            if constexpr (HALF) x = x + nrc[k];
                        } else {
                            l = prior(r, k);
                            x = msg(r, k);
                        }
                        const float lam = k == r ? l + dgv[cur * LD + r] : l + (own + x);
                        cnt += lam > 0.f ? 1 : 0;
                    }
                    ok = __reduce_add_sync(kFull, cnt) == 1;
                }
            }
            // every block's transposed writes and per-row state precede every read of the next
            // iteration
            ahead = vote_all(ok);
            if (!ahead) {
                cur ^= 1;
                ++t;
            }
        }
        if (tr_on && a.tr_partner) {
            for (int r = tid; r < a.s_cap; r += NTH) {
                int pk = -1;
                if (r < s) pk = out_from_best ? (int)bestp[r] : choice[r];
                a.tr_partner[(size_t)shot * a.s_cap + r] = (int16_t)pk;
            }
        }
        if (tid == 0 && crank == 0) {
            if (ic.obs_pred) ic.obs_pred[shot] = (uint8_t)out_par;
            if (ic.flags)
                ic.flags[shot] = (uint8_t)((any_conv ? F_CONVERGED : 0) | (forced_ran ? F_FORCED_RAN : 0) |
                                          (out_forced ? F_FROM_FORCED : 0));
            if (ic.iters) ic.iters[shot] = (int16_t)t;
            acc_it += (unsigned long long)t;
            acc_msg += (unsigned long long)s * s * t;
            acc_def += (unsigned long long)s;
            acc_shots += 1;
        }
        __syncthreads();
    }
    if (tid == 0 && crank == 0 && a.ctr && acc_shots) {
        atomicAdd(a.ctr + C_ITERS, acc_it);
        atomicAdd(a.ctr + C_MSGS, acc_msg);
        atomicAdd(a.ctr + C_DEFECTS, acc_def);
        atomicAdd(a.ctr + C_TIER_MSGS + a.tier, acc_msg);
        atomicAdd(a.ctr + C_TIER_SHOTS + a.tier, acc_shots);
        atomicAdd(a.ctr + C_FC_RUNS, acc_fc);
        atomicAdd(a.ctr + C_FC_ROUNDS, acc_fcr);
    }
}


template <int CH, typename MS, bool ALONE>
cudaError_t run_wide1(const DecodeArgs& a, int slots, cudaStream_t st) {
    using SH = WideShape<CH, MS, 1, ALONE>;
    auto kern = decode_wide_kernel<CH, MS, 1, ALONE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (e != cudaSuccess) return e;
    kern<<<slots, SH::W * 32, SH::smem, st>>>(a);
    return cudaGetLastError();
}

// One block per shot.  `slots`: blocks, no more than the shots or the resident blocks.
template <int CH, typename MS>
cudaError_t run_wide(const DecodeArgs& a, int slots, int num_sms, cudaStream_t st) {
    if constexpr (wide_blocks(CH, (int)sizeof(MS)) == 2)
        if (slots <= num_sms) return run_wide1<CH, MS, true>(a, slots, st);
    return run_wide1<CH, MS, false>(a, slots, st);
}

// Cluster form: the largest number of clusters of CL blocks that can be resident at once
// on the current device (0 if none), cached per device.
template <int CH, typename MS, int CL>
int wide_cluster_capacity() {
    static_assert(CL > 1, "cluster form");
    constexpr int kDev = 16;
    static std::atomic<int> cache[kDev] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
    if (dev < kDev) {
        const int v = cache[dev].load();
        if (v > 0) return v - 1;
    }
    using SH = WideShape<CH, MS, CL>;
    auto kern = decode_wide_kernel<CH, MS, CL>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem) != cudaSuccess) return 0;
    if (CL > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(SH::W * 32);
    cfg.dynamicSmemBytes = SH::smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    if (dev < kDev) cache[dev].store(n + 1);
    return n;
}

// Launches min(slots, capacity) clusters of CL blocks; the caller's scratch holds `slots`
// slots of WideShape::slot_bytes (one per cluster).
template <int CH, typename MS, int CL>
cudaError_t run_wide_cluster(const DecodeArgs& a, int slots, cudaStream_t st) {
    const int cap = wide_cluster_capacity<CH, MS, CL>();
    if (cap <= 0) return cudaErrorInvalidConfiguration;
    const int clusters = slots < cap ? slots : cap;
    if (clusters <= 0) return cudaSuccess;
    using SH = WideShape<CH, MS, CL>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * CL));
    cfg.blockDim = dim3(SH::W * 32);
    cfg.dynamicSmemBytes = SH::smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, decode_wide_kernel<CH, MS, CL>, a);
}

}  // namespace
}  // namespace bp4m
