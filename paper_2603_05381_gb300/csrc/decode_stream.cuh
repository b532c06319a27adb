#pragma once
// Streaming tier of the BP4M decoder in FP64 (FP32 and 16-bit messages: decode_wide.cuh): shots
// with more unsatisfied detectors than the shared-memory tiers hold, their message matrices in a
// per-block global scratch slot.
//
// One warp owns one factor row at a time (its CH*32 columns in registers).  Slot (LD = 32 CH):
//   Lg[r][k]     prior l_rk in log2 units, -inf for k >= s
//   Mt[b][r][k]  incoming message M[k][r], double buffered (b = iteration parity); diagonal 0, so
//                Q_rr = l_rr and lambda_rr = l_rr + Mo[r][r]
//   Mo[r][k]     the row's own outputs M[r][k], updated in place by the owning warp
// Outputs go to Mt[next][k][r]; a batch of W consecutive rows (one per warp) stages them in
// shared memory and writes W consecutive elements per column k.  Iteration = decision pass
// (lambda of the previous update, convergence vote, candidates / forced convergence), then the
// update pass; BP4M with early exit takes the decisions of all but the last iteration inside
// the update pass that reads the same rows.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "decode_smem.cuh"
#include "device.cuh"

namespace bp4m {
namespace {

constexpr int kStreamWarps = 16;

// Dynamic shared memory of one block: two output stages and the per-row state.
template <int CH>
constexpr size_t stream_smem_bytes() {
    return (size_t)2 * kStreamWarps * (32 * CH + 2) * sizeof(double) +
           (size_t)(32 * CH) * (sizeof(double) + 2 * sizeof(int) + 2 * sizeof(short) + 1) + 32;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
    return v;
}

// Bytes of one slot: priors and three message matrices of LD x LD.
constexpr size_t stream_slot_bytes(int ld) { return (size_t)ld * ld * 4 * sizeof(double); }

template <int CH, bool TRACE>
__global__ void __launch_bounds__(kStreamWarps * 32, 1) decode_stream_kernel(const DecodeArgs a) {
    using T = double;
    constexpr int W = kStreamWarps;
    constexpr int NTH = W * 32;
    constexpr int LD = 32 * CH;
    constexpr int SP = LD + 2;  // output stage pitch
    extern __shared__ __align__(16) unsigned char smem[];
    T* stage0 = reinterpret_cast<T*>(smem);
    double* rowacc = stage0 + 2 * W * SP;
    int* dets = reinterpret_cast<int*>(rowacc + LD);
    int* choice = dets + LD;
    short* bestp = reinterpret_cast<short*>(choice + LD);
    short* order = bestp + LD;  // static-partition forced convergence: factors in processing order
    unsigned char* matched = reinterpret_cast<unsigned char*>(order + LD);
    __shared__ int sh_item, sh_s, sh_best_par, sh_best_forced, sh_improve, sh_use_best;
    __shared__ double sh_best_w;

    const size_t mat = (size_t)LD * LD;
    T* Lg = reinterpret_cast<T*>(a.gscratch) + (size_t)blockIdx.x * 4 * mat;
    T* Mtb[2] = {Lg + mat, Lg + 2 * mat};
    T* Mo = Lg + 3 * mat;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t count = a.count ? (int64_t)*a.count : a.count_val;
    const T ainv = (T)(1.0 / a.alpha);
    const bool full = (a.decoder == 1) || !a.early_exit;
    T* trl = reinterpret_cast<T*>(a.tr_lambda);
    const T ninf = Num<T>::ninf();
    unsigned long long acc_it = 0, acc_msg = 0, acc_def = 0, acc_shots = 0, acc_fc = 0, acc_fcr = 0;

    for (;;) {
        if (tid == 0) sh_item = atomicAdd(a.next, 1);
        __syncthreads();
        const int item = sh_item;
        if (item >= count) break;
        const ItemCtx ic = resolve_item(a, a.list ? (int64_t)a.list[item] : (int64_t)item);
        const int64_t shot = ic.shot;
        const int n = ic.tb.n_det;
        const T* __restrict__ Ltab = Num<T>::L(ic.tb);
        if (warp == 0) {
            const int s0 = compact_defects(ic.synd + (size_t)shot * ic.tb.n_words, ic.tb.n_words, dets, LD, lane);
            if (lane == 0) sh_s = s0;
        }
        __syncthreads();
        const int s = sh_s;
        if (s > LD || s < 2) {
            if (tid == 0 && a.ctr) atomicAdd(a.ctr + C_ERRORS, 1ull);
            continue;
        }
        const bool tr_on = TRACE && s <= a.s_cap;
        for (int r = warp; r < s; r += W) {
            const T* trow = Ltab + (size_t)dets[r] * n;
            for (int k = lane; k < LD; k += 32) {
                Lg[(size_t)r * LD + k] = k < s ? (T)(__ldg(trow + dets[k]) * (T)kLog2e) : ninf;
                Mtb[0][(size_t)r * LD + k] = T(0);
                Mtb[1][(size_t)r * LD + k] = T(0);
                Mo[(size_t)r * LD + k] = T(0);
            }
        }
        for (int r = tid; r < LD; r += NTH) {
            matched[r] = r >= s;
            bestp[r] = -1;
        }
        if (tid == 0) {
            sh_best_w = Num<double>::pinf();
            sh_best_par = 0;
            sh_best_forced = 0;
            sh_use_best = 0;
        }
        __syncthreads();

        int cur = 0;
        int t = 0;
        bool any_conv = false, forced_ran = false;
        int out_par = 0, out_forced = 0, out_from_best = 0;

        // BP4M with early exit: the decisions of lambda^t are taken inside the update pass that
        // reads the same rows; only the last iteration, which may need forced convergence, keeps
        // the separate decision pass
        const bool merged = !TRACE && a.decoder == 0 && a.early_exit;
        for (;;) {
            const T* Mc = Mtb[cur];
            const bool fuse = merged && t > 0 && t < a.T;
            if (t > 0 && !fuse) {
                // ---- decisions of lambda^t = l + (M[r][k] + M[k][r])
                int ok_all = 1;
                for (int r = warp; r < s; r += W) {
                    const T* lrow = Lg + (size_t)r * LD;
                    const T* xrow = Mc + (size_t)r * LD;
                    const T* orow = Mo + (size_t)r * LD;
                    // kept count and a kept column of the row (the only one when the count is 1,
                    // the case in which it is used: otherwise forced convergence replaces it)
                    int cnt = 0, kl = -1;
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int k = lane + 32 * c;
                        const T lam = lrow[k] + (orow[k] + xrow[k]);
                        const bool kp = lam > T(0);
                        cnt += kp ? 1 : 0;
                        kl = kp ? k : kl;
                        if (tr_on && trl && k < s) trl[((size_t)shot * a.s_cap + r) * a.s_cap + k] = lam * (T)kLn2;
                    }
#pragma unroll
                    for (int off = 16; off; off >>= 1) {
                        cnt += __shfl_xor_sync(kFull, cnt, off);
                        kl = max(kl, __shfl_xor_sync(kFull, kl, off));
                    }
                    if (lane == 0) choice[r] = kl >= 0 ? kl : 0x7fffffff;
                    ok_all &= (cnt == 1);
                }
                const int conv = __syncthreads_and(ok_all);
                bool have_cand = false, cand_forced = false;
                if (conv) {
                    any_conv = true;
                    have_cand = true;
                } else if (a.decoder == 1 || t == a.T) {
                    // ---- forced convergence on lambda^t by locally dominant rounds
                    forced_ran = true;
                    for (int r = tid; r < s; r += NTH) matched[r] = 0;
                    __syncthreads();
                    if (a.forced_static) {
                        // the paper's static partition: row r's block is v_rk, k >= r; its
                        // maximum (ties: smaller k) represents factor r; representatives are
                        // ranked by posterior (ties: smaller r) and processed in that order
                        for (int r = warp; r < s; r += W) {
                            const T* lrow = Lg + (size_t)r * LD;
                            const T* xrow = Mc + (size_t)r * LD;
                            const T* orow = Mo + (size_t)r * LD;
                            T bl = ninf;
                            int bk = 0x7fffffff;
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int k = lane + 32 * c;
                                if (k >= r && k < s) {
                                    const T lam = lrow[k] + (orow[k] + xrow[k]);
                                    if (bk == 0x7fffffff || lam > bl) {
                                        bl = lam;
                                        bk = k;
                                    }
                                }
                            }
#pragma unroll
                            for (int off = 16; off; off >>= 1) {
                                const T ol = __shfl_xor_sync(kFull, bl, off);
                                const int okk = __shfl_xor_sync(kFull, bk, off);
                                if (okk != 0x7fffffff && (bk == 0x7fffffff || ol > bl || (ol == bl && okk < bk))) {
                                    bl = ol;
                                    bk = okk;
                                }
                            }
                            if (lane == 0) {
                                choice[r] = bk != 0x7fffffff ? bk : r;
                                rowacc[r] = (double)bl;
                            }
                        }
                        __syncthreads();
                        for (int r = tid; r < s; r += NTH) {
                            const double v = rowacc[r];
                            int rank = 0;
                            for (int j = 0; j < s; ++j) {
                                const double u = rowacc[j];
                                rank += (u > v || (u == v && j < r)) ? 1 : 0;
                            }
                            order[rank] = (short)r;
                        }
                        __syncthreads();
                        if (tid == 0) {
                            // a factor whose representative's other factor is taken goes to the
                            // boundary (a case the paper does not treat)
                            for (int q = 0; q < s; ++q) {
                                const int rr = order[q];
                                if (matched[rr]) continue;
                                const int k = choice[rr];
                                matched[rr] = 1;
                                if (k == rr || matched[k]) {
                                    choice[rr] = rr;
                                } else {
                                    matched[k] = 1;
                                    choice[k] = rr;
                                }
                            }
                            acc_fcr += 1;
                        }
                        __syncthreads();
                    }
                    for (int round = 0; round < s && !a.forced_static; ++round) {
                        for (int r = warp; r < s; r += W) {
                            if (matched[r]) continue;  // uniform per warp
                            const T* lrow = Lg + (size_t)r * LD;
                            const T* xrow = Mc + (size_t)r * LD;
                            const T* orow = Mo + (size_t)r * LD;
                            T bl = ninf;
                            int bk = 0x7fffffff;
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int k = lane + 32 * c;
                                if (k < s && (k == r || !matched[k])) {
                                    const T lam = lrow[k] + (orow[k] + xrow[k]);
                                    if (bk == 0x7fffffff || lam > bl) {
                                        bl = lam;
                                        bk = k;
                                    }
                                }
                            }
#pragma unroll
                            for (int off = 16; off; off >>= 1) {
                                const T ol = __shfl_xor_sync(kFull, bl, off);
                                const int okk = __shfl_xor_sync(kFull, bk, off);
                                if (okk != 0x7fffffff && (bk == 0x7fffffff || ol > bl || (ol == bl && okk < bk))) {
                                    bl = ol;
                                    bk = okk;
                                }
                            }
                            if (lane == 0) choice[r] = bk != 0x7fffffff ? bk : r;
                        }
                        __syncthreads();
                        int left = 0;
                        for (int r = tid; r < s; r += NTH) {
                            if (matched[r]) continue;
                            const int pk = choice[r];
                            const bool newm = (pk == r) || (choice[pk] == r);
                            rowacc[r] = newm ? 1.0 : 0.0;
                            left += !newm;
                        }
                        __syncthreads();
                        for (int r = tid; r < s; r += NTH)
                            if (!matched[r] && rowacc[r] != 0.0) matched[r] = 1;
                        if (tid == 0) acc_fcr += 1;
                        const int left_all = __syncthreads_count(left);
                        if (left_all == 0) break;
                    }
                    if (tid == 0) acc_fc += 1;
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
                __syncthreads();
            }
            // ---- update pass: M' for every row, batch by batch
            T* Mn = Mtb[cur ^ 1];
            const int nbatch = (s + W - 1) / W;
            int ok_w = 1;  // fused decisions: every row of this warp keeps exactly one variable
            for (int b = 0; b < nbatch; ++b) {
                const int r = b * W + warp;
                T* const stage = stage0 + (b & 1) * W * SP;
                T* srow = stage + warp * SP;
                if (r < s) {
                    const T* lrow = Lg + (size_t)r * LD;
                    const T* xrow = Mc + (size_t)r * LD;
                    T* orow = Mo + (size_t)r * LD;
                    // one pass over the row: Q = l + M[k][r]/alpha and its maximum, second
                    // maximum and argmax; with the fused decisions also the kept count of
                    // lambda^t = l + (M[r][k] + M[k][r]) and a kept column (the only one when
                    // the count is 1, the case in which it is used)
                    T q[CH];
                    T m1 = ninf, m2 = ninf;
                    int am = 0x7fffffff;
                    int cnt = 0, kl = -1;
                    auto row_pass = [&](auto fused) {
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            q[c] = ninf;
                            if (32 * c >= s) continue;  // past s in every lane: would add exactly 0
                            const int k = lane + 32 * c;
                            const T lv = lrow[k], xv = xrow[k];
                            if constexpr (decltype(fused)::value) {
                                const T lam = lv + (orow[k] + xv);
                                const bool kp = lam > T(0);
                                cnt += kp ? 1 : 0;
                                kl = kp ? k : kl;
                            }
                            const T v = B2<T>::fma_(xv, ainv, lv);
                            q[c] = v;
                            const bool gt = v > m1;
                            m2 = B2<T>::mx(m2, B2<T>::mn(v, m1));
                            m1 = B2<T>::mx(m1, v);
                            am = gt ? k : am;
                        }
                    };
                    if (fuse)
                        row_pass(std::true_type{});
                    else
                        row_pass(std::false_type{});
#pragma unroll
                    for (int off = 16; off; off >>= 1) {
                        const T o1 = __shfl_xor_sync(kFull, m1, off);
                        const T o2 = __shfl_xor_sync(kFull, m2, off);
                        const int ok = __shfl_xor_sync(kFull, am, off);
                        combine_max(m1, m2, am, o1, o2, ok);
                    }
                    if (fuse) {
#pragma unroll
                        for (int off = 16; off; off >>= 1) {
                            cnt += __shfl_xor_sync(kFull, cnt, off);
                            kl = max(kl, __shfl_xor_sync(kFull, kl, off));
                        }
                        if (lane == 0) choice[r] = kl >= 0 ? kl : 0x7fffffff;
                        ok_w &= (cnt == 1);
                    }
                    T S = T(0);
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        if (32 * c >= s) continue;
                        const T u = B2<T>::ex2(B2<T>::mn(q[c], m2) - m2);
                        q[c] = u;
                        S += u;
                    }
                    S = warp_sum(S);
                    const T cf = B2<T>::ex2(m2 - m1);
                    const T Aa = B2<T>::fma_(cf, S - T(1), T(1));
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            if (32 * c >= s) continue;
                            const int k = lane + 32 * c;
                            const T out = -m1 - B2<T>::lg2(B2<T>::fma_(-cf, q[c], Aa));
                            orow[k] = out;
                            srow[k] = out;
                        }
                        if ((am & 31) == lane) {
                            const T oam = -m2 - B2<T>::lg2(S - T(1));
                            orow[am] = oam;
                            srow[am] = oam;
                        }
                        __syncwarp();
                        if (lane == 0) srow[r] = T(0);  // the diagonal of Mt stays 0
                }
                __syncthreads();
                // transposed write of the batch: Mn[k][b*W + w] = stage[w][k]
                const int r0 = b * W;
                const int rows = min(W, s - r0);
                // (two stages: the next batch writes the other one, and the barrier after its rows
                // protects this one)
                for (int e = tid; e < s * W; e += NTH) {
                    const int k = e / W, w = e % W;
                    if (w < rows) Mn[(size_t)k * LD + r0 + w] = stage[w * SP + k];
                }
            }
            __syncthreads();  // the last batch's transposed write precedes every read of Mn
            const int fconv = fuse && __syncthreads_and(ok_w);
            if (fconv) {
                // lambda^t converged: its matching is the output (the update just made is unused)
                any_conv = true;
                int pc = 0;
                for (int r = tid; r < s; r += NTH) {
                    const int k = choice[r];
                    if (k >= r) pc ^= ic.tb.P[(size_t)dets[r] * n + dets[k]];
                }
                out_par = __syncthreads_count(pc) & 1;
                out_forced = 0;
                break;
            }
            cur ^= 1;
            ++t;
        }
        if (tr_on && a.tr_partner) {
            for (int r = tid; r < a.s_cap; r += NTH) {
                int pk = -1;
                if (r < s) pk = out_from_best ? (int)bestp[r] : choice[r];
                a.tr_partner[(size_t)shot * a.s_cap + r] = (int16_t)pk;
            }
        }
        if (tid == 0) {
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
    if (tid == 0 && a.ctr) {
        atomicAdd(a.ctr + C_ITERS, acc_it);
        atomicAdd(a.ctr + C_MSGS, acc_msg);
        atomicAdd(a.ctr + C_DEFECTS, acc_def);
        atomicAdd(a.ctr + C_TIER_MSGS + a.tier, acc_msg);
        atomicAdd(a.ctr + C_TIER_SHOTS + a.tier, acc_shots);
        atomicAdd(a.ctr + C_FC_RUNS, acc_fc);
        atomicAdd(a.ctr + C_FC_ROUNDS, acc_fcr);
    }
}

template <int CH>
cudaError_t run_stream(const DecodeArgs& a, int slots, cudaStream_t st) {
    const size_t smem = stream_smem_bytes<CH>();
    const bool tr = a.tr_lambda != nullptr || a.tr_partner != nullptr;
    auto kern = tr ? decode_stream_kernel<CH, true> : decode_stream_kernel<CH, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<slots, kStreamWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace
}  // namespace bp4m
