#pragma once
// BP4M / BP4MF decoding of small shots, several per warp (FP32 arithmetic, s <= 32).
//
// Same factor graph, update, decisions and forced convergence as decode_smem.cuh, for shots of
// at most 32 unsatisfied detectors: LG lanes of a warp own one shot, one row (factor) per lane,
// with CH columns in registers (CH >= s), so a warp decodes 32 / LG shots at once and no block
// barrier is needed.  Every FP32 result equals decode_smem.cuh's one-thread-per-row form bit for
// bit: a row's exponentials are added in the same order (even and odd columns apart, ascending,
// then the two sums), and the columns a narrower form leaves out would have added exactly 0.
//
// Why: one 32-lane warp per shot padded to 32 columns spent (32 / s)^2 times the work a shot of
// s defects needs (16 x at the s = 8 of a d = 9 code-capacity shot at p = 0.10), and these
// shots are the bulk of the code-capacity sweep and of circuits at low p.  Bound by
// instruction issue; the message matrix stays in shared memory only because rows meet columns.
// Measured with the lists of 8, 16, 24 and 32 rows against one 32-row list (a call of
// sample_and_decode): 10^6 d = 9 code-capacity shots at p = 0.10 15.9 -> 4.3 ms, 10^6 d = 7 circuit
// shots at p = 0.002 7.1 -> 2.9 ms.
//
// A warp takes `chunk` items of the list at a time and hands them to its groups as they finish
// (early exits leave the groups of a warp at different iterations); a group without a shot idles.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "decode_smem.cuh"
#include "device.cuh"

namespace bp4m {
namespace {

constexpr int kSmallWarps = 4;

// Shared memory of one warp.  Row pitch P = CH + 4 elements: the quarter-warp 16-byte row reads
// (FP32; half-warp 8-byte reads with 16-bit messages) start in distinct bank groups, and a
// transposed write or read has consecutive lanes in consecutive elements.  Groups are padded so
// that their transposed writes do not meet in the same banks.
template <int LG, int CH, typename MS>
struct SmallShape {
    static constexpr int NG = 32 / LG;
    static constexpr int P = CH + 4;
    static constexpr bool LREG = LG < 32;  // priors in registers, else in shared memory
    static constexpr bool HALF = sizeof(MS) == 2;
    static constexpr int GS = CH * P + (LG == 8 ? 8 : LG == 16 ? 16 : 0);
    static constexpr int mt_bytes = (NG * GS * (int)sizeof(MS) + 15) / 16 * 16;
    static constexpr int lm_bytes = LREG ? 0 : CH * P * 4;
    static constexpr int ref_bytes = HALF ? NG * CH * 4 : 0;
    static constexpr int det_bytes = NG * CH * 4;
    static constexpr int warp_bytes = (mt_bytes + lm_bytes + ref_bytes + det_bytes + 15) / 16 * 16;
    static constexpr int block_bytes = kSmallWarps * warp_bytes;
};

// Blocks of kSmallWarps warps per SM the kernel is compiled for (registers).
constexpr int small_blocks(int lg) { return lg == 8 ? 8 : lg == 16 ? 6 : 5; }

template <int LG, int CH, typename MS, bool TRACE>
__global__ void __launch_bounds__(kSmallWarps * 32, small_blocks(LG)) decode_small_kernel(const DecodeArgs a) {
    using SH = SmallShape<LG, CH, MS>;
    using IO = MsgIO<MS, float>;
    constexpr bool HALF = SH::HALF;
    constexpr bool LREG = SH::LREG;
    constexpr int NG = SH::NG;
    constexpr int P = SH::P;
    static_assert(CH % 4 == 0 && CH <= LG, "columns in blocks of four, one lane per row");
    extern __shared__ __align__(16) unsigned char smem_small[];
    __shared__ unsigned long long sh_acc[kSmallWarps][NG][6];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = lane % LG;          // row of this lane in its shot
    const int gb = lane - i;          // first lane of the group
    const int grp = gb / LG;
    const unsigned gbits = LG == 32 ? kFull : ((1u << (LG & 31)) - 1u);
    unsigned char* const wbase = smem_small + warp * SH::warp_bytes;
    MS* const Mt = reinterpret_cast<MS*>(wbase) + grp * SH::GS;  // Mt[i][k] = M[k][i]; diagonal 0 (16-bit: r_i)
    float* const Lm = reinterpret_cast<float*>(wbase + SH::mt_bytes);
    float* const nref = reinterpret_cast<float*>(wbase + SH::mt_bytes + SH::lm_bytes) + grp * CH;  // 16-bit: -r_k
    int* const dets = reinterpret_cast<int*>(wbase + SH::mt_bytes + SH::lm_bytes + SH::ref_bytes) + grp * CH;
    unsigned long long* const acc = sh_acc[warp][grp];  // iterations, updates, defects, shots, forced runs, rounds
    if (i < 6) acc[i] = 0;
    __syncwarp();

    const int count = *a.count;
    const float ainv = (float)(1.0 / a.alpha);
    const float2 ainv2 = make_float2(ainv, ainv);
    const bool full = (a.decoder == 1) || !a.early_exit;
    const float ninf = Num<float>::ninf();
    float* const trl = reinterpret_cast<float*>(a.tr_lambda);
    // items a warp takes at once: few enough that every warp of the launch gets some
    int chunk = count / (int)(gridDim.x * kSmallWarps * 4);
    chunk = chunk < 1 ? 1 : chunk > 32 ? 32 : chunk;

    int chunk_pos = 0, chunk_n = 0, chunk_item = 0;
    bool exhausted = false;
    // the group's shot
    bool live = false;
    int code = 0, s = 0, t = 0;
    float dg = 0.f;       // M[i][i], this row's message to its boundary variable
    float lii = ninf;     // its prior
    float lr[LREG ? CH : 1] = {};
    bool any_conv = false, forced_ran = false;
    // candidates (BP4MF, full-T mode): the lightest so far and this row's partner in it
    double best_w = 0.0;
    int best_par = 0, best_forced = 0, bestp = -1;
    int watch = 0;  // LG == 32: the row watched for the convergence decision

    // priors and messages of this lane's row
    auto L4 = [&](int j) -> float4 {
        if constexpr (LREG)
            return make_float4(lr[4 * j], lr[4 * j + 1], lr[4 * j + 2], lr[4 * j + 3]);
        else
            return *reinterpret_cast<const float4*>(Lm + i * P + 4 * j);
    };
    auto L1 = [&](int c) -> float {
        if constexpr (LREG)
            return lr[c];
        else
            return Lm[i * P + c];
    };
    auto X4 = [&](int j) -> float4 {  // M[4j .. 4j+3][i]
        if constexpr (HALF) {
            const uint2 r = *reinterpret_cast<const uint2*>(Mt + i * P + 4 * j);
            const float4 n = *reinterpret_cast<const float4*>(nref + 4 * j);
            const float2 lo = __fadd2_rn(IO::unpack(r.x), make_float2(n.x, n.y));
            const float2 hi = __fadd2_rn(IO::unpack(r.y), make_float2(n.z, n.w));
            return make_float4(lo.x, lo.y, hi.x, hi.y);
        } else {
            return *reinterpret_cast<const float4*>(Mt + i * P + 4 * j);
        }
    };
    auto msg = [&](int to, int from) -> float {  // M[from][to]
        if constexpr (HALF)
            return IO::ld(Mt + to * P + from) + nref[from];
        else
            return IO::ld(Mt + to * P + from);
    };

    for (;;) {
        // ---- refill: an item for every group without a shot
        unsigned need = __ballot_sync(kFull, !live);
        while (need && !exhausted) {
            if (chunk_pos >= chunk_n) {
                int b = 0;
                if (lane == 0) b = atomicAdd(a.next, chunk);
                b = __shfl_sync(kFull, b, 0);
                chunk_n = min(chunk, count - b);
                chunk_pos = 0;
                if (chunk_n <= 0) {
                    exhausted = true;
                    break;
                }
                if (lane < chunk_n) chunk_item = a.list[(int64_t)(b + lane) * a.list_dir];
            }
            const int rank = __popc(need & ((1u << gb) - 1u)) / LG;
            const int take = min(__popc(need) / LG, chunk_n - chunk_pos);
            const int it = __shfl_sync(kFull, chunk_item, (chunk_pos + rank) & 31);
            const bool got = !live && rank < take;
            chunk_pos += take;
            if (got) code = it;
            ItemCtx ic{};
            if (got) ic = resolve_item(a, code);
            // sorted list of the shot's unsatisfied detectors
            const int nw = got ? ic.tb.n_words : 0;
            const uint32_t* sw = got ? ic.synd + (size_t)ic.shot * nw : nullptr;
            int base = 0;
            for (int w0 = 0; __any_sync(kFull, w0 < nw); w0 += LG) {
                uint32_t word = w0 + i < nw ? __ldg(sw + w0 + i) : 0u;
                const int c = __popc(word);
                int incl = c;
#pragma unroll
                for (int off = 1; off < LG; off <<= 1) {
                    const int y = __shfl_up_sync(kFull, incl, off, LG);
                    if (i >= off) incl += y;
                }
                int pos = base + incl - c;
                while (word) {
                    const int b = __ffs(word) - 1;
                    word &= word - 1;
                    if (pos < CH) dets[pos] = (w0 + i) * 32 + b;
                    ++pos;
                }
                base += __shfl_sync(kFull, incl, LG - 1, LG);
            }
            __syncwarp();
            if (got) {
                s = base;
                const int n = ic.tb.n_det;
                if (s > CH || s < 1) {
                    if (i == 0 && a.ctr) atomicAdd(a.ctr + C_ERRORS, 1ull);
                } else if (s == 1) {
                    // a single factor with a single variable: the leave-one-out set is empty, the
                    // message is +inf and v_00 is kept in every iteration
                    const int its = full ? a.T : 1;
                    const bool tr_on = TRACE && s <= a.s_cap;
                    if (i == 0) {
                        const int d0 = dets[0];
                        if (ic.obs_pred) ic.obs_pred[ic.shot] = ic.tb.P[(size_t)d0 * n + d0];
                        if (ic.flags) ic.flags[ic.shot] = F_CONVERGED;
                        if (ic.iters) ic.iters[ic.shot] = (int16_t)its;
                        if (tr_on && trl) trl[(size_t)ic.shot * a.s_cap * a.s_cap] = Num<float>::pinf();
                        if (tr_on && a.tr_partner) {
                            a.tr_partner[(size_t)ic.shot * a.s_cap] = 0;
                            for (int k = 1; k < a.s_cap; ++k) a.tr_partner[(size_t)ic.shot * a.s_cap + k] = -1;
                        }
                        acc[0] += (unsigned long long)its;
                        acc[1] += (unsigned long long)its;
                        acc[2] += 1;
                        acc[3] += 1;
                    }
                } else {
                    // ---- the shot's priors (log2 units); columns past s are -inf, so that they never
                    // win a maximum, add nothing to a sum and are never kept
                    live = true;
                    t = 0;
                    any_conv = forced_ran = false;
                    best_w = Num<double>::pinf();
                    best_par = best_forced = 0;
                    bestp = -1;
                    watch = 0;
                    dg = 0.f;
                    lii = ninf;
                    if (i < CH) {
                        const float* trow = i < s ? ic.tb.L32 + (size_t)dets[i] * n : nullptr;
                        if (i < s) lii = __ldg(trow + dets[i]) * (float)kLog2e;
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            const float l = (i < s && c < s) ? __ldg(trow + dets[c]) * (float)kLog2e : ninf;
                            if constexpr (LREG)
                                lr[c] = l;
                            else
                                Lm[i * P + c] = l;
                            Mt[i * P + c] = MS(0.f);
                        }
                        if constexpr (HALF) nref[i] = 0.f;
                    }
                }
            }
            __syncwarp();
            need = __ballot_sync(kFull, !live);
        }
        if (!__any_sync(kFull, live)) break;

        const bool act = live && i < s;
        // ---- Q = l + M[k][i] / alpha, and the row's maximum and second maximum
        float2 q[CH / 2];
        float m1 = ninf, m2 = ninf;
        float2 cnt2 = make_float2(0.f, 0.f);
        if (act) {
#pragma unroll
            for (int j = 0; j < CH / 4; ++j) {
                const float4 l = L4(j), x = X4(j);
                const float2 l0 = make_float2(l.x, l.y), l1 = make_float2(l.z, l.w);
                const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
                const float2 p0 = __ffma2_rn(x0, ainv2, l0), p1 = __ffma2_rn(x1, ainv2, l1);
                q[2 * j] = p0;
                q[2 * j + 1] = p1;
                const float h0 = fmaxf(p0.x, p0.y), n0 = fminf(p0.x, p0.y);
                const float h1 = fmaxf(p1.x, p1.y), n1 = fminf(p1.x, p1.y);
                const float hi = fmaxf(h0, h1), lo = max3f(n0, n1, fminf(h0, h1));
                m2 = max3f(m2, lo, fminf(m1, hi));
                m1 = fmaxf(m1, hi);
                if constexpr (LREG) {
                    // kept variables of lambda^t = l + (M[i][k] + M[k][i]); for k == i both messages
                    // read as 0 here and the boundary variable's count is corrected below
                    const float2 o0 = make_float2(msg(4 * j, i), msg(4 * j + 1, i));
                    const float2 o1 = make_float2(msg(4 * j + 2, i), msg(4 * j + 3, i));
                    const float2 y0 = __fadd2_rn(l0, __fadd2_rn(o0, x0)), y1 = __fadd2_rn(l1, __fadd2_rn(o1, x1));
                    cnt2 = __fadd2_rn(cnt2, make_float2(y0.x > 0.f ? 1.f : 0.f, y0.y > 0.f ? 1.f : 0.f));
                    cnt2 = __fadd2_rn(cnt2, make_float2(y1.x > 0.f ? 1.f : 0.f, y1.y > 0.f ? 1.f : 0.f));
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) q[j] = make_float2(ninf, ninf);
        }
        if (TRACE && act && t > 0 && trl && s <= a.s_cap) {
            const ItemCtx ic = resolve_item(a, code);
            for (int k = 0; k < s; ++k) {
                float l = 0.f;
#pragma unroll
                for (int c = 0; c < CH; ++c)
                    if (c == k) l = L1(c);
                const float lam = k == i ? l + dg : l + (msg(k, i) + msg(i, k));
                trl[((size_t)ic.shot * a.s_cap + i) * a.s_cap + k] = lam * (float)kLn2;
            }
        }
        // ---- convergence: every row keeps exactly one variable
        bool conv;
        if constexpr (LREG) {
            float cnt = cnt2.x + cnt2.y;
            cnt += (lii + dg > 0.f ? 1.f : 0.f) - (lii > 0.f ? 1.f : 0.f);
            const unsigned bad = __ballot_sync(kFull, act && cnt != 1.f);
            conv = live && t > 0 && ((bad >> gb) & gbits) == 0u;
        } else {
            // one watched row decides most iterations; every row is counted when it keeps one
            conv = live && t > 0;
            if (conv) {
                const int k = lane < CH ? lane : CH - 1;
                const float l = Lm[watch * P + k];
                const float dgw = __shfl_sync(kFull, dg, watch);
                const float lam = k == watch ? l + dgw : l + (msg(k, watch) + msg(watch, k));
                conv = __popc(__ballot_sync(kFull, lane < s && lam > 0.f)) == 1;
            }
            if (conv) {
                int cnt = 0;
                if (act) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const float l = L1(c);
                        const float lam = c == i ? l + dg : l + (msg(c, i) + msg(i, c));
                        cnt += lam > 0.f ? 1 : 0;
                    }
                }
                const unsigned bad = __ballot_sync(kFull, act && cnt != 1);
                conv = bad == 0u;
                if (!conv) watch = __ffs((int)bad) - 1;
            }
        }
        // ---- candidates
        const bool cand = live && t > 0 && (conv || a.decoder == 1 || t == a.T);
        if (__any_sync(kFull, cand)) {
            int choice = -1;
            if (conv) {
                any_conv = true;
                // the only kept variable of the row
                if (act) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const float l = L1(c);
                        const float lam = c == i ? l + dg : l + (msg(c, i) + msg(i, c));
                        if (lam > 0.f) choice = c;
                    }
                }
            }
            const bool fneed = cand && !conv;
            if (__any_sync(kFull, fneed)) {
                if (fneed) forced_ran = true;
                if (a.forced_static) {
                    // the paper's static partition: row i's block is v_ik, k >= i; its maximum (ties:
                    // smaller k) represents factor i; representatives are processed by posterior
                    // (ties: smaller i); a factor whose representative's other factor is taken goes to
                    // the boundary
                    float bl = ninf;
                    int bk = -1;
                    if (fneed && act) {
#pragma unroll
                        for (int c = 0; c < CH; ++c)
                            if (c >= i && c < s) {
                                const float lam = c == i ? lii + dg : L1(c) + (msg(c, i) + msg(i, c));
                                if (bk < 0 || lam > bl) {
                                    bl = lam;
                                    bk = c;
                                }
                            }
                        choice = bk >= 0 ? bk : i;
                    }
                    int rank = 0;
                    for (int j = 0; j < LG; ++j) {
                        const float u = __shfl_sync(kFull, bl, j, LG);
                        if (j < s) rank += (u > bl || (u == bl && j < i)) ? 1 : 0;
                    }
                    unsigned taken = 0;
                    for (int r = 0; __any_sync(kFull, fneed && r < s); ++r) {
                        const unsigned who = (__ballot_sync(kFull, fneed && act && rank == r) >> gb) & gbits;
                        const int ii = who ? __ffs((int)who) - 1 : 0;
                        const int k = __shfl_sync(kFull, choice, ii, LG);
                        if (fneed && r < s && who && !((taken >> ii) & 1u)) {
                            taken |= 1u << ii;
                            if (k == ii || ((taken >> k) & 1u)) {
                                if (i == ii) choice = ii;
                            } else {
                                taken |= 1u << k;
                                if (i == k) choice = ii;
                            }
                        }
                    }
                    if (fneed && i == 0) acc[5] += 1;
                } else {
                    // greedy matching by rounds of locally dominant choices (see decode_smem.cuh).  A
                    // row whose choice is still unmatched keeps it: the best of a set that has only
                    // shrunk around it.
                    unsigned avail = fneed ? (s == 32 ? kFull : (1u << s) - 1u) : 0u;
                    for (int round = 0; __any_sync(kFull, avail != 0u && round < s); ++round) {
                        const bool run = avail != 0u && round < s;
                        const bool open = run && act && ((avail >> i) & 1u);
                        const bool scan = open && (round == 0 || !((avail >> choice) & 1u));
                        if (scan) {
                            float bl = ninf;
                            int bk = -1;
#pragma unroll
                            for (int c = 0; c < CH; ++c)
                                if ((avail >> c) & 1u) {
                                    const float lam = c == i ? lii + dg : L1(c) + (msg(c, i) + msg(i, c));
                                    if (bk < 0 || lam > bl) {
                                        bl = lam;
                                        bk = c;
                                    }
                                }
                            choice = bk >= 0 ? bk : i;
                        }
                        const int pk = __shfl_sync(kFull, choice, open ? choice : 0, LG);
                        const unsigned newm = (__ballot_sync(kFull, open && (choice == i || pk == i)) >> gb) & gbits;
                        if (run) {
                            avail &= ~newm;
                            if (i == 0) acc[5] += 1;
                        }
                    }
                }
                if (fneed && i == 0) acc[4] += 1;
            }
            // candidate parity (and weight when candidates are compared)
            ItemCtx ic{};
            if (cand) ic = resolve_item(a, code);
            int pc = 0;
            double w = 0.0;
            if (cand && act && choice >= i) {
                const size_t off = (size_t)dets[i] * ic.tb.n_det + dets[choice];
                pc = ic.tb.P[off];
                if (full) w = ic.tb.W64[off];
            }
            const int par = __popc((__ballot_sync(kFull, pc != 0) >> gb) & gbits) & 1;
            bool finish = cand && !full;
            int out_par = par, out_forced = cand && !conv, out_p = choice;
            if (full) {
                double ws = 0.0;
                for (int r = 0; r < CH; ++r) {
                    const double wr = __shfl_sync(kFull, w, r, LG);
                    if (r < s) ws += wr;
                }
                if (cand) {
                    bool use_best = false;
                    if (a.decoder == 1 || conv) {
                        if (ws < best_w) {
                            best_w = ws;
                            best_par = par;
                            best_forced = !conv;
                            bestp = choice;
                        }
                    } else {
                        use_best = best_w <= ws;
                    }
                    if (t == a.T || (a.decoder == 0 && !conv)) {
                        finish = true;
                        if (!(a.decoder == 0 && !conv && !use_best)) {
                            out_par = best_par;
                            out_forced = best_forced;
                            out_p = bestp;
                        }
                    }
                }
            }
            if (finish) {
                if (TRACE && a.tr_partner && s <= a.s_cap) {
                    if (act) a.tr_partner[(size_t)ic.shot * a.s_cap + i] = (int16_t)out_p;
                    for (int k = s + i; k < a.s_cap; k += LG) a.tr_partner[(size_t)ic.shot * a.s_cap + k] = -1;
                }
                if (i == 0) {
                    if (ic.obs_pred) ic.obs_pred[ic.shot] = (uint8_t)out_par;
                    if (ic.flags)
                        ic.flags[ic.shot] = (uint8_t)((any_conv ? F_CONVERGED : 0) | (forced_ran ? F_FORCED_RAN : 0) |
                                                      (out_forced ? F_FROM_FORCED : 0));
                    if (ic.iters) ic.iters[ic.shot] = (int16_t)t;
                    acc[0] += (unsigned long long)t;
                    acc[1] += (unsigned long long)s * s * t;
                    acc[2] += (unsigned long long)s;
                    acc[3] += 1;
                }
                live = false;
            }
        }
        __syncwarp();  // every read of Mt precedes the writes below
        // ---- leave-one-out max* of every row, in place (see decode_smem.cuh)
        if (live && i < s) {
            const float2 m22 = make_float2(m2, m2), neg1 = make_float2(-1.f, -1.f);
            float2 s2 = make_float2(0.f, 0.f);
            unsigned top = 0;  // the column above m2, first column in the highest of CH bits
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) {
                const float2 dq = __ffma2_rn(q[j], neg1, m22);
                const float2 u = make_float2(B2<float>::ex2(-dq.x), B2<float>::ex2(-dq.y));
                q[j] = u;
                s2 = __fadd2_rn(s2, make_float2(sat1(u.x), sat1(u.y)));
                top = __funnelshift_l(__float_as_uint(dq.x), top, 1);
                top = __funnelshift_l(__float_as_uint(dq.y), top, 1);
            }
            const float S = s2.x + s2.y;
            const float cf = B2<float>::ex2(m2 - m1);
            const float A = __fmaf_rn(cf, S - 1.f, 1.f);
            float rf = 0.f, dref = 0.f;
            if constexpr (HALF) {
                rf = IO::unpack(IO::pack(m1, 0.f)).x;
                dref = rf - m1;
            }
            const float2 ncf = make_float2(-cf, -cf), A2 = make_float2(A, A);
            const float2 nm1 = HALF ? make_float2(dref, dref) : make_float2(-m1, -m1);
            MS* const col = Mt + i;
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) {
                const float2 y = __ffma2_rn(ncf, q[j], A2);
                const float2 out = __ffma2_rn(make_float2(B2<float>::lg2(y.x), B2<float>::lg2(y.y)), neg1, nm1);
                if constexpr (HALF) {
                    const unsigned pk2 = IO::pack(out.x, out.y);
                    *reinterpret_cast<unsigned short*>(col + 2 * j * P) = (unsigned short)(pk2 & 0xFFFFu);
                    *reinterpret_cast<unsigned short*>(col + (2 * j + 1) * P) = (unsigned short)(pk2 >> 16);
                } else {
                    col[2 * j * P] = out.x;
                    col[(2 * j + 1) * P] = out.y;
                }
            }
            if (top) {
                const int am = CH - 32 + __clz((int)top);
                const float lgS = B2<float>::lg2(S - 1.f);
                if constexpr (HALF)
                    IO::st(col + am * P, __fmaf_rn(lgS, -1.f, rf - m2));
                else
                    col[am * P] = -m2 - lgS;
            }
            if constexpr (HALF) {
                dg = IO::ld(col + i * P) + (-rf);
                IO::st(col + i * P, rf);  // the diagonal holds r_i, which decodes to exactly 0
                nref[i] = -rf;
            } else {
                dg = col[i * P];
                col[i * P] = 0.f;
            }
        }
        if (live) ++t;
        __syncwarp();
    }
    // The block's sums: one addition a counter, none where nothing was decoded.  (One a counter and group was
    // 136,000 additions to seven addresses in an 8-row launch, 70 us whatever its shots: a fused run of one
    // d = 5 code-capacity shot took 161 us, 72 now.)
    __syncthreads();
    if (threadIdx.x < 6 && a.ctr) {
        const int k = threadIdx.x;
        unsigned long long v = 0;
        for (int w = 0; w < kSmallWarps; ++w)
            for (int q = 0; q < NG; ++q) v += sh_acc[w][q][k];
        if (v) {
            const int slot = k == 0 ? C_ITERS : k == 1 ? C_MSGS : k == 2 ? C_DEFECTS : k == 3 ? C_TIER_SHOTS + a.tier : k == 4 ? C_FC_RUNS : C_FC_ROUNDS;
            atomicAdd(a.ctr + slot, v);
            if (k == 1) atomicAdd(a.ctr + C_TIER_MSGS + a.tier, v);
        }
    }
}

template <int LG, int CH, typename MS, bool TRACE>
cudaError_t run_small1(const DecodeArgs& a, int num_sms, cudaStream_t st, bool prep) {
    using SH = SmallShape<LG, CH, MS>;
    auto kern = decode_small_kernel<LG, CH, MS, TRACE>;
    if (prep) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SH::block_bytes);
    static std::atomic<int> cache[kOccDevices] = {};
    int per_sm = 0;
    cudaError_t e = resident_blocks(kern, kSmallWarps * 32, SH::block_bytes, cache, &per_sm);
    if (e != cudaSuccess) return e;
    // few items: one per warp first
    DecodeArgs b = a;
    b.max_items = (a.max_items + kSmallWarps - 1) / kSmallWarps;
    kern<<<persistent_grid(per_sm * num_sms, b), kSmallWarps * 32, SH::block_bytes, st>>>(a);
    return cudaGetLastError();
}

template <int LG, int CH, typename MS>
cudaError_t run_small(const DecodeArgs& a, int num_sms, cudaStream_t st, bool prep) {
    const bool tr = a.tr_lambda != nullptr || a.tr_partner != nullptr;
    if (prep) {
        cudaError_t e = run_small1<LG, CH, MS, false>(a, num_sms, st, true);
        return e != cudaSuccess ? e : run_small1<LG, CH, MS, true>(a, num_sms, st, true);
    }
    return tr ? run_small1<LG, CH, MS, true>(a, num_sms, st, false)
              : run_small1<LG, CH, MS, false>(a, num_sms, st, false);
}

}  // namespace
}  // namespace bp4m
