#pragma once
// BP4M / BP4MF decoding of one shot per thread block.
//
// Per shot with s unsatisfied detectors (Sec. "Bipartite Graph Representation"): factor c_i
// per detector, variable v_ij per pair and v_ii to the boundary; prior LLR l_ij gathered
// from the per-graph table.  Log-domain sum-product with the flooding schedule (Sec.
// "Belief Propagation"):
//   Q[i][k]  = l_ik + M[k][i] / alpha (k != i),  Q[i][i] = l_ii
//   M'[i][j] = -max*_{k != j} Q[i][k],           max*(x) = ln sum exp(x)
//   lambda_ij = l_ij + (M'[i][j] + M'[j][i]),    lambda_ii = l_ii + M'[i][i]
// The leave-one-out max* of a row uses its largest entry m1 (at k = a), second largest m2
// and S = sum_{k != a} exp(Q_k - m2) >= 1:
//   j == a:  max*_{k != a} = m2 + ln S
//   j != a:  max*_{k != j} = m1 + ln(1 + exp(m2 - m1) (S - exp(Q_j - m2)))
// which is exact algebra, has no cancellation beyond S - exp(Q_j - m2) >= 0, and costs one
// exp and one log per message.  Marginalization keeps v iff lambda_v > 0; convergence =
// every factor keeps exactly one variable (Sec. "Checking convergence").  Forced
// convergence (Sec. "Forced convergence") is the greedy matching in the order
// (lambda desc, i asc, j asc); it is computed here by rounds of locally dominant
// choices (a variable that is the best remaining one at both of its factors is accepted),
// which yields exactly the same matching as the sequential greedy scan.
//
// Layout (shared-memory tiers): Mt[i][k] = M[k][i], the message arriving at factor i from
// the factor k side; Lm[i][k] = l_ik.  With 16-bit message storage every message leaving
// factor k is stored relative to a per-row reference r_k (the row's largest Q of that
// update, rounded to the 16-bit format): Mt[i][k] holds M[k][i] + r_k, which lies in
// [-lg2(s), 0] for every column but the row's argmax, so the 11-bit (FP16) or 8-bit (BF16)
// mantissa resolves the message to a few 1e-4 instead of a few 1e-2 of its magnitude; the
// reader adds -r_k (kept in FP32 per row).  The diagonal holds r_k itself, which decodes
// to exactly 0.  Row i is processed by G threads, thread g taking
// the columns of col_off() (FP32: adjacent pairs 2g, 2g+1, then every 2G; FP64: g + G*c).  The update is in place: every thread caches its row in registers,
// the block synchronises, then each thread writes its outputs M'[i][k] into Mt[k][i].
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <type_traits>
#include <atomic>

#include "device.cuh"

namespace bp4m {
namespace {


template <typename T>
struct Num;

template <>
struct Num<float> {
    static __device__ __forceinline__ float ninf() { return __int_as_float(0xff800000); }
    static __device__ __forceinline__ float pinf() { return __int_as_float(0x7f800000); }
    static __device__ __forceinline__ float ex(float x) { return __expf(x); }
    static __device__ __forceinline__ float lg(float x) { return __logf(x); }
    static __device__ __forceinline__ float lg1p(float x) { return __logf(1.0f + x); }
    static __device__ __forceinline__ const float* L(const DevTables& t) { return t.L32; }
};

template <>
struct Num<double> {
    static __device__ __forceinline__ double ninf() { return __longlong_as_double(0xfff0000000000000ull); }
    static __device__ __forceinline__ double pinf() { return __longlong_as_double(0x7ff0000000000000ull); }
    static __device__ __forceinline__ double ex(double x) { return exp(x); }
    static __device__ __forceinline__ double lg(double x) { return log(x); }
    static __device__ __forceinline__ double lg1p(double x) { return log1p(x); }
    static __device__ __forceinline__ const double* L(const DevTables& t) { return t.L64; }
};

constexpr unsigned kFull = 0xffffffffu;

// Warp 0 turns the shot's bit-packed syndrome into the sorted detector list.
__device__ __forceinline__ int compact_defects(const uint32_t* __restrict__ sw, int nw, int* dets,
                                               int cap, int lane) {
    int base = 0;
    for (int w0 = 0; w0 < nw; w0 += 32) {
        uint32_t word = (w0 + lane < nw) ? __ldg(sw + w0 + lane) : 0u;
        const int c = __popc(word);
        int incl = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += y;
        }
        int pos = base + incl - c;
        while (word) {
            const int b = __ffs(word) - 1;
            word &= word - 1;
            if (pos < cap) dets[pos] = (w0 + lane) * 32 + b;
            ++pos;
        }
        base += __shfl_sync(kFull, incl, 31);
    }
    return base;
}

// Blocks per SM requested from the compiler: enough to keep registers at or below 128.
__host__ __device__ constexpr int min_blocks(int nt) { return 65536 / (nt * 128) > 1 ? 65536 / (nt * 128) : 1; }

// Base-2 transcendental helpers of the shared-memory tiers: messages are kept in log2
// units (every prior is scaled by log2(e) when gathered), so exp and log are single
// ex2/lg2 operations.
template <typename T>
struct B2;

template <>
struct B2<float> {
    static __device__ __forceinline__ float ex2(float x) {
        float y;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
        return y;
    }
    static __device__ __forceinline__ float lg2(float x) {
        float y;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
        return y;
    }
    static __device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ float mx(float a, float b) { return fmaxf(a, b); }
    static __device__ __forceinline__ float mn(float a, float b) { return fminf(a, b); }
};

template <>
struct B2<double> {
    static __device__ __forceinline__ double ex2(double x) { return exp2(x); }
    static __device__ __forceinline__ double lg2(double x) { return log2(x); }
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
    static __device__ __forceinline__ double mx(double a, double b) { return fmax(a, b); }
    static __device__ __forceinline__ double mn(double a, double b) { return fmin(a, b); }
};

// Asynchronous global->shared copies: 16 bytes past L1, or 4 bytes
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    const size_t g = __cvta_generic_to_global(gmem_src);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    const size_t g = __cvta_generic_to_global(gmem_src);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr double kLog2e = 1.4426950408889634074;
constexpr double kLn2 = 0.69314718055994530942;

// Column ownership.  FP32 (PAIR): thread g of a row owns adjacent column pairs, its
// register c holding column k0 + col_off(c) with k0 = 2g and col_off(c) = (c & 1) +
// 2G (c >> 1), so that one 64-bit shared load fetches both columns of a pair.  FP64:
// k0 = g, col_off(c) = G c.
template <bool PAIR, int G>
__host__ __device__ constexpr int col_off(int c) {
    return PAIR ? ((c & 1) + 2 * G * (c >> 1)) : G * c;
}
template <bool PAIR, int G>
__host__ __device__ constexpr int owner_of(int k) {
    return PAIR ? ((k >> 1) % G) : (k % G);
}
template <bool PAIR, int G>
__host__ __device__ constexpr int reg_of(int k) {
    return PAIR ? (2 * (k / (2 * G)) + (k & 1)) : (k / G);
}

// Row pitch in elements.  FP32: pitch = GP x odd (GP = max(G, 2)), the smallest such value
// >= smax.  Then both shared-memory access shapes are conflict free: a half warp's 64-bit
// row read (32/G rows x G pairs) starts the rows in distinct 4-byte bank groups, and a
// warp's transposed write or read (G rows k = 2g + b, G apart by 2, x 32/G consecutive
// rows i) places the G rows 2 x pitch = 8 x odd banks apart (G = 4).  FP64: smax + 1.
template <typename T>
__host__ __device__ constexpr int pitch_of(int smax, int g) {
    return sizeof(T) == 8 ? smax + 1 : (g < 2 ? 2 : g) * (((smax + (g < 2 ? 2 : g) - 1) / (g < 2 ? 2 : g)) | 1);
}

// Storage of the message matrix.  MS = T keeps messages in the arithmetic type; MS = __half
// or __nv_bfloat16 (with T = float) stores them in 16 bits, converted with round to nearest
// and saturation to the largest finite value on the way in, and exactly to FP32 on the way
// out; all arithmetic stays FP32.
template <typename MS, typename T>
struct MsgIO {
    static __device__ __forceinline__ T ld(const MS* p) { return *p; }
    static __device__ __forceinline__ void st(MS* p, T v) { *p = v; }
};

template <>
struct MsgIO<__half, float> {
    static __device__ __forceinline__ float ld(const __half* p) { return __half2float(*p); }
    static __device__ __forceinline__ float2 ld2(const __half* p) {
        return __half22float2(*reinterpret_cast<const __half2*>(p));
    }
    // pack (lo, hi) with saturation; returns the packed pair
    static __device__ __forceinline__ unsigned pack(float lo, float hi) {
        unsigned r;
        asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
        return r;
    }
    static __device__ __forceinline__ float2 unpack(unsigned r) {
        return __half22float2(*reinterpret_cast<const __half2*>(&r));
    }
    static __device__ __forceinline__ void st(__half* p, float v) {
        const unsigned r = pack(v, 0.f);
        *reinterpret_cast<unsigned short*>(p) = (unsigned short)(r & 0xFFFFu);
    }
};

template <>
struct MsgIO<__nv_bfloat16, float> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ float2 ld2(const __nv_bfloat16* p) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
    }
    static __device__ __forceinline__ unsigned pack(float lo, float hi) {
        unsigned r;
        asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
        return r;
    }
    static __device__ __forceinline__ float2 unpack(unsigned r) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r));
    }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) {
        const unsigned r = pack(v, 0.f);
        *reinterpret_cast<unsigned short*>(p) = (unsigned short)(r & 0xFFFFu);
    }
};

// Pitch of the message matrix in elements.  16-bit storage: 2G x odd, so that the 32-bit
// pair reads of a warp (32/G rows x G pairs) and its transposed 16-bit writes (G rows,
// 2 apart, x 32/G consecutive columns) are free of bank conflicts.
template <typename T, typename MS>
__host__ __device__ constexpr int msg_pitch_of(int smax, int g) {
    return sizeof(MS) == 2 ? 2 * g * (((smax + 2 * g - 1) / (2 * g)) | 1) : pitch_of<T>(smax, g);
}

// Byte offset of the 16-bit path's reference array in the dynamic shared memory, after
// Mt, Lm, Dg, rowacc, dets, choice, bestp and matched (8-byte aligned).
// With a helper warp there are two detector lists.
template <typename T, typename MS>
__host__ __device__ constexpr size_t nref_offset(int smax, int g, bool help) {
    return (((size_t)smax * msg_pitch_of<T, MS>(smax, g) * sizeof(MS) + 15) / 16 * 16 +
            (size_t)(smax * pitch_of<T>(smax, g) + smax + (smax & 1)) * sizeof(T) +
            (size_t)smax * (sizeof(double) + (help ? 3 : 2) * sizeof(int) + sizeof(short) + 1) + 7) / 8 * 8;
}

// A thread's register-cached row entries (CH columns).  FP32 keeps them as float2 pairs,
// columns (2j, 2j+1) in one 64-bit register pair, so that the packed FP32x2 add and FMA of
// sm_100 and later apply to two columns per instruction.
template <typename T, int N>
struct Regs {
    T v[N];
    __device__ __forceinline__ T& operator[](int c) { return v[c]; }
};

template <int N>
struct Regs<float, N> {
    static_assert(N % 2 == 0, "FP32 rows are cached in column pairs");
    float2 p[N / 2];
    __device__ __forceinline__ float& operator[](int c) { return (c & 1) ? p[c >> 1].y : p[c >> 1].x; }
};

// min(u, 1) for u >= 0 (saturate), on the FMA pipe: the leave-one-out sum takes the row's
// maximum, 2^(m1 - m2) >= 1, as 1.
__device__ __forceinline__ float sat1(float u) {
    float r;
    asm("add.sat.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(u));
    return r;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// (max, second max, column of the max) of two partial row scans; ties go to the smaller
// column.  Commutative, so every thread of a row group ends with the same triple.
template <typename T>
__device__ __forceinline__ void combine_max(T& m1, T& m2, int& k, T o1, T o2, int ok) {
    if (o1 > m1 || (o1 == m1 && ok < k)) {
        m2 = B2<T>::mx(m1, o2);
        m1 = o1;
        k = ok;
    } else {
        m2 = B2<T>::mx(m2, o1);
    }
}

// Blocks per SM the kernel is compiled for.  FP32 arithmetic: as many as shared memory holds
// and registers allow without spills: nine of 96 threads (48 rows), six of 128 (64 rows), three of
// 320 (80 rows), two of 384 and 448 (96 and 112 rows; 79 and 106 KB), and two of 512 (128 rows)
// with 16-bit messages (102 KB); the others are limited by shared memory or 128 registers.
__host__ __device__ constexpr int blocks_for(int nt, int elem_bytes, int msg_bytes) {
    if (elem_bytes != 4) return min_blocks(nt);
    return nt == 96 ? 9 : nt == 128 ? 6 : nt == 320 ? 3 : nt == 384 || nt == 448 ? 2 : nt == 512 && msg_bytes == 2 ? 2 : min_blocks(nt);
}

// Convergence decision (FP32 arithmetic).  A shot has converged only if every row keeps exactly
// one variable, so one row that does not settles an iteration's decision.  The block's last warp
// watches kWatch rows that were seen violating; only when none of them violates is every row
// counted (in about 1% of the iterations of d = 13 circuit shots, 20 of whose rows violate in the
// median iteration).  Counting every row in every iteration took an add, a multiply and an
// own-output read per message, or a register copy of the outputs (24 warp instructions per 32
// updates at 144 rows, 19 without).
//
// Bound: the special-function unit takes 0.094 SM-cycles an update (ex2 and lg2), the compares
// and maxima of the row scan about as much; the phases of an iteration run one after another
// between its two barriers, so that the tiers of one block per SM reach about 0.3 of that.
// Measured per tier (d = 13 circuit, 100,000 shots; G updates/s at the start and now): 96 rows
// 888 -> 1035, 112 rows 1004 -> 1189, 128 rows 875 -> 994, 144 rows 836 -> 970, 160 rows
// 906 -> 1054; 64 rows (d = 21 code capacity) 1039 -> 1325.  Double-buffered messages with the
// priors in registers (one barrier an iteration, half the shared-memory reads) measured the same
// or slower: 96 registers a thread made it spill.
constexpr int kWatch = 4;

// The FP32-arithmetic forms of 128 and 144 rows that run one block per SM have a helper warp: it
// watches beside the others' reads instead of holding up the vote, and fetches the next shot's
// detector list during the first iteration.  (160 rows: twenty warps of 96 registers leave no
// room for it.  Where two blocks share an SM the other block fills the gaps.)
__host__ __device__ constexpr bool helper_warp(int smax, int elem_bytes, int msg_bytes, bool rw) {
    return elem_bytes == 4 && !rw && (smax == 144 || (smax == 128 && msg_bytes == 4));
}
__host__ __device__ constexpr int block_threads(int ch, int g, int elem_bytes, int msg_bytes, bool rw) {
    return ch * g * g + (helper_warp(ch * g, elem_bytes, msg_bytes, rw) ? 32 : 0);
}

// RW = true: the B-BP4MF second stage.  The shot's priors, pair weights and parities are
// computed in the block from the shortest paths of every defect over per-qubit weights derived
// from the first stage's posteriors (instead of being gathered from the static tables).
template <typename T, int CH, int G, bool TRACE, bool RW = false, typename MS = T>
__global__ void __launch_bounds__(block_threads(CH, G, (int)sizeof(T), (int)sizeof(MS), RW), blocks_for(CH * G * G, (int)sizeof(T), (int)sizeof(MS))) decode_smem_kernel(const DecodeArgs a) {
    constexpr int SMAX = CH * G;
    constexpr bool HELP = helper_warp(SMAX, (int)sizeof(T), (int)sizeof(MS), RW);
    constexpr int NT = block_threads(CH, G, (int)sizeof(T), (int)sizeof(MS), RW);
    constexpr int R = 32 / G;
    constexpr int P = pitch_of<T>(SMAX, G);          // priors
    constexpr int PM = msg_pitch_of<T, MS>(SMAX, G);  // messages
    constexpr bool HALF = sizeof(MS) == 2;
    static_assert(!HALF || sizeof(T) == 4, "16-bit messages use FP32 arithmetic");
    using IO = MsgIO<MS, T>;
    static_assert(NT % 32 == 0 && NT <= 1024, "block size");
    using Mask = typename std::conditional<(CH > 32), unsigned long long, unsigned int>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    MS* const Mt = reinterpret_cast<MS*>(smem);  // Mt[i][k] = M[k][i]; diagonal kept 0
    T* const Lm = reinterpret_cast<T*>(smem + ((size_t)SMAX * PM * sizeof(MS) + 15) / 16 * 16);  // Lm[i][k] = l_ik (log2), -inf past s
    T* const Dg = Lm + SMAX * P;                 // Dg[i] = M[i][i] (factor i to its boundary variable)
    double* rowacc = reinterpret_cast<double*>(Dg + SMAX + (SMAX & 1));
    int* const dets0 = reinterpret_cast<int*>(rowacc + SMAX);
    int* dets = dets0;  // HELP: the current one of two
    int* choice = dets0 + (HELP ? 2 : 1) * SMAX;
    short* bestp = reinterpret_cast<short*>(choice + SMAX);
    unsigned char* matched = reinterpret_cast<unsigned char*>(bestp + SMAX);
    // 16-bit messages: nrefv[k] = -r_k, minus the reference of the messages leaving factor k
    float* const nrefv = reinterpret_cast<float*>(smem + nref_offset<T, MS>(SMAX, G, HELP));
    // static-partition forced convergence: factors in processing order
    short* order = reinterpret_cast<short*>(smem + nref_offset<T, MS>(SMAX, G, HELP) + (HALF ? (size_t)SMAX * 4 : 0));
    // RW only: per-shot W (FP64) and parity over local ranks, distances and predecessors per warp
    // and the weight of each qubit, in this block's global scratch slot (layout of rw_slot_layout)
    const int rw_nodes = a.tb.n_det + 1;
    unsigned char* rw_slot = RW ? reinterpret_cast<unsigned char*>(a.gscratch) + (size_t)blockIdx.x * a.rw_slot_bytes
                                : nullptr;
    double* Wsh = reinterpret_cast<double*>(rw_slot);
    double* rw_dist = Wsh + SMAX * SMAX;
    double* rw_w = rw_dist + (NT / 32) * rw_nodes;  // [rw_units] weights of the shot's qubits
    uint32_t* rw_pred = reinterpret_cast<uint32_t*>(rw_w + a.rw_units);
    unsigned char* Psh = reinterpret_cast<unsigned char*>(rw_pred + (NT / 32) * rw_nodes);
    __shared__ int sh_item, sh_s, sh_flags, sh_best_par, sh_best_forced, sh_improve, sh_use_best;
    __shared__ double sh_best_w;
    __shared__ int sh_next_code[2], sh_next_s[2];  // HELP: the shots fetched ahead
    __shared__ unsigned sh_open[(SMAX + 31) / 32];  // forced convergence: unmatched rows
    __shared__ int sh_watch[kWatch];
    __shared__ unsigned sh_bad[NT / 32];  // full count: each warp's rows that do not keep exactly one

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i = warp * R + (lane % R);   // row (factor) of this thread
    const int g = lane / R;                // column group of this thread within the row
    constexpr bool PAIR = sizeof(T) == 4;
    const int k0 = PAIR ? 2 * g : g;       // first column of this thread
    const bool own_diag = owner_of<PAIR, G>(i) == g;   // this thread holds column k = i of its row
    const int c_diag = reg_of<PAIR, G>(i);
    const int count = *a.count;
    const T ainv = (T)(1.0 / a.alpha);
    const bool full = (a.decoder == 1) || !a.early_exit;
    T* trl = reinterpret_cast<T*>(a.tr_lambda);
    const T ninf = Num<T>::ninf();
    // counters of this block's shots: updated by thread 0 only, so kept in shared memory rather
    // than in twelve registers of every thread
    __shared__ unsigned long long sh_acc[6];
    unsigned long long &acc_it = sh_acc[0], &acc_msg = sh_acc[1], &acc_def = sh_acc[2], &acc_shots = sh_acc[3],
                       &acc_fc = sh_acc[4], &acc_fcr = sh_acc[5];
    if (tid == 0)
        for (int k = 0; k < 6; ++k) sh_acc[k] = 0;

    T* const row_l = Lm + i * P + k0;    // priors l_ik, register c at [col_off(c)]
    MS* const row_m = Mt + i * PM + k0;  // incoming messages M[k][i]
    MS* const col_m = Mt + k0 * PM + i;  // own outputs M[i][k] live at Mt[k][i], register c at [col_off(c) PM]
#define COL(c) (k0 + col_off<PAIR, G>(c))
#define RL(c) l_ld1(c)
#define RM(c) m_ld1(row_m + col_off<PAIR, G>(c), COL(c))
#define CMP(c) (col_m + col_off<PAIR, G>(c) * PM)
#define CM(c) m_ld1(CMP(c), i)
#define RL2(j) l_ld2(j)
#define RM2(j) m_ld2(row_m + col_off<PAIR, G>(2 * (j)), k0 + col_off<PAIR, G>(2 * (j)))
    auto l_ld1 = [&](int c) -> T { return row_l[col_off<PAIR, G>(c)]; };
    auto l_ld2 = [&](int j) -> float2 { return *reinterpret_cast<const float2*>(row_l + col_off<PAIR, G>(2 * j)); };
    // messages arriving at row i from columns k, k + 1 (16-bit: decoded with the source rows'
    // references), and one arriving from column k
    auto m_ld2 = [&](const MS* p, int k) -> float2 {
        if constexpr (HALF)
            return __fadd2_rn(IO::ld2(p), *reinterpret_cast<const float2*>(nrefv + k));
        else
            return *reinterpret_cast<const float2*>(p);
    };
    auto m_ld1 = [&](const MS* p, int k) -> T {
        if constexpr (HALF)
            return IO::ld(p) + nrefv[k];
        else
            return IO::ld(p);
    };

    // HELP: the last warp takes the block's next item into buffer b (code -1: none left)
    auto fetch_next = [&](int b) {
        int item = 0;
        if (lane == 0) item = atomicAdd(a.next, 1);
        item = __shfl_sync(kFull, item, 0);
        int c = -1, s0 = 0;
        if (item < count) {
            c = a.list[(int64_t)item * a.list_dir];
            const ItemCtx ic = resolve_item(a, c);
            s0 = compact_defects(ic.synd + (size_t)ic.shot * ic.tb.n_words, ic.tb.n_words, dets0 + b * SMAX, SMAX, lane);
        }
        if (lane == 0) {
            sh_next_code[b] = c;
            sh_next_s[b] = s0;
        }
    };
    int pb = 0;
    if (HELP) {
        if (warp == NT / 32 - 1) fetch_next(0);
        __syncthreads();
    }

    for (;;) {
        // the graph and outputs are looked up where they are needed: kept across the iterations
        // they would take twenty registers
        int code, s;
        if constexpr (HELP) {
            code = sh_next_code[pb];
            if (code < 0) break;
            s = sh_next_s[pb];
            dets = dets0 + pb * SMAX;
        } else {
            if (tid == 0) sh_item = atomicAdd(a.next, 1);
            __syncthreads();
            const int item = sh_item;
            if (item >= count) break;
            code = a.list[(int64_t)item * a.list_dir];
            if (warp == 0) {
                const ItemCtx ic = resolve_item(a, code);
                const int s0 = compact_defects(ic.synd + (size_t)ic.shot * ic.tb.n_words, ic.tb.n_words, dets, SMAX, lane);
                if (lane == 0) sh_s = s0;
            }
            __syncthreads();
            s = sh_s;
        }
        const ItemCtx ic0 = resolve_item(a, code);
        const int64_t shot = ic0.shot;
        const int n = ic0.tb.n_det;
        const T* __restrict__ Ltab = Num<T>::L(ic0.tb);
        if (s > SMAX || s < (HELP ? 2 : 1)) {
            if (tid == 0 && a.ctr) atomicAdd(a.ctr + C_ERRORS, 1ull);
            if constexpr (HELP) {
                __syncthreads();
                if (warp == NT / 32 - 1) fetch_next(pb);
                __syncthreads();
            }
            continue;
        }
        const bool tr_on = TRACE && s <= a.s_cap;
        if (!HELP && s == 1 && !RW) {
            // a single factor with a single variable: the leave-one-out set is empty, the
            // message is +inf and v_00 is kept in every iteration
            if (tid == 0) {
                const int its = full ? a.T : 1;
                const int d0 = dets[0];
                if (ic0.obs_pred) ic0.obs_pred[shot] = ic0.tb.P[(size_t)d0 * n + d0];
                if (ic0.flags) ic0.flags[shot] = F_CONVERGED;
                if (ic0.iters) ic0.iters[shot] = (int16_t)its;
                if (tr_on && trl) trl[(size_t)shot * a.s_cap * a.s_cap] = Num<T>::pinf();
                if (tr_on && a.tr_partner) {
                    a.tr_partner[(size_t)shot * a.s_cap] = 0;
                    for (int k = 1; k < a.s_cap; ++k) a.tr_partner[(size_t)shot * a.s_cap + k] = -1;
                }
                acc_it += (unsigned long long)its;
                acc_msg += (unsigned long long)its;
                acc_def += 1;
                acc_shots += 1;
            }
            continue;
        }
        const bool act = i < s;
        // rows warp*R .. warp*R+R-1 belong to this warp; a warp with none of them active
        // skips the read and compute phases (it still takes part in every barrier)
        const bool wact = warp * R < s;
        Regs<T, CH> q;
        // ---- gather the shot's priors (log2 units); columns past s are -inf so that they
        // never win a max, add nothing to a sum and are never kept
        if constexpr (std::is_same<T, float>::value && !RW) {
            // The table is symmetric: each pair k >= r is fetched once, row by row (a warp's 32
            // columns of one table row lie in about ten 128-byte lines), with every copy of the
            // shot in flight at once, and mirrored in shared memory.
            float* const st = reinterpret_cast<float*>(Lm);
            for (int r = warp; r < s; r += NT / 32) {
                const T* trow = Ltab + (size_t)dets[r] * n;
                for (int k = r + lane; k < s; k += 32) cp_async4(st + r * P + k, trow + dets[k]);
            }
            cp_async_commit();
            cp_async_wait_all();
            __syncthreads();
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int k = COL(c);
                q[c] = act && k < s ? st[k >= i ? i * P + k : k * P + i] * (float)kLog2e : ninf;
            }
            __syncthreads();
            if (act) {
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    row_l[col_off<PAIR, G>(c)] = q[c];
                    row_m[col_off<PAIR, G>(c)] = MS(0.f);
                }
            }
        } else if (!RW) {
            for (int r = warp; r < s; r += NT / 32) {
                const T* trow = Ltab + (size_t)dets[r] * n;
                for (int k = lane; k < SMAX; k += 32) {
                    Lm[r * P + k] = k < s ? (T)(__ldg(trow + dets[k]) * (T)kLog2e) : ninf;
                    Mt[r * PM + k] = MS(0.f);
                }
            }
        } else {
            // Shortest paths from every defect (one warp per source) over edge weights
            // |ln((1-P)/P)| of the qubit behind the edge (edges above one half were flipped out of
            // the syndrome), floored at kRwMinWeight; the boundary node n is a sink.  Distances and
            // parities are those of Dijkstra's algorithm that pops nodes in (distance, index) order
            // and changes a predecessor only on a strict improvement: rounding is monotone and
            // weights are positive, so relaxing every node from its neighbours until nothing
            // changes ends in the same distances, and v's predecessor is the neighbour u, first in
            // (distance, index) order, then the first entry of v's list, with dist[u] + w equal to
            // dist[v].  Weights are taken once per qubit of the shot: a logarithm per relaxed edge
            // and source, by one lane, was most of this stage (FP64 runs at two operations a clock
            // and SM): 28.5 -> 3.2 ms for 10,000 d = 9 shots of both stages.  Distances are positive, so
            // they compare as integers.
            for (int u = tid; u < a.rw_units; u += NT) {
                double pq = a.rw_post[(size_t)shot * a.rw_units + u];
                pq = pq < 1e-300 ? 1e-300 : (pq > 1.0 - 1e-16 ? 1.0 - 1e-16 : pq);
                // an edge above one half was taken as present (flipped out of the syndrome): it
                // weighs as its complement
                if (pq > 0.5) pq = 1.0 - pq;
                rw_w[u] = fmax(log((1.0 - pq) / pq), kRwMinWeight);
            }
            __syncthreads();
            long long* const dist = reinterpret_cast<long long*>(rw_dist + warp * rw_nodes);
            uint32_t* const pred = rw_pred + warp * rw_nodes;
            const long long dinf = __double_as_longlong(Num<double>::pinf());
            for (int r = warp; r < s; r += NT / 32) {
                const int src = dets[r];
                for (int v = lane; v < rw_nodes; v += 32) dist[v] = v == src ? 0 : dinf;
                __syncwarp();
                bool again = true;
                for (int sweep = 0; again && sweep <= rw_nodes; ++sweep) {  // (a path has fewer edges than nodes)
                    bool changed = false;
                    for (int v0 = 0; v0 < n; v0 += 32) {
                        const int v = v0 + lane;
                        long long best = v < n ? dist[v] : 0;
                        bool up = false;
                        if (v < n) {
                            const int e1 = a.rw_off[v + 1];
                            for (int e = a.rw_off[v]; e < e1; ++e) {
                                const uint32_t pk = a.rw_adj[e];
                                const int u = (int)(pk & 0x7FFFu);
                                if (u == n) continue;
                                const long long nd = __double_as_longlong(__longlong_as_double(dist[u]) + rw_w[(pk >> 15) & 0x7FFFu]);
                                if (nd < best) {
                                    best = nd;
                                    up = true;
                                }
                            }
                        }
                        __syncwarp();
                        if (up) dist[v] = best;
                        changed |= up;
                        __syncwarp();
                    }
                    again = __any_sync(kFull, changed);
                }
                // the boundary's distance, and every node's predecessor (node | obs << 15)
                for (int v = lane; v < rw_nodes; v += 32) {
                    const int e1 = a.rw_off[v + 1];
                    long long best = v == n ? dinf : dist[v], du = dinf;
                    uint32_t p = 0xFFFFFFFFu;
                    for (int e = a.rw_off[v]; e < e1; ++e) {
                        const uint32_t pk = a.rw_adj[e];
                        const int u = (int)(pk & 0x7FFFu);
                        if (u == n) continue;
                        const long long d = dist[u];
                        const long long nd = __double_as_longlong(__longlong_as_double(d) + rw_w[(pk >> 15) & 0x7FFFu]);
                        const bool better = v == n && nd < best;
                        if (nd != dinf && (better || (nd == best && d < du))) {
                            best = nd;
                            du = d;
                            p = (uint32_t)u | (pk >> 31) << 15;
                        }
                    }
                    pred[v] = v == src ? 0xFFFFFFFFu : p;
                    if (v == n) dist[n] = best;
                }
                __syncwarp();
                for (int k = r + lane; k < s; k += 32) {
                    const int tgt = k == r ? n : dets[k];
                    unsigned char par = 0;
                    for (uint32_t p = pred[tgt]; p != 0xFFFFFFFFu; p = pred[p & 0x7FFFu]) par ^= (unsigned char)(p >> 15);
                    Wsh[r * SMAX + k] = __longlong_as_double(dist[tgt]);
                    Psh[r * SMAX + k] = par;
                }
                __syncwarp();
            }
            __syncthreads();
            // priors of the pairs k >= r, mirrored
            for (int r = warp; r < s; r += NT / 32) {
                for (int k = lane; k < SMAX; k += 32) {
                    if (k >= s) {
                        Lm[r * P + k] = ninf;
                    } else if (k >= r) {
                        const double W = Wsh[r * SMAX + k];
                        const double l = W == Num<double>::pinf() ? -1.0e30 : -W - log1p(-exp(-W));
                        Lm[r * P + k] = Lm[k * P + r] = (T)(l * kLog2e);
                        Wsh[k * SMAX + r] = W;
                        Psh[k * SMAX + r] = Psh[r * SMAX + k];
                    }
                    Mt[r * PM + k] = MS(0.f);
                }
            }
        }
        if (tid < SMAX) {
            Dg[tid] = T(0);
            matched[tid] = tid >= s;
            bestp[tid] = -1;
            if constexpr (HALF) nrefv[tid] = 0.f;
        }
        if (tid == 0) {
            sh_flags = 0;
            sh_best_w = Num<double>::pinf();
            sh_best_par = 0;
            sh_best_forced = 0;
            sh_use_best = 0;
        }
        __syncthreads();
        if (RW && s == 1) {
            // one defect: matched to the boundary along its reweighted path
            if (tid == 0) {
                const int its = full ? a.T : 1;
                if (ic0.obs_pred) ic0.obs_pred[shot] = Psh[0];
                if (ic0.flags) ic0.flags[shot] = F_CONVERGED;
                if (ic0.iters) ic0.iters[shot] = (int16_t)its;
                acc_it += (unsigned long long)its;
                acc_msg += (unsigned long long)its;
                acc_def += 1;
                acc_shots += 1;
            }
            continue;
        }

        constexpr int WW = NT / 32 - 1;  // the warp that watches
        int wj = 0;                      // the watched row tried first
        int t = 0;
        // set where a candidate finishes the shot
        int out_par, out_forced, out_from_best, partner;

        // FP32: Q = l + M[k][i]/alpha for the next update, with the row's maximum m1 and second
        // maximum m2 scanned in the same loop (it needs only Q), so that the shared-memory loads
        // and the scan's ALU work overlap.  The column of m1 is not tracked here: the exponential
        // loop below finds it as the one column above m2.
        T m1 = ninf, m2 = ninf;
        auto read_rows = [&]() {
          if constexpr (std::is_same<T, float>::value) {
            if (!wact) return;
            m1 = ninf;
            m2 = ninf;
            if (!act) {
#pragma unroll
                for (int c = 0; c < CH; ++c) q[c] = ninf;
            } else {
                const float2 ainv2 = make_float2(ainv, ainv);
#pragma unroll
                for (int j = 0; j < CH / 2; j += 2) {
                    const float2 p0 = __ffma2_rn(RM2(j), ainv2, RL2(j));
                    const float2 p1 = __ffma2_rn(RM2(j + 1), ainv2, RL2(j + 1));
                    q.p[j] = p0;
                    q.p[j + 1] = p1;
                    // four columns' maximum and second maximum into the row's
                    const float h0 = fmaxf(p0.x, p0.y), l0 = fminf(p0.x, p0.y);
                    const float h1 = fmaxf(p1.x, p1.y), l1 = fminf(p1.x, p1.y);
                    const float hi = fmaxf(h0, h1), lo = max3f(l0, l1, fminf(h0, h1));
                    m2 = max3f(m2, lo, fminf(m1, hi));
                    m1 = fmaxf(m1, hi);
                }
            }
#pragma unroll
            for (int off = R; off < 32; off <<= 1) {
                const T o1 = __shfl_xor_sync(kFull, m1, off);
                const T o2 = __shfl_xor_sync(kFull, m2, off);
                m2 = max3f(m2, o2, fminf(m1, o1));
                m1 = fmaxf(m1, o1);
            }
          }
        };
        // FP32: leave-one-out max* of every row.  With m1 (at column am) and m2 the two largest Q of
        // the row and S = sum_k min(2^(Q_k - m2), 1), so that S - 1 = sum_{k != am} 2^(Q_k - m2) >= 1:
        //   k != am: M'[i][k] = -(m1 + lg2(1 + 2^(m2 - m1) (S - 1 - 2^(Q_k - m2))))
        //   k == am: M'[i][k] = -(m2 + lg2(S - 1))
        // (the generic value is written for every column, the thread with a column above m2 then
        // overwrites it; where m1 == m2 no column is above m2 and both formulas give the same
        // value: 2^(m2 - m1) = 1 and S - 1 is exact).  Row i's outputs M'[i][k] go to Mn[k][i].
        auto update_rows = [&]() {
          if constexpr (std::is_same<T, float>::value) {
            if (!wact) return;
            // 2^(Q - m2) from m2 - Q, whose sign bit marks the column above m2: one funnel shift a
            // column collects them, first column in the highest bit
            const float2 m22 = make_float2(m2, m2), neg1 = make_float2(-1.f, -1.f);
            float2 s2 = make_float2(0.f, 0.f);
            unsigned top0 = 0, top1 = 0;
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) {
                const float2 dq = __ffma2_rn(q.p[j], neg1, m22);
                const float2 u = make_float2(B2<float>::ex2(-dq.x), B2<float>::ex2(-dq.y));
                q.p[j] = u;
                s2 = __fadd2_rn(s2, make_float2(sat1(u.x), sat1(u.y)));
                unsigned& top = j < 16 ? top0 : top1;
                top = __funnelshift_l(__float_as_uint(dq.x), top, 1);
                top = __funnelshift_l(__float_as_uint(dq.y), top, 1);
            }
            float S32 = s2.x + s2.y;
#pragma unroll
            for (int off = R; off < 32; off <<= 1) S32 += __shfl_xor_sync(kFull, S32, off);
            if (!act) return;
            const float cf32 = B2<float>::ex2(m2 - m1);
            const float Aa32 = __fmaf_rn(cf32, S32 - 1.f, 1.f);
            // 16-bit storage: this row's reference r_i = m1 rounded to the format (so that it is
            // exact there); stored values out + r_i = -lg2(Aa - cf u) + (r_i - m1)
            float rf = 0.f, dref32 = 0.f;
            if constexpr (HALF) {
                rf = IO::unpack(IO::pack(m1, 0.f)).x;
                dref32 = rf - m1;
            }
            // out = -m1 - lg2(Aa - cf u), the subtraction as an exact fma with -1
            const float2 ncf = make_float2(-cf32, -cf32), A2 = make_float2(Aa32, Aa32);
            const float2 nm1 = HALF ? make_float2(dref32, dref32) : make_float2(-m1, -m1);
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) {
                const float2 y = __ffma2_rn(ncf, q.p[j], A2);
                const float2 lg = make_float2(B2<float>::lg2(y.x), B2<float>::lg2(y.y));
                const float2 out = __ffma2_rn(lg, neg1, nm1);
                if constexpr (HALF) {
                    // store the rounded pair (relative to r_i): both ends of a variable read the
                    // same message
                    const unsigned pk2 = IO::pack(out.x, out.y);
                    *reinterpret_cast<unsigned short*>(CMP(2 * j)) = (unsigned short)(pk2 & 0xFFFFu);
                    *reinterpret_cast<unsigned short*>(CMP(2 * j + 1)) = (unsigned short)(pk2 >> 16);
                } else {
                    *CMP(2 * j) = out.x;
                    *CMP(2 * j + 1) = out.y;
                }
            }
            if (top0 | top1) {
                constexpr int N0 = CH < 32 ? CH : 32;
                const int c = top0 ? N0 - 32 + __clz((int)top0) : CH - 32 + __clz((int)top1);
                const int am = COL(c);
                const float lgS = B2<float>::lg2(S32 - 1.f);
                if constexpr (HALF)
                    IO::st(Mt + am * PM + i, __fmaf_rn(lgS, -1.f, rf - m2));
                else
                    IO::st(Mt + am * PM + i, -m2 - lgS);
            }
            if (own_diag) {
                MS* const md = Mt + i * PM + i;
                if constexpr (HALF) {
                    // the diagonal holds r_i, which decodes to exactly 0
                    Dg[i] = IO::ld(md) + (-rf);
                    IO::st(md, rf);
                    nrefv[i] = -rf;
                } else {
                    Dg[i] = IO::ld(md);
                    *md = MS(0.f);
                }
            }
          }
        };
        if (tid < kWatch) sh_watch[tid] = tid * s / kWatch;
        // FP32: 1 if a watched row does not keep exactly one variable of lambda^t.  The rows are tried
        // from the one that violated last; one that keeps exactly one moves on.
        auto watch_rows = [&]() -> int {
          if constexpr (std::is_same<T, float>::value) {
            for (int tries = 0; tries < kWatch; ++tries) {
                const int r = sh_watch[wj];
                int cnt = 0;
#pragma unroll
                for (int j = 0; j < (SMAX + 31) / 32; ++j) {
                    const int k = min(lane + 32 * j, s - 1);
                    const float l = Lm[r * P + k];
                    const float lam = k == r ? l + Dg[r] : l + (m_ld1(Mt + k * PM + r, r) + m_ld1(Mt + r * PM + k, k));
                    cnt += lane + 32 * j < s && lam > 0.f ? 1 : 0;
                }
                if (__reduce_add_sync(kFull, cnt) != 1) return 1;
                if (lane == 0) sh_watch[wj] = r + 1 < s ? r + 1 : 0;
                wj = (wj + 1) % kWatch;
                __syncwarp();
            }
            return 0;
          }
          return 1;
        };

        for (;;) {
            // ---- convergence of lambda^t: every row keeps exactly one variable; the watched row
            // settles most votes (in a d = 13 circuit shot 20 rows violate in the median iteration)
            Mask bits = 0;
            int conv = 0, chosen = -1;
            if constexpr (std::is_same<T, float>::value) {
                if (TRACE && tr_on && trl && t > 0 && act) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int k = COL(c);
                        if (k < s)
                            trl[((size_t)shot * a.s_cap + i) * a.s_cap + k] =
                                (k == i ? RL(c) + Dg[i] : RL(c) + (CM(c) + RM(c))) * (float)kLn2;
                    }
                }
                read_rows();
                {
                    int violated = t == 0;
                    if (warp == WW) {
                        if (t > 0) violated = watch_rows();
                        if (HELP && t == 0) fetch_next(pb ^ 1);
                    }
                    // (also the barrier between reading Mt and overwriting it)
                    conv = !__syncthreads_or(violated);
                    if (conv) {
                        // no watched row violates: count every row, and find its kept column
                        int k1 = -1, cnt = 0;
                        if (act) {
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int k = COL(c);
                                const float l = RL(c);
                                const float lam = k == i ? l + Dg[i] : l + (CM(c) + RM(c));
                                cnt += lam > 0.f ? 1 : 0;
                                if (lam > 0.f) k1 = k;
                            }
                        }
#pragma unroll
                        for (int off = R; off < 32; off <<= 1) {
                            cnt += __shfl_xor_sync(kFull, cnt, off);
                            k1 = max(k1, __shfl_xor_sync(kFull, k1, off));
                        }
                        chosen = k1;
                        const bool bad = act && cnt != 1;
                        const unsigned badrows = __ballot_sync(kFull, bad) & (R == 32 ? kFull : (1u << (R & 31)) - 1u);
                        if (lane == 0) sh_bad[warp] = badrows;
                        conv = __syncthreads_and(!bad);
                        if (!conv && warp == WW) {
                            // watch violating rows, the first at or after each share of the rows
                            for (int j = 0; j < kWatch; ++j) {
                                int w = j * (NT / 32) / kWatch;
                                while (sh_bad[w] == 0u) w = w + 1 < NT / 32 ? w + 1 : 0;
                                if (lane == 0) sh_watch[j] = w * R + __ffs((int)sh_bad[w]) - 1;
                            }
                        }
                    }
                }
            } else {
                // FP64: every row is counted in the read phase.  Bound by the FP64 pipe (two operations
                // a clock and SM): columns past s, whole registers of them (k = g + G c >= s in every
                // thread of the block), are left out of every loop; they would add exactly 0.  At
                // s <= 4 of 32 columns (d = 3) they were most of the work: 4.05 -> 0.99 ms for 10^4 shots.
                if (!wact) {
                } else if (!act) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) q[c] = ninf;
                } else if (t == 0) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) q[c] = G * c < s ? B2<T>::fma_(RM(c), ainv, RL(c)) : ninf;
                } else {
                    Mask b0 = 0, b1 = 0;
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        q[c] = ninf;
                        if (G * c >= s) continue;
                        const T l = RL(c);
                        const T x = RM(c);
                        q[c] = B2<T>::fma_(x, ainv, l);
                        const T lam = l + (CM(c) + x);
                        if (c & 1)
                            b1 |= (Mask)(lam > T(0) ? 1u : 0u) << c;
                        else
                            b0 |= (Mask)(lam > T(0) ? 1u : 0u) << c;
                        if (tr_on && trl && COL(c) < s)
                            trl[((size_t)shot * a.s_cap + i) * a.s_cap + COL(c)] = lam * (T)kLn2;
                    }
                    bits = b0 | b1;
                    if (own_diag) {
                        // the boundary variable v_ii: lambda_ii = l_ii + M[i][i]
                        const T lam = Lm[i * P + i] + Dg[i];
                        bits = (bits & ~((Mask)1 << c_diag)) | ((Mask)(lam > T(0) ? 1u : 0u) << c_diag);
                        if (tr_on && trl) trl[((size_t)shot * a.s_cap + i) * a.s_cap + i] = lam * (T)kLn2;
                    }
                }
                // kept count << 16 plus (first kept column + 1), summed over the row's G threads:
                // the count is exact, the column is the row's only kept one when the count is 1
                int pk = ((sizeof(Mask) == 8 ? __popcll((unsigned long long)bits) : __popc((unsigned)bits)) << 16) +
                         (bits ? COL((sizeof(Mask) == 8 ? __ffsll((long long)bits) : __ffs((int)bits)) - 1) + 1 : 0);
#pragma unroll
                for (int off = R; off < 32; off <<= 1) pk += __shfl_xor_sync(kFull, pk, off);
                const int cnt = pk >> 16;
                chosen = (pk & 0xFFFF) - 1;
                conv = __syncthreads_and(t > 0 && (!act || cnt == 1));
            }

            bool requeue = false;  // Q gave way to the posteriors of forced convergence
            if (t > 0) {
                bool have_cand = false, cand_forced = false;
                int cand_p = -1;
                if (conv) {
                    if (tid == 0) sh_flags |= F_CONVERGED;
                    have_cand = true;
                    cand_p = chosen;
                } else if (a.decoder == 1 || t == a.T) {
                    // ---- forced convergence on lambda^t by locally dominant rounds
                    if (tid == 0) sh_flags |= F_FORCED_RAN;
                    if (act && g == 0) matched[i] = 0;
                    __syncthreads();
                    const T dgi = act ? Dg[i] : T(0);
                    if (a.forced_static) {
                        // the paper's static partition: row i's block is v_ik, k >= i; its
                        // maximum (ties: smaller k) represents factor i; representatives are
                        // ranked by posterior (ties: smaller i) and processed in that order
                        T bl = ninf;
                        int bk = -1;
                        if (act) {
#pragma unroll
                            for (int c = 0; c < CH; ++c) {
                                const int k = COL(c);
                                if (k >= i && k < s) {
                                    const T lam = k == i ? RL(c) + dgi : RL(c) + (CM(c) + RM(c));
                                    if (bk < 0 || lam > bl) {
                                        bl = lam;
                                        bk = k;
                                    }
                                }
                            }
                        }
#pragma unroll
                        for (int off = R; off < 32; off <<= 1) {
                            const T ol = __shfl_xor_sync(kFull, bl, off);
                            const int ok = __shfl_xor_sync(kFull, bk, off);
                            if (ok >= 0 && (bk < 0 || ol > bl || (ol == bl && ok < bk))) {
                                bl = ol;
                                bk = ok;
                            }
                        }
                        if (act && g == 0) {
                            choice[i] = bk >= 0 ? bk : i;
                            rowacc[i] = (double)bl;
                        }
                        __syncthreads();
                        if (tid < s) {
                            const double v = rowacc[tid];
                            int rank = 0;
                            for (int j = 0; j < s; ++j) {
                                const double u = rowacc[j];
                                rank += (u > v || (u == v && j < tid)) ? 1 : 0;
                            }
                            order[rank] = (short)tid;
                        }
                        __syncthreads();
                        if (tid == 0) {
                            // a factor whose representative's other factor is taken goes to
                            // the boundary (a case the paper does not treat)
                            for (int r = 0; r < s; ++r) {
                                const int ii = order[r];
                                if (matched[ii]) continue;
                                const int k = choice[ii];
                                matched[ii] = 1;
                                if (k == ii || matched[k]) {
                                    choice[ii] = ii;
                                } else {
                                    matched[k] = 1;
                                    choice[k] = ii;
                                }
                            }
                            acc_fcr += 1;
                        }
                        __syncthreads();
                    }
                    // Rows choose their best unmatched column; a variable chosen by both its rows (or
                    // the boundary) is accepted.  Unmatched rows are a bit set, columns are compared
                    // without branches, and a row whose choice is still unmatched keeps it: the best
                    // of a set that has only shrunk around it.
                    if (!a.forced_static) {
                        if (tid < (SMAX + 31) / 32) sh_open[tid] = s >= 32 * (tid + 1) ? kFull : s <= 32 * tid ? 0u : (1u << (s & 31)) - 1u;
                        __syncthreads();
                    }
                    int ch = -1;
                    if (!a.forced_static && act) {
                        // the row's posteriors take the place of Q (read again if the shot goes on)
#pragma unroll
                        for (int c = 0; c < CH; ++c) q[c] = COL(c) == i ? RL(c) + dgi : RL(c) + (CM(c) + RM(c));
                    }
                    requeue = !a.forced_static;
                    for (int round = 0; round < s && !a.forced_static; ++round) {
                        const bool open = act && ((sh_open[i >> 5] >> (i & 31)) & 1u);
                        const bool scan = open && (round == 0 || !((sh_open[ch >> 5] >> (ch & 31)) & 1u));
                        if (__any_sync(kFull, scan)) {
                            T bl = ninf;
                            int bk = -1;
                            if (scan) {
#pragma unroll
                                for (int c = 0; c < CH; ++c) {
                                    const int k = COL(c);
                                    const bool up = ((sh_open[k >> 5] >> (k & 31)) & 1u) && (bk < 0 || q[c] > bl);
                                    bl = up ? q[c] : bl;
                                    bk = up ? k : bk;
                                }
                            }
#pragma unroll
                            for (int off = R; off < 32; off <<= 1) {
                                const T ol = __shfl_xor_sync(kFull, bl, off);
                                const int ok = __shfl_xor_sync(kFull, bk, off);
                                if (ok >= 0 && (bk < 0 || ol > bl || (ol == bl && ok < bk))) {
                                    bl = ol;
                                    bk = ok;
                                }
                            }
                            if (scan) {
                                ch = bk >= 0 ? bk : i;
                                if (g == 0) choice[i] = ch;
                            }
                        }
                        __syncthreads();
                        const bool newm = open && (ch == i || choice[ch] == i);
                        __syncthreads();
                        if (newm && g == 0) atomicAnd(&sh_open[i >> 5], ~(1u << (i & 31)));
                        const int left = __syncthreads_count(open && g == 0 && !newm);
                        if (tid == 0) acc_fcr += 1;
                        if (left == 0) break;
                    }
                    if (tid == 0) acc_fc += 1;
                    have_cand = true;
                    cand_forced = true;
                    if (act && g == 0) cand_p = choice[i];
                }
                if (have_cand) {
                    // ---- candidate parity (and weight when candidates are compared)
                    int pc = 0;
                    if (act && g == 0) {
                        const int k = cand_p;
                        double w = 0.0;
                        if (k >= i) {
                            if (RW) {
                                pc = Psh[i * SMAX + k];
                                if (full) w = Wsh[i * SMAX + k];
                            } else {
                                const ItemCtx ic = resolve_item(a, code);
                                const size_t off = (size_t)dets[i] * ic.tb.n_det + dets[k];
                                pc = ic.tb.P[off];
                                if (full) w = ic.tb.W64[off];
                            }
                        }
                        rowacc[i] = w;
                    }
                    const int par = __syncthreads_count(pc) & 1;
                    bool finish = false;
                    if (!full) {
                        out_par = par;
                        out_forced = cand_forced;
                        out_from_best = 0;
                        partner = cand_p;
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
                        if (sh_improve && act && g == 0) bestp[i] = (short)cand_p;
                        if (t == a.T || (a.decoder == 0 && cand_forced)) {
                            finish = true;
                            if (a.decoder == 0 && cand_forced && !sh_use_best) {
                                out_par = par;
                                out_forced = 1;
                                out_from_best = 0;
                                partner = cand_p;
                            } else {
                                out_par = sh_best_par;
                                out_forced = sh_best_forced;
                                out_from_best = 1;
                                partner = -1;
                            }
                        }
                        __syncthreads();
                    }
                    if (finish) break;
                }
            }

            // ---- compute phase, in place (FP64: the scan for (m1, m2, am) first)
            if (requeue) {
                if constexpr (std::is_same<T, float>::value) {
                    read_rows();
                } else if (act) {
#pragma unroll
                    for (int c = 0; c < CH; ++c) q[c] = G * c < s ? B2<T>::fma_(RM(c), ainv, RL(c)) : ninf;
                }
                __syncthreads();
            }
            if constexpr (std::is_same<T, float>::value) {
                update_rows();
            } else {
                if (wact) {
                    int am = 0x7fffffff;
                    T a1 = ninf, a2 = ninf, b1 = ninf, b2 = ninf;
                    int ac = 0x7fffffff, bc = 0x7fffffff;
#pragma unroll
                    for (int c = 0; c < CH; c += 2) {
                        if (G * c >= s) continue;
                        const T v = q[c];
                        const bool gt = v > a1;
                        a2 = B2<T>::mx(a2, B2<T>::mn(v, a1));
                        a1 = B2<T>::mx(a1, v);
                        ac = gt ? c : ac;
                        if (c + 1 < CH) {
                            const T w = q[c + 1];
                            const bool gw = w > b1;
                            b2 = B2<T>::mx(b2, B2<T>::mn(w, b1));
                            b1 = B2<T>::mx(b1, w);
                            bc = gw ? c + 1 : bc;
                        }
                    }
                    // column indices of the two partial maxima (ties to the smaller column)
                    int ka = ac < CH ? COL(ac) : 0x7fffffff;
                    int kb = bc < CH ? COL(bc) : 0x7fffffff;
                    combine_max(a1, a2, ka, b1, b2, kb);
                    m1 = a1;
                    m2 = a2;
                    am = ka;
#pragma unroll
                    for (int off = R; off < 32; off <<= 1) {
                        const T o1 = __shfl_xor_sync(kFull, m1, off);
                        const T o2 = __shfl_xor_sync(kFull, m2, off);
                        const int ok = __shfl_xor_sync(kFull, am, off);
                        combine_max(m1, m2, am, o1, o2, ok);
                    }
                    // FP64 (16-bit storage runs only with FP32 arithmetic)
                    static_assert(!HALF, "16-bit storage is FP32 only");
                    T sa = T(0), sb = T(0);
#pragma unroll
                    for (int c = 0; c < CH; c += 2) {
                        if (G * c >= s) continue;
                        const T u = B2<T>::ex2(B2<T>::mn(q[c], m2) - m2);
                        q[c] = u;
                        sa += u;
                        if (c + 1 < CH) {
                            const T w = B2<T>::ex2(B2<T>::mn(q[c + 1], m2) - m2);
                            q[c + 1] = w;
                            sb += w;
                        }
                    }
                    T S = sa + sb;
#pragma unroll
                    for (int off = R; off < 32; off <<= 1) S += __shfl_xor_sync(kFull, S, off);
                    const T cf = B2<T>::ex2(m2 - m1);
                    const T Aa = B2<T>::fma_(cf, S - T(1), T(1));
                    if (act) {
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            if (G * c >= s) continue;
                            const T out = -m1 - B2<T>::lg2(B2<T>::fma_(-cf, q[c], Aa));
                            *CMP(c) = out;
                        }
                        const T oam = -m2 - B2<T>::lg2(S - T(1));
                        if (owner_of<PAIR, G>(am) == g) Mt[am * PM + i] = oam;
                        if (own_diag) {
                            Dg[i] = IO::ld(Mt + i * PM + i);
                            Mt[i * PM + i] = MS(0.f);
                        }
                    }
                }
            }
            __syncthreads();
            ++t;
        }

        // ---- outputs of the shot
        if (tr_on && a.tr_partner) {
            if (act && g == 0) {
                const int pk = out_from_best ? (int)bestp[i] : partner;
                a.tr_partner[(size_t)shot * a.s_cap + i] = (int16_t)pk;
            }
            for (int k = s + tid; k < a.s_cap; k += NT) a.tr_partner[(size_t)shot * a.s_cap + k] = -1;
        }
        if (tid == 0) {
            const ItemCtx ic = resolve_item(a, code);
            if (ic.obs_pred) ic.obs_pred[ic.shot] = (uint8_t)out_par;
            if (ic.flags)
                ic.flags[ic.shot] = (uint8_t)(sh_flags | (out_forced ? F_FROM_FORCED : 0));
            if (ic.iters) ic.iters[ic.shot] = (int16_t)t;
            acc_it += (unsigned long long)t;
            acc_msg += (unsigned long long)s * s * t;
            acc_def += (unsigned long long)s;
            acc_shots += 1;
        }
        if constexpr (HELP) pb ^= 1;
        __syncthreads();
    }
    if (tid == 0 && a.ctr && acc_shots) {
        atomicAdd(a.ctr + C_ITERS, acc_it);
        atomicAdd(a.ctr + C_MSGS, acc_msg);
        atomicAdd(a.ctr + C_DEFECTS, acc_def);
        atomicAdd(a.ctr + C_TIER_MSGS + a.tier, acc_msg);
        atomicAdd(a.ctr + C_TIER_SHOTS + a.tier, acc_shots);
        atomicAdd(a.ctr + C_FC_RUNS, acc_fc);
        atomicAdd(a.ctr + C_FC_ROUNDS, acc_fcr);
    }
#undef COL
#undef RL
#undef RM
#undef CM
#undef CMP
#undef RL2
#undef RM2
}

// ------------------------------------------------------------------ tier table

// Row counts of the lists (0: not used).  FP32: 8..32 several shots per warp (decode_small.cuh),
// 48..160 one shot per block; FP64 and the FP32 reweighting decode: coarser.  The 16-row steps
// above 32 follow the defect counts (d = 13 circuit shots at p = 0.005: s = 126 +- 16).
constexpr int kRows32[kGlobalList] = {8, 16, 24, 32, 48, 64, 80, 96, 112, 128, 144, 160};
constexpr int kRowsRw32[kGlobalList] = {0, 0, 0, 32, 0, 64, 0, 96, 112, 128, 144, 160};
constexpr int kRows64[kGlobalList] = {0, 0, 0, 32, 0, 64, 0, 0, 112, 0, 0, 0};

// Bytes of one RW scratch slot: W [SMAX][SMAX] doubles, path distances [warps][nodes] doubles,
// qubit weights [units] doubles, predecessors [warps][nodes] words, parity [SMAX][SMAX] bytes.
inline int64_t rw_slot_layout(int smax, int nt, int nodes, int units) {
    const int64_t b = 8 * ((int64_t)smax * smax + (int64_t)(nt / 32) * nodes + units) +
                      4 * (int64_t)(nt / 32) * nodes + (int64_t)smax * smax;
    return (b + 255) / 256 * 256;
}

template <typename T, int CH, int G, typename MS = T, bool RW = false>
size_t smem_bytes_of() {
    constexpr int SMAX = CH * G;
    return nref_offset<T, MS>(SMAX, G, helper_warp(SMAX, (int)sizeof(T), (int)sizeof(MS), RW)) +
           (sizeof(MS) == 2 ? (size_t)SMAX * sizeof(float) : 0) + (size_t)SMAX * 2 + 16;
}

// Resident blocks per SM of a kernel on the current device, asked for once per kernel and device.
constexpr int kOccDevices = 16;
template <typename K>
cudaError_t resident_blocks(K kern, int threads, size_t smem, std::atomic<int>* cache, int* per_sm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kOccDevices && (*per_sm = cache[dev].load()) > 0) return cudaSuccess;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (*per_sm < 1) return cudaErrorInvalidConfiguration;
    if (dev >= 0 && dev < kOccDevices) cache[dev].store(*per_sm);
    return cudaSuccess;
}

// Grid of a persistent launch: every resident block, or one per item where the items are fewer.
inline int persistent_grid(int resident, const DecodeArgs& a) {
    return a.max_items > 0 && a.max_items < resident ? (int)a.max_items : resident;
}

template <typename T, int CH, int G, bool TRACE, typename MS = T>
cudaError_t run_tier(const DecodeArgs& a, int num_sms, cudaStream_t st, bool prepare_only) {
    const size_t smem = smem_bytes_of<T, CH, G, MS>();
    auto kern = decode_smem_kernel<T, CH, G, TRACE, false, MS>;
    if (prepare_only)
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    constexpr int NT = block_threads(CH, G, (int)sizeof(T), (int)sizeof(MS), false);
    static std::atomic<int> cache[kOccDevices] = {};
    int per_sm = 0;
    cudaError_t e = resident_blocks(kern, NT, smem, cache, &per_sm);
    if (e != cudaSuccess) return e;
    kern<<<persistent_grid(per_sm * num_sms, a), NT, smem, st>>>(a);
    return cudaGetLastError();
}

// Every tier has a production instantiation and a traced one (tests).
template <typename T, int CH, int G, typename MS = T>
cudaError_t run_tier2(const DecodeArgs& a, int num_sms, cudaStream_t st, bool prep) {
    const bool tr = a.tr_lambda != nullptr || a.tr_partner != nullptr;
    if (prep) {
        cudaError_t e = run_tier<T, CH, G, false, MS>(a, num_sms, st, true);
        return e != cudaSuccess ? e : run_tier<T, CH, G, true, MS>(a, num_sms, st, true);
    }
    return tr ? run_tier<T, CH, G, true, MS>(a, num_sms, st, false)
              : run_tier<T, CH, G, false, MS>(a, num_sms, st, false);
}

}  // namespace
}  // namespace bp4m
