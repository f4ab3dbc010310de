// Exact full-data pass (Alg. 1 last step, Eq. 1) with the distance
// contraction on the fifth-generation tensor cores.
//
// Results are those of the plain definition used everywhere in exact mode:
// label = argmin_j d32(x, c_j) with the lowest index on ties, where d32 is
// the FP32 direct form, and f = the exact sum of d32(x, c_label) rounded once.
// The tensor cores only narrow the centroids down:
//
//   * each x is split into xh = bf16(x) and xm = bf16(x - xh), every -2 c
//     likewise into ch and cm; a tile of 128 rows takes the MMAs xh.ch, xh.cm
//     and xm.ch (tcgen05.mma kind::f16, BF16 operands, M = 128, N = k rounded
//     up to 16, K = 16) on top of an FP32 accumulator in tensor memory that
//     starts from ||c_j||^2 (a little less, see below), so the accumulator is
//     g_j = ||c_j||^2 - 2 x.c_j;
//   * the epilogue takes the least g of a row from the tensor-memory load
//     itself (tcgen05.ld.red, sm_103a), adds the certificate's threshold and
//     keeps the bit mask of the columns below: no other centroid can be the
//     d32 argmin.  Each remaining column costs one packed add and one funnel
//     shift that moves its sign into the mask;
//   * the label and the distance are the least d32 among the masked columns,
//     lowest index on ties: one for almost every row, and a row with more
//     costs its own extra distances only.
//
// Error of g_j against ||c_j||^2 - 2 x.c_j (exact reals).  BF16 keeps 8
// significant bits: |x - xh| <= 2^-8 |x|, and x - xh is exact in FP32, so
// |x - xh - xm| <= 2^-16 |x|; c likewise.  The products left out are xm cm,
// (x - xh - xm) c and (xh + xm)(c - ch - cm): per dimension at most
// 3 2^-16 (1 + 2^-6) |x c|.  The products taken are exact in FP32.  The
// accumulation is taken to add at most (K + 1) 2^-23 of the magnitude
// accumulated so far per MMA instruction (products aligned and truncated once
// against the largest term, then added): 3 ksteps instructions on magnitudes
// of at most (1 + 2^-6)(||c_j||^2 + 2 ||x|| ||c_j||).  ||c_j||^2 itself is an
// FP32 FMA chain (64 2^-24).  tcx_gamma sums these with a quarter to spare; it
// bounds |g_j - (||c_j||^2 - 2 x.c_j)| by gB (||c_j||^2 + 2 ||x|| ||c_j||), at
// most gB (2 ||c_j||^2 + ||x||^2).
//
// Threshold.  With the largest ||c||^2 in that bound, one far centroid would
// make every row keep the centroids near it.  So the accumulator starts from
// (1 - 2 gB) ||c_j||^2 (less by 0.005 gB, which covers its roundings): then the squared distance D_j =
// ||x||^2 + ||c_j||^2 - 2 x.c_j is at least ||x||^2 + g_j - gB ||x||^2, and for
// the centroid of the least g, g1, at most
//   D <= ||x||^2 + g1 + gB (||x||^2 + 4.01 N),   N = ||c||^2 of that centroid.
// N <= (||x|| + sqrt D)^2 <= 1.5 ||x||^2 + 3 D, hence (gB < 2^-12)
//   D <= d1 = 1.006 (max(0, ||x||^2 + g1) + 7.2 gB ||x||^2),
// and a centroid whose g exceeds g1 by more than
//   thr = gB (2 ||x||^2 + 4.01 min(max ||c||^2, 1.5 ||x||^2 + 3 d1)) + gp2 d1
// has a D larger by gp2 D and more, so a larger direct form (its relative
// error is in gp2).  A gap below 2^-60 is never accepted (subnormal data), and
// rows whose magnitudes come near the FP32 range keep all columns.  Up to 32
// centroids the minimum is left out (a mask of one word costs little).
// Measured (the call, log-normal rows with sigma = 3, k = 200) with the largest
// ||c||^2 alone in the bound and so: 10^6 x 16 1,886 and 153 us, 10^6 x 32 1,899
// and 191 us, 5 10^6 x 8 8,802 and 514 us.
//
// Shift.  The bound grows with the distance from the origin, the gaps between
// distances do not: rows with a mean of a hundred standard deviations would
// keep nearly all columns.  So the operands are x - u and c - u, u the mean of
// up to 16 centroids, where that at least halves their mean ||c||^2 (any u
// leaves ||x - c|| as it is); the direct form takes x and c as they are.
// Each difference is rounded once, which changes ||c - u||^2 - 2 (x - u).(c - u)
// by at most 2^-22 of the magnitudes in the bound (in tcx_gamma) and ||x - u||^2
// by 2^-22 of itself (in xn2).  Up to 32 centroids (one mask word) keeping
// every column costs less than the FP32-ALU pass, and nothing is shifted.
// Measured, kernel alone, rows with a mean of 300 standard deviations: 10^6 x
// 16, k = 200 2,110 -> 93 us; 2 10^6 x 32, k = 50 758 -> 99 us; 2 10^6 x 64, k =
// 100 2,650 -> 207 us.  With both, centred rows take 1% longer (10^7 x 64, k =
// 100: 867 -> 879 us).
//
// CTA roles (one CTA per SM, persistent over tiles blockIdx.x + i grid): the
// warp after the epilogue warps issues the copies of X, the next one the
// MMAs; NG epilogue warpgroups, group b taking the tiles i = b (mod NG) with
// accumulator b and operand buffer b.  A thread of a group owns one row of
// its tile: it reads the row from the stage into registers (which frees the
// stage), writes xh and xm in the 128-byte-swizzle K-major layout, and keeps
// x for the direct form.
//
// X comes in two ways.  n % 4 == 0: 2-D TMA copies of 128 rows x 32 columns,
// 128-byte swizzle, zero-filled past n.  Other n: the 128 rows are one
// contiguous piece of X, brought by one bulk copy and read with a row stride
// of n floats (odd n: no bank conflicts).
//
// What bounds it: latency within a tile (wait, split, MMA, tensor-memory load,
// distance are one chain per group; 48% issue, 25% of the DRAM rate at 10^6 x
// 16, k = 25), hence as many groups as fit.  The former passes (three
// split-TF32 products, two reads of the accumulator with a compare and a
// select per column, rows rebuilt from two tiles) issued 2-3 times as many
// instructions: 10^7 x 64, k = 100: 2.83 ms then, 0.88 ms now (2.9 TB/s of
// rows); 4 10^6 x 32, k = 50: 228 and 181 us; 10^6 x 16, k = 25: 49 and 33 us.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "bm_device.cuh"
#include "bm_tcgen05.cuh"

namespace bm {

constexpr int kTxRows = 128;                  // rows per tile (MMA M)
constexpr int kTxAtomBytes = kTxRows * 128;   // 128 rows of 128 bytes
constexpr int kTxMaxStages = 8;
__host__ __device__ constexpr int tx_threads(int groups) { return 32 * (4 * groups + 2); }

struct TxShape {
    int groups;      // epilogue warpgroups = accumulators = operand buffers
    int Npad;        // MMA N: k rounded up to 16
    int acc_stride;  // tensor-memory columns per accumulator (k rounded up to 32)
    int tmem_cols;   // columns allocated
    int stages;      // X tiles in flight
    int flat;        // 1: X by 1-D bulk copies (n % 4 != 0)
    int cf;          // 1: FP32 centroids in shared memory, 0: read from global memory
    tc::WaitLimit wait;  // limit of every bounded wait
};

// Rows of NP <= 32 hold xh and xm side by side in 128 bytes, rows of 64 in two
// atoms; the centroid tiles likewise.
template <int NP>
struct TxK {
    static constexpr int KW = NP < 16 ? 16 : NP;             // columns of a piece
    static constexpr int atoms = NP > 32 ? 2 : 1;
    static constexpr int steps = KW / 16;                    // K = 16 instructions per product
    static constexpr int CS = NP + 4;                        // FP32 centroid rows: odd number of 16-byte units
};

// Shared memory (1024-byte aligned pieces): [X stages][operand buffers: groups
// x atoms x 16 KB][ch, cm: atoms x Npad x 128 B][-C: k x CS floats][CC].
template <int NP>
size_t tx_smem_bytes(const TxShape& s, int k) {
    using K = TxK<NP>;
    return 1024 + (size_t)(s.stages + s.groups) * K::atoms * kTxAtomBytes + (size_t)K::atoms * s.Npad * 128 +
           (s.cf ? (size_t)k * K::CS * 4 : 0) + (size_t)s.acc_stride * 4;
}

// MW: 32-column words of a row's mask (1: k <= 32, 4: k <= 128, 8: k <= 256).
template <int NP, int NG, int MW>
__global__ void __launch_bounds__(tx_threads(NG), 1)
tcx_fullpass_kernel(const __grid_constant__ CUtensorMap tmap, const float* __restrict__ X, long long m, int n,
                    const float* __restrict__ Cw, int cw, int k, const double* sel_f, int W, int* __restrict__ labels,
                    Globals* g, float gB, float gp2, int incumbent, TxShape sh) {
    using K = TxK<NP>;
    constexpr int kStage = K::atoms * kTxAtomBytes;
    constexpr bool kShift = MW > 1;              // see "Shift" in the file comment
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (tc::s_addr(smem_raw) & 1023)) & 1023);
    const int S = sh.stages;
    unsigned char* xs = base;                                        // X stages
    unsigned char* xb = xs + (size_t)S * kStage;                     // xh | xm, one per group
    unsigned char* cb = xb + (size_t)NG * kStage;                    // ch | cm
    float* Cf = reinterpret_cast<float*>(cb + (size_t)K::atoms * sh.Npad * 128);   // -C (sh.cf)
    float* CC = Cf + (sh.cf ? (size_t)k * K::CS : 0);                // (1 - 2 gB) ||c_j||^2, +inf past k
    constexpr int kEpi = 4 * NG, kProducer = kEpi, kMma = kEpi + 1, kThreads = tx_threads(NG);
    __shared__ __align__(8) unsigned long long full[kTxMaxStages], empty[kTxMaxStages], conv[NG], accf[NG];
    __shared__ unsigned tmem_slot;
    __shared__ int abort_flag;
    __shared__ unsigned __int128 red128[kThreads / 32];
    __shared__ unsigned long long red64[kThreads / 32];
    __shared__ unsigned int redu[kThreads / 32];
    __shared__ __align__(16) float mu_s[NP], sq_s[NP];               // the shift; mean squares
    __shared__ int wsel;
    __shared__ bool last;

    if (g->nonfinite) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int* abort = &abort_flag;
    if (tid == 0) {
        int best = 0;
        if (sel_f)
            for (int w = 1; w < W; ++w)
                if (sel_f[w] < sel_f[best]) best = w;
        wsel = best;
        abort_flag = 0;
        for (int s = 0; s < S; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 4); }
        for (int b = 0; b < NG; ++b) { tc::mbar_init(&conv[b], 4); tc::mbar_init(&accf[b], 1); }
        tc::mbar_init_fence();
    }
    if (warp == kMma) tc::tmem_alloc(&tmem_slot, (unsigned)sh.tmem_cols);
    __syncthreads();
    const float* C = Cw + (long long)wsel * k * cw;
    // the FP32 copy of -c and the shift
    if (sh.cf)
        for (int e = tid; e < k * NP; e += kThreads) {
            const int j = e / NP, d = e % NP;
            Cf[(size_t)j * K::CS + d] = d < cw ? -C[(size_t)j * cw + d] : 0.f;
        }
    if (kShift && tid < NP) {
        const int cnt = min(k, 16);
        const float w = 1.f / (float)cnt;
        float mu = 0.f, sq = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < cnt && tid < cw) {
                const float c = C[(size_t)(i * k / cnt) * cw + tid];
                mu = __fmaf_rn(c, w, mu);
                sq = __fmaf_rn(c * w, c, sq);
            }
        mu_s[tid] = mu;
        sq_s[tid] = sq;
    }
    // the operand buffers' columns that no row writes (NP = 8) are zero
    if (NP < 16)
        for (int e = tid; e < NG * kStage / 16; e += kThreads)
            reinterpret_cast<uint4*>(xb)[e] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const float4* mu4 = reinterpret_cast<const float4*>(mu_s);
    auto c4 = [&](int j, int q) {                                    // elements 4 q .. 4 q + 3 of centroid j
        if (sh.cf) {
            const float4 v = reinterpret_cast<const float4*>(Cf + (size_t)j * K::CS)[q];
            return make_float4(-v.x, -v.y, -v.z, -v.w);
        }
        return 4 * q < cw ? __ldg(reinterpret_cast<const float4*>(C + (size_t)j * cw) + q)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto sub4 = [](const float4& v, const float4& u) {
        return make_float4(__fsub_rn(v.x, u.x), __fsub_rn(v.y, u.y), __fsub_rn(v.z, u.z), __fsub_rn(v.w, u.w));
    };
    // Shift where that halves the mean ||c||^2 of those centroids, i.e. where
    // ||u||^2 is more than half of it (every warp decides, alike).
    bool shift = false;
    if (kShift) {
        float mu2 = 0.f, sq = 0.f;
        for (int d = lane; d < NP; d += 32) {
            mu2 = __fmaf_rn(mu_s[d], mu_s[d], mu2);
            sq += sq_s[d];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mu2 += __shfl_xor_sync(0xffffffffu, mu2, o);
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
        }
        shift = 2.f * mu2 > sq;
    }
    // ||c||^2 and its upper bound, a thread per centroid; the operands
    static_assert(kThreads >= 256, "a thread per accumulator column");
    {
        float cc = 0.f, up = 0.f;
        auto add = [&](float c) {
            cc = __fmaf_rn(c, c, cc);
            up = __fmaf_ru(c, c, up);
        };
        if (tid < k)
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) {
                float4 v = c4(tid, q);
                if (shift) v = sub4(v, mu4[q]);
                add(v.x); add(v.y); add(v.z); add(v.w);
            }
        if (tid < sh.acc_stride) CC[tid] = tid < k ? cc * (1.f - 2.005f * gB) : __int_as_float(0x7f800000);
        const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(up));
        if (lane == 0) redu[warp] = mx;
    }
    for (int e = tid; e < sh.Npad * (K::KW / 8); e += kThreads) {
        const int j = e / (K::KW / 8), c = e % (K::KW / 8);
        float v[8] = {};
        if (j < k && 8 * c < NP) {
            float4 a = c4(j, 2 * c), b = c4(j, 2 * c + 1);
            if (shift) { a = sub4(a, mu4[2 * c]); b = sub4(b, mu4[2 * c + 1]); }
            v[0] = -2.f * a.x; v[1] = -2.f * a.y; v[2] = -2.f * a.z; v[3] = -2.f * a.w;
            v[4] = -2.f * b.x; v[5] = -2.f * b.y; v[6] = -2.f * b.z; v[7] = -2.f * b.w;
        }
        uint4 h, l;
        tc::split_bf16(v, h, l);
        const int cm = K::atoms == 2 ? c : K::KW / 8 + c;            // chunk of cm in its row
        *reinterpret_cast<uint4*>(cb + (size_t)j * 128 + ((c ^ (j & 7)) << 4)) = h;
        *reinterpret_cast<uint4*>(cb + (K::atoms == 2 ? (size_t)sh.Npad * 128 : 0) + (size_t)j * 128 +
                                  ((cm ^ (j & 7)) << 4)) = l;
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = tmem_slot;
    const long long ntiles = (m + kTxRows - 1) / kTxRows;
    const long long grid = gridDim.x;

    unsigned __int128 facc = 0;
    unsigned int inex = 0, resc = 0;
    long long issued = 0;             // producer: copies issued; MMA warp: tiles committed
    if (warp == kProducer) {
        // ---------------------------------------------------------- producer
        if (lane == 0) {
            long long it = 0;
            int s = 0;
            unsigned ph = 0;                                // (it / S) & 1, kept incrementally
            for (;; ++it) {
                const long long tile = blockIdx.x + it * grid;
                if (tile >= ntiles) break;
                if (it >= S && !tc::wait(&empty[s], ph ^ 1u, abort, g, sh.wait)) break;
                if (sh.flat) {
                    const long long rows = min((long long)kTxRows, m - tile * kTxRows);
                    const unsigned bytes = (unsigned)(rows * n * 4) & ~15u;     // the rest by the row's thread
                    tc::expect_tx(&full[s], bytes);
                    if (bytes) tc::bulk_g2s(xs + (size_t)s * kStage, X + tile * kTxRows * n, bytes, &full[s]);
                } else {
                    tc::expect_tx(&full[s], (unsigned)kStage);
                    for (int a = 0; a < K::atoms; ++a)
                        tc::tma_load_2d(xs + (size_t)s * kStage + (size_t)a * kTxAtomBytes, &tmap, 32 * a,
                                        (int)(tile * kTxRows), &full[s]);
                }
                if (++s == S) { s = 0; ph ^= 1u; }
            }
            issued = it;
        }
    } else if (warp == kMma) {
        // --------------------------------------------------------------- MMA
        if (lane == 0) {
            const unsigned idesc = tc::idesc_bf16(kTxRows, sh.Npad);
            const unsigned bh = tc::s_addr(cb);
            const unsigned bm = K::atoms == 2 ? bh + (unsigned)sh.Npad * 128 : bh + K::KW * 2;
            long long it = 0;
            for (;; ++it) {
                const long long tile = blockIdx.x + it * grid;
                if (tile >= ntiles) break;
                const int b = (int)(it % NG);
                if (!tc::wait(&conv[b], (unsigned)((it / NG) & 1), abort, g, sh.wait)) break;
                tc::fence_after();
                const unsigned ah = tc::s_addr(xb + (size_t)b * kStage);
                const unsigned am = K::atoms == 2 ? ah + kTxAtomBytes : ah + K::KW * 2;
                const unsigned d = tmem + (unsigned)(b * sh.acc_stride);
#pragma unroll
                for (int kk = 0; kk < K::steps; ++kk) {
                    tc::mma_bf16(d, tc::desc_sw128(am + 32 * kk), tc::desc_sw128(bh + 32 * kk), idesc, 1);
                    tc::mma_bf16(d, tc::desc_sw128(ah + 32 * kk), tc::desc_sw128(bm + 32 * kk), idesc, 1);
                }
#pragma unroll
                for (int kk = 0; kk < K::steps; ++kk)
                    tc::mma_bf16(d, tc::desc_sw128(ah + 32 * kk), tc::desc_sw128(bh + 32 * kk), idesc, 1);
                tc::commit(&accf[b]);
            }
            issued = it;
        }
    } else {
        // --------------------------------------------------- epilogue groups
        // (a body of its own for shifted rows: a branch per row cost the
        // unshifted ones 2 to 5%)
        auto epilogue = [&](auto shifted) __attribute__((always_inline)) {
        const Grids gr = grids_from_maxbits(g->maxbits);
        const float cmax2 = __uint_as_float(__reduce_max_sync(0xffffffffu, lane < kThreads / 32 ? redu[lane] : 0u));
        // (each constant of the threshold has 2^-10 of itself to spare for roundings)
        const float k_max = fmaxf(4.02f * gB * cmax2, 0x1p-60f);
        const float k_gp = gp2 * (1.f + 0x1p-10f), k_own = 12.4f * gB + k_gp;
        const int b = warp >> 2, q4 = warp & 3;
        const int r = q4 * 32 + lane;                        // row within the tile = TMEM lane
        unsigned char* xrow = xb + (size_t)b * kStage + r * 128;
        const unsigned trow = tmem + ((unsigned)(q4 * 32) << 16) + (unsigned)(b * sh.acc_stride);
        const int nw = MW == 1 ? 1 : sh.acc_stride >> 5;
        const FastSum fs(gr.gf);
        unsigned long long fast = 0;
        auto init_acc = [&]() {                              // the accumulator starts from CC
#pragma unroll 1
            for (int w = 0; w < nw; ++w) tc::st32_shared(trow + 32u * w, CC + 32 * w);
            tc::wait_st();
        };
        init_acc();
        int s = b % S;
        long long use = b / S;
        for (long long it = b, u = 0;; it += NG, ++u) {
            const long long tile = blockIdx.x + it * grid;
            if (tile >= ntiles) break;
            const unsigned char* st = xs + (size_t)s * kStage;
            const long long row = tile * kTxRows + r;
            const bool valid = row < m;
            // 1. the row: registers, then xh and xm into the group's buffer;
            //    the stage is free once every warp of the group has read it.
            //    (With an odd stage count two groups share a stage in turn:
            //    the previous use is over before its next copy is waited for,
            //    so the wait cannot meet an older phase of the same parity.)
            if (S % NG != 0 && use > 0 && !tc::wait_warp(&empty[s], (unsigned)((use - 1) & 1), abort, g, sh.wait)) break;
            if (!tc::wait_warp(&full[s], (unsigned)(use & 1), abort, g, sh.wait)) break;
            float x[NP];
            if (sh.flat) {
                const float* p = reinterpret_cast<const float*>(st) + r * n;
                const long long have = (min((long long)kTxRows, m - tile * kTxRows) * n) & ~3ll;
#pragma unroll
                for (int d = 0; d < NP; ++d) {
                    x[d] = 0.f;
                    if (d < n && valid) x[d] = r * n + d < have ? p[d] : __ldg(X + row * n + d);
                }
            } else {
#pragma unroll
                for (int q = 0; q < NP / 4; ++q) {
                    const float4 v = *reinterpret_cast<const float4*>(st + (q >> 3) * kTxAtomBytes + r * 128 +
                                                                      (((q & 7) ^ (r & 7)) << 4));
                    x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
                }
            }
            __syncwarp();
            if (lane == 0) tc::arrive(&empty[s]);
            float2 n2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < NP / 8; ++c) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = x[8 * c + i];
                if constexpr (decltype(shifted)::value) {
                    const float4 u0 = mu4[2 * c], u1 = mu4[2 * c + 1];
                    v[0] = __fsub_rn(v[0], u0.x); v[1] = __fsub_rn(v[1], u0.y);
                    v[2] = __fsub_rn(v[2], u0.z); v[3] = __fsub_rn(v[3], u0.w);
                    v[4] = __fsub_rn(v[4], u1.x); v[5] = __fsub_rn(v[5], u1.y);
                    v[6] = __fsub_rn(v[6], u1.z); v[7] = __fsub_rn(v[7], u1.w);
                }
#pragma unroll
                for (int i = 0; i < 8; i += 2)
                    n2 = __ffma2_ru(make_float2(v[i], v[i + 1]), make_float2(v[i], v[i + 1]), n2);
                uint4 h, l;
                tc::split_bf16(v, h, l);
                const int cm = K::atoms == 2 ? c : K::KW / 8 + c;
                *reinterpret_cast<uint4*>(xrow + ((c ^ (r & 7)) << 4)) = h;
                *reinterpret_cast<uint4*>(xrow + (K::atoms == 2 ? kTxAtomBytes : 0) + ((cm ^ (r & 7)) << 4)) = l;
            }
            tc::fence_proxy_async();
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::arrive(&conv[b]);
            s += NG;
            while (s >= S) { s -= S; ++use; }
            float xn2 = __fadd_ru(n2.x, n2.y);
            if constexpr (decltype(shifted)::value) xn2 = __fmul_ru(xn2, 1.f + 0x1p-21f);
            // what the threshold takes from ||x||^2
            const float d_lo = __fmul_ru(7.3f * gB, xn2);
            const float t_max = __fmaf_ru(2.002f * gB, xn2, k_max);
            const bool sane = t_max < 0x1p106f;               // ||x||^2 + 2 cmax^2 below 2^122; else: every column
            const float t_own = fmaxf(__fmul_ru(8.2f * gB, xn2), 0x1p-60f);
            // 2. the accumulator: least g, then the columns within the threshold
            if (!tc::wait_warp(&accf[b], (unsigned)(u & 1), abort, g, sh.wait)) break;
            tc::fence_after();
            unsigned va[32], mk[MW];
            float g1 = __int_as_float(0x7f800000);
#pragma unroll 1
            for (int w = 0; w < nw; ++w) {
                float mn;
                tc::ld32_min(trow + 32u * w, va, mn);
                g1 = fminf(g1, mn);
            }
            // every column with g <= g1 + thr lies strictly below L
            const float d1 = __fmaf_ru(1.007f, fmaxf(0.f, __fadd_ru(g1, xn2)), d_lo);
            float thr = __fmaf_ru(k_gp, d1, t_max);
            if (MW > 1) thr = fminf(thr, __fmaf_ru(k_own, d1, t_own));
            const float L = __fadd_ru(g1, thr);
            int cnt = 0;
#pragma unroll
            for (int w = 0; w < MW; ++w) {
                mk[w] = 0;
                if (w < nw) {
                    if (MW > 1) tc::ld32(trow + 32u * w, va);  // (one word: still in registers)
                    mk[w] = tc::below_mask32(va, L);
                    if (!sane) mk[w] = 32 * w + 32 <= k ? ~0u : ~0u << (32 * w + 32 - k);
                    cnt += __popc(mk[w]);
                }
            }
            init_acc();                                       // for the group's next tile
            // 3. label and distance: the least d32 among those columns
            auto d32j = [&](int j) {
                float acc = 0.f;
                auto add4 = [&](int q, const float4& c) {      // c holds -c
                    float2 t0 = __fadd2_rn(make_float2(x[4 * q], x[4 * q + 1]), make_float2(c.x, c.y));
                    float2 t1 = __fadd2_rn(make_float2(x[4 * q + 2], x[4 * q + 3]), make_float2(c.z, c.w));
                    t0 = __fmul2_rn(t0, t0);
                    t1 = __fmul2_rn(t1, t1);
                    acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, t0.x), t0.y), t1.x), t1.y);
                };
                if (sh.cf) {
                    const float4* cj = reinterpret_cast<const float4*>(Cf + (size_t)j * K::CS);
#pragma unroll
                    for (int q = 0; q < NP / 4; ++q) add4(q, cj[q]);
                } else {
                    const float* cj = C + (size_t)j * cw;
#pragma unroll
                    for (int q = 0; q < NP / 4; ++q)
                        if (4 * q < cw) {
                            const float4 c = __ldg(reinterpret_cast<const float4*>(cj) + q);
                            add4(q, make_float4(-c.x, -c.y, -c.z, -c.w));
                        }
                }
                return acc;
            };
            auto lowest = [&]() {                              // of the columns left (bit 31 first)
                int j = 32 * MW - 1;
#pragma unroll
                for (int w = MW - 1; w >= 0; --w)
                    if (mk[w]) j = 32 * w + __clz((int)mk[w]);
                return j;
            };
            int lab = min(lowest(), k - 1);
            float dv = d32j(lab);
            if (!valid) cnt = 0;
            if (cnt > 1) ++resc;
            while (__any_sync(0xffffffffu, cnt > 1)) {         // the other candidates, in ascending order
                if (cnt > 1) {
                    int j = lowest();
#pragma unroll
                    for (int w = 0; w < MW; ++w)
                        if (w == (j >> 5)) mk[w] &= ~(0x80000000u >> (j & 31));
                    --cnt;
                    j = min(lowest(), k - 1);
                    const float d = d32j(j);
                    if (d < dv) { dv = d; lab = j; }
                }
            }
            const bool quick = dv >= fs.lim && dv < __int_as_float(0x7f800000);
            if (valid && quick) fast += fs.units(dv);
            if (__any_sync(0xffffffffu, valid && !quick))
                if (valid && !quick) acc_obj(facc, dv, gr.gf, inex);
            if (valid && labels) labels[row] = lab;
            if ((u & 63) == 63) { facc += (unsigned __int128)fast << 40; fast = 0; }
        }
        facc += (unsigned __int128)fast << 40;
        };
        if (kShift && shift) epilogue(std::true_type{});
        else epilogue(std::false_type{});
    }

    // teardown.  Without an abort every copy and every MMA was consumed by a
    // wait of the epilogue.  After an abort (a bounded wait ran out), once
    // every role has stopped (the barrier below; the flag is final then),
    // the producer waits for its copies still in flight (only the last S can
    // be: each earlier stage was released by the epilogue after its copy
    // landed) and the MMA thread for its last commit, which covers every MMA
    // it issued, so that nothing writes this CTA's shared or tensor memory
    // after it is released.
    tc::fence_before();
    __syncthreads();
    if (*abort) {
        if (warp == kProducer && lane == 0)
            for (long long i = (issued > S ? issued - S : 0); i < issued; ++i)
                for (unsigned p = 0; p < (1u << 22) && !tc::try_wait(&full[i % S], (unsigned)((i / S) & 1)); ++p) {}
        if (warp == kMma && lane == 0 && issued > 0)
            for (unsigned p = 0;
                 p < (1u << 22) && !tc::try_wait(&accf[(issued - 1) % NG], (unsigned)(((issued - 1) / NG) & 1));
                 ++p) {}
        __syncthreads();
    }
    if (warp == kMma) {
        tc::fence_after();
        tc::tmem_dealloc(tmem, (unsigned)sh.tmem_cols);
    }
    // objective: CTA reduction, then the grid-wide total (last CTA rounds it)
    const unsigned __int128 F = warp_sum_u128(facc);
    const unsigned long long IR = warp_sum(((unsigned long long)inex << 32) | resc);
    if (lane == 0) { red128[warp] = F; red64[warp] = IR; }
    __syncthreads();
    if (tid == 0) {
        unsigned __int128 T = 0;
        unsigned long long ir = 0;
        for (int i = 0; i < kThreads / 32; ++i) { T += red128[i]; ir += red64[i]; }
        for (int i = 0; i < 4; ++i) {
            const unsigned long long chunk = (unsigned long long)((T >> (32 * i)) & 0xffffffffu);
            if (chunk) atomicAdd(&g->obj_words[i], chunk);
        }
        if (ir >> 32) atomicAdd(&g->inexact, ir >> 32);
        if (ir & 0xffffffffull) atomicAdd(&g->rescored, ir & 0xffffffffull);
        __threadfence();
        last = (atomicAdd(&g->done_ctas, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (last && tid == 0) {
        __threadfence();
        unsigned __int128 T = 0;
        for (int i = 0; i < 4; ++i) {
            T += (unsigned __int128)atomicAdd(&g->obj_words[i], 0ull) << (32 * i);
            g->obj_words[i] = 0;
        }
        const double f = u128_to_double(T, grids_from_maxbits(g->maxbits).gf);
        g->f_full = f;
        if (incumbent && f < g->f_incumbent) g->f_incumbent = f;
        g->best_worker = wsel;
        g->done_ctas = 0;
    }
}

// ------------------------------------------------------------ host side
namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// Groups: as many as the registers of a row allow (NP = 64: 2, 32: 3, else 4,
// or 6 when one mask word holds k: 10^6 x 16, k = 25 took 40 us with 4) or
// tensor memory (k > 128: 2).  Stages: as many as fit in 221 KB (the rest is
// the kernel's static arrays), a multiple of the group count or, with two
// groups, also 3 (see the kernel); the FP32 centroids are read from global
// memory where they do not fit beside the stages.
__host__ __device__ constexpr int tx_groups(int NP, int MW) { return NP == 64 || MW == 8 ? 2 : NP == 32 ? 3 : MW == 1 ? 6 : 4; }
template <int NP>
bool tx_shape(int k, TxShape& s) {
    if (k < 1 || k > 256) return false;
    s.Npad = (k + 15) & ~15;
    s.acc_stride = (s.Npad + 31) & ~31;
    s.groups = tx_groups(NP, k <= 32 ? 1 : k <= 128 ? 4 : 8);
    s.tmem_cols = 32;
    while (s.tmem_cols < s.groups * s.acc_stride) s.tmem_cols <<= 1;
    constexpr size_t kDyn = 221 * 1024;
    for (s.cf = 1; s.cf >= 0; --s.cf)
        for (s.stages = kTxMaxStages; s.stages >= s.groups; --s.stages)
            if ((s.stages % s.groups == 0 || (s.groups == 2 && s.stages == 3)) && tx_smem_bytes<NP>(s, k) <= kDyn)
                return true;
    return false;
}

template <int NP, int MW>
cudaError_t launch_t(const CUtensorMap& tm, const float* X, long long m, int n, const float* C, int cw, int k,
                     const double* sel_f, int W, int* labels, Globals* g, float gB, float gp2, int incumbent, int sms,
                     const TxShape& sh, cudaStream_t st) {
    constexpr int NG = tx_groups(NP, MW), threads = tx_threads(NG);
    const size_t smem = tx_smem_bytes<NP>(sh, k);
    cudaFuncAttributes fa;
    cudaError_t e = func_attributes((const void*)tcx_fullpass_kernel<NP, NG, MW>, &fa);
    if (e != cudaSuccess) return e;
    const int warps_alloc = (threads / 32 + 3) & ~3;            // warps are given registers in fours
    if ((long long)fa.numRegs * 32 * warps_alloc > 65536 || smem + fa.sharedSizeBytes > 227 * 1024)
        return cudaErrorNotSupported;
    e = allow_max_smem((const void*)tcx_fullpass_kernel<NP, NG, MW>);
    if (e != cudaSuccess) return e;
    const long long tiles = (m + kTxRows - 1) / kTxRows;
    const long long grid = std::max<long long>(1, std::min<long long>((long long)sms, tiles));
    tcx_fullpass_kernel<NP, NG, MW><<<(unsigned)grid, threads, smem, st>>>(tm, X, m, n, C, cw, k, sel_f, W, labels, g,
                                                                           gB, gp2, incumbent, sh);
    return cudaGetLastError();
}

// Certificate factor of the split products (see the file comment).
float tcx_gamma(int steps) {
    return 1.25f * (3.0f * 0x1p-16f * (1.f + 0x1p-6f) + (3 * steps) * 17 * 0x1p-23f * (1.f + 0x1p-6f) + 0x1p-18f +
                    0x1p-21f);
}

// Limits of the bounded waits of the next launches (process-wide).
std::atomic<unsigned> g_wait_polls{tc::kDefaultWait.polls}, g_wait_ns{tc::kDefaultWait.ns};

template <int NP>
cudaError_t launch_np(const float* X, long long m, int n, const float* C, int cw, int k, const double* sel_f, int W,
                      int* labels, Globals* g, float gB, float gp2, int incumbent, int sms, cudaStream_t st) {
    TxShape sh;
    if (!tx_shape<NP>(k, sh)) return cudaErrorNotSupported;
    sh.wait = {g_wait_polls.load(), g_wait_ns.load()};
    sh.flat = n % 4 != 0;
    CUtensorMap tm{};
    if (!sh.flat) {
        const cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)m};
        const cuuint64_t strides[1] = {(cuuint64_t)n * 4};
        const cuuint32_t box[2] = {32, kTxRows};
        const cuuint32_t estr[2] = {1, 1};
        const CUresult r = encode_fn()(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(X), dims, strides,
                                       box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorNotSupported;
    }
    const float gBt = std::max(gB, tcx_gamma(TxK<NP>::steps));
    if (k <= 32)
        return launch_t<NP, 1>(tm, X, m, n, C, cw, k, sel_f, W, labels, g, gBt, gp2, incumbent, sms, sh, st);
    if (k <= 128)
        return launch_t<NP, 4>(tm, X, m, n, C, cw, k, sel_f, W, labels, g, gBt, gp2, incumbent, sms, sh, st);
    return launch_t<NP, 8>(tm, X, m, n, C, cw, k, sel_f, W, labels, g, gBt, gp2, incumbent, sms, sh, st);
}

}  // namespace

// Whether the tensor-core pass takes (X, n, k): X 16-byte aligned, n <= 64,
// 1 <= k <= 256, m < 2^31, and the shape fits the shared memory.
bool tcx_eligible(const float* X, long long m, int n, int np, int k) {
    TxShape s;
    return (((uintptr_t)X) & 15) == 0 && m >= 1 && m < (1ll << 31) && (n % 4 != 0 || encode_fn() != nullptr) &&
           (np <= 8 ? tx_shape<8>(k, s) : np == 16 ? tx_shape<16>(k, s) : np == 32 ? tx_shape<32>(k, s)
                                                                                  : tx_shape<64>(k, s));
}

void set_tcx_wait_limit(unsigned polls, unsigned ns) {
    g_wait_polls.store(polls ? polls : tc::kDefaultWait.polls);
    g_wait_ns.store(polls ? ns : tc::kDefaultWait.ns);
}
// The limit the tensor-core passes (exact and precision form) launch with.
tc::WaitLimit tcx_wait_limit() { return {g_wait_polls.load(), g_wait_ns.load()}; }

// Launch the tensor-core exact pass; cudaErrorNotSupported when not eligible.
cudaError_t launch_tcx_fullpass(int np, const float* X, long long m, int n, const float* C, int k,
                                const double* sel_f, int W, int* labels, Globals* g, float gB, float gp2,
                                int incumbent, int sms, cudaStream_t st) {
    if (!tcx_eligible(X, m, n, np, k)) return cudaErrorNotSupported;
    switch (np) {
        case 4:
        case 8: return launch_np<8>(X, m, n, C, np, k, sel_f, W, labels, g, gB, gp2, incumbent, sms, st);
        case 16: return launch_np<16>(X, m, n, C, np, k, sel_f, W, labels, g, gB, gp2, incumbent, sms, st);
        case 32: return launch_np<32>(X, m, n, C, np, k, sel_f, W, labels, g, gB, gp2, incumbent, sms, st);
        case 64: return launch_np<64>(X, m, n, C, np, k, sel_f, W, labels, g, gB, gp2, incumbent, sms, st);
    }
    return cudaErrorNotSupported;
}

}  // namespace bm
