// Sampling and gather (a1, a2) for all workers of a round in one launch.
//
// Algorithm 1 draws, for every worker and round, one sample to recompute
// f_hat_w and one sample per pass (Sec. 4.1: "a new uniformly random sample
// ... in each iteration").  None of them depends on clustering results, so
// they are all drawn up front, a job per (worker, sample), and gathered
// into contiguous padded rows that the worker kernel then reuses.
//
// A sample of size s is the first s distinct values among the bounded draws
// r_0, r_1, ... of its Philox stream, in order of first occurrence.  Larger
// samples are drawn by many CTAs each (sample_wide_*).  Else, when a bitmap of the m values fits in shared memory, a job marks the values it has
// taken in that bitmap (sample_by_bitmap); otherwise it inserts its draws into
// an open-addressing table in global memory whose slots hold
// (generation << 32 | t): the generation of the job marks a slot as used, so
// the table is cleared only when its slots change between this form and that
// of sample_wide_* (or the latter's generations run out), and the value of a
// slot is draws[t].  A draw t is kept when the slot of its value holds t itself (the least t).
#include <algorithm>
#include <cstdint>

#include "bm_device.cuh"
#include "bm_sample.cuh"

namespace bm {

__device__ __forceinline__ unsigned int tab_hash(unsigned int r) { return r * 0x9E3779B1u; }

// Insert draw (r, t); the slot keeps the least t of value r.  Returns false
// only if the bounded retry or probe limits ran out (reported as an error).
__device__ bool tab_insert(unsigned long long* tab, unsigned int mask, unsigned int gen, unsigned int r,
                           unsigned int t, const unsigned int* draws) {
    unsigned int h = tab_hash(r) & mask;
    const unsigned long long mine = ((unsigned long long)gen << 32) | t;
    for (unsigned int probe = 0; probe <= mask; ++probe) {
        unsigned long long cur = atomicAdd(&tab[h], 0ull);
        bool next = false;
        for (int spin = 0; spin < 1024 && !next; ++spin) {   // each retry sees a newer slot value
            if ((unsigned int)(cur >> 32) != gen) {          // free in this generation
                const unsigned long long prev = atomicCAS(&tab[h], cur, mine);
                if (prev == cur) return true;
                cur = prev;
                continue;
            }
            const unsigned int tt = (unsigned int)cur;
            if (draws[tt] != r) { next = true; break; }      // another value: next slot
            if (tt <= t) return true;                        // an earlier draw holds it
            const unsigned long long prev = atomicCAS(&tab[h], cur, mine);
            if (prev == cur) return true;
            cur = prev;
        }
        if (!next) return false;
        h = (h + 1u) & mask;
    }
    return false;
}

__device__ bool tab_is_first(const unsigned long long* tab, unsigned int mask, unsigned int gen,
                             unsigned int r, unsigned int t, const unsigned int* draws) {
    unsigned int h = tab_hash(r) & mask;
    for (unsigned int probe = 0; probe <= mask; ++probe) {
        const unsigned long long cur = tab[h];
        if ((unsigned int)(cur >> 32) != gen) return false;
        const unsigned int tt = (unsigned int)cur;
        if (draws[tt] == r) return tt == t;
        h = (h + 1u) & mask;
    }
    return false;
}

__device__ __forceinline__ long long pow2_at_least(long long v) {
    long long p = 1;
    while (p < v) p <<= 1;
    return p;
}

// The same sample with a shared-memory bitmap of the m values (used when it
// fits): the draws are taken in chunks of kSampleDraws x kSampleThreads in
// counter order, kSampleDraws consecutive draws per thread.  A draw
// t of value r is the first occurrence of r when r's bit is clear at the
// start of t's chunk and t is the least draw of r inside the chunk (a small
// shared hash table keyed by r keeps that least t).  The chunk's first
// occurrences extend the sample in t order and then set their bits.  Returns
// the number of values found (s, or fewer when `cap` draws were not enough).
__device__ long long sample_by_bitmap(const SampleArgs& a, long long s, unsigned long long k1, long long cap,
                                      long long* idx, long long* red64) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* mini = reinterpret_cast<unsigned long long*>(smem_raw);   // kMiniSlots
    unsigned int* bits = reinterpret_cast<unsigned int*>(mini + kMiniSlots);      // bitmap_words
    const long long m = a.m;
    for (int i = threadIdx.x; i < a.bitmap_words; i += kSampleThreads) bits[i] = 0u;
    for (int i = threadIdx.x; i < kMiniSlots; i += kSampleThreads) mini[i] = ~0ull;
    __syncthreads();
    const unsigned long long thr = lemire_thr((unsigned long long)m);
    long long got = 0;
    constexpr int D = kSampleDraws;
    for (long long t0 = 0; t0 < cap && got < s; t0 += (long long)D * kSampleThreads) {     // block-uniform
        unsigned int r[D], h[D];
        bool cand[D];
        unsigned long long key[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {             // this thread's D consecutive draws
            const long long t = t0 + (long long)D * threadIdx.x + d;
            r[d] = 0; h[d] = 0; cand[d] = false;
            if (t < cap) {
                const P4 blk = philox4x64_10((unsigned long long)t, 0, 0, 0, a.seed, k1);
                r[d] = (unsigned int)uniform_below(blk, (unsigned long long)m, thr);
                cand[d] = ((bits[r[d] >> 5] >> (r[d] & 31)) & 1u) == 0u;
            }
            key[d] = ((unsigned long long)r[d] << 32) | (unsigned int)t;
            // at most D kSampleThreads keys in 2 D kSampleThreads slots: a
            // free slot always exists
            if (cand[d]) {
                h[d] = tab_hash(r[d]) & (kMiniSlots - 1);
                for (int p = 0; p < kMiniSlots; ++p) {
                    unsigned long long cur = mini[h[d]];
                    if (cur == ~0ull) {
                        cur = atomicCAS(&mini[h[d]], ~0ull, key[d]);
                        if (cur == ~0ull) break;
                    }
                    if ((unsigned int)(cur >> 32) == r[d]) { atomicMin(&mini[h[d]], key[d]); break; }
                    h[d] = (h[d] + 1u) & (kMiniSlots - 1);
                }
            }
        }
        __syncthreads();
        bool first[D];
        int cnt = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            first[d] = cand[d] && mini[h[d]] == key[d];
            cnt += first[d];
        }
        __syncthreads();
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if (cand[d]) mini[h[d]] = ~0ull;             // empty again for the next chunk
            if (first[d]) atomicOr(&bits[r[d] >> 5], 1u << (r[d] & 31));
        }
        long long total;
        long long pos = got + block_exscan((long long)cnt, red64, &total);
#pragma unroll
        for (int d = 0; d < D; ++d)
            if (first[d]) {
                if (pos < s) idx[pos] = (long long)r[d];
                ++pos;
            }
        got += total;
    }
    __syncthreads();
    return got < s ? got : s;
}

// The stream and the sample size of a job.
struct JobStream { int purpose, worker, rnd, pss; long long s; };
__device__ JobStream job_stream(const SampleArgs& a, int job) {
    JobStream js{a.purpose, a.worker, a.rnd, a.pss, a.step_s};
    if (a.mode == kSampleRound) {
        const int slots = a.P + 1;
        js.worker = a.worker_base + job / slots;
        const int q = job % slots;
        js.purpose = (q < a.P) ? kPurposePass : kPurposeEval;
        js.pss = (q < a.P) ? q : 0;
        js.s = policy_size(a.sp, a.seed, stream_k1(kPurposeSize, js.worker, a.rnd, 0));
    } else if (a.mode == kSampleFinal) {
        long long s_lo = a.s_min, s_hi = a.s_max;
        if (a.set_len > 0) {
            s_lo = a.set[0]; s_hi = a.set[0];
            for (int i = 1; i < a.set_len; ++i) { s_lo = min(s_lo, a.set[i]); s_hi = max(s_hi, a.set[i]); }
        }
        const long long acc = (long long)a.glob->accepts, Ls = (long long)a.glob->L_sum;
        js.s = s_hi;
        if (acc > 0) js.s = min(max((2 * Ls + acc) / (2 * acc), s_lo), s_hi);
        if (a.step_s > 0) js.s = a.step_s;        // s_opt given by the host (a fit sharded over ranks)
        js.purpose = kPurposeFinal; js.worker = 0; js.rnd = 0; js.pss = 0;
    }
    return js;
}

// ------------------------------------------------- many CTAs per job
// Larger samples of at most half the rows.  One CTA per job draws its sample
// in a serial chain of chunks (two dependent round trips to memory per chunk,
// or block barriers), which left most of the GPU idle: drawing and gathering
// one sample of 64,000 of 4 10^6 rows took 0.84 ms.  Here a job's draws are
// taken all at once by many CTAs, in three launches for all jobs:
//   sample_wide_draw   draw t of value r claims the slot of r in the job's
//                      table (open addressing; the slot keeps the least t of
//                      r) and notes the slot;
//   sample_wide_count  draw t is a first occurrence when its slot holds t;
//                      one bit per draw and a count per chunk of 1024 draws;
//   sample_wide_emit   the first s of them, in draw order, become the sample:
//                      a CTA adds up the counts of the chunks before its own,
//                      writes its indices and gathers its rows.
// The number of draws T(s) covers s distinct values but for a probability
// below 10^-14 (mean + 8 standard deviations + 5% + 1024 draws, p >= 1/2 of a
// new value each); falling short is reported.  Bound by the table's random
// 32-byte sectors (8 bytes used of each) and the gathered rows: sampling and
// gathering 64,000 of 4 10^6 x 32 0.84 -> 0.06 ms, the 704 samples of a round
// of 64 workers (2,000 to 131,072 rows) 9.4 -> 4.2 ms.
__device__ long long wide_draws(const SampleArgs& a, long long s) {
    const float f = (float)s / (float)a.m;
    const float mean = -(float)a.m * log1pf(-f);
    const float sd = sqrtf((float)s * f) / (1.f - f);
    return min(a.Tcap, (long long)(mean * 1.05f + 8.f * sd) + 1024);
}
struct WideJob { unsigned long long k1; long long s, T; unsigned mask; };
__device__ __forceinline__ WideJob wide_job(const SampleArgs& a, int job) {
    __shared__ WideJob wj;
    if (threadIdx.x == 0) {
        const JobStream js = job_stream(a, job);
        wj.k1 = stream_k1(js.purpose, js.worker, js.rnd, js.pss);
        wj.s = js.s;
        wj.T = js.s > 0 ? wide_draws(a, js.s) : 0;
        wj.mask = (unsigned)(min(a.H, pow2_at_least(2 * wj.T)) - 1);
    }
    __syncthreads();
    return wj;
}

constexpr int kWideThreads = 256;
constexpr int kWidePer = kWideDraws / kWideThreads;
__global__ void __launch_bounds__(kWideThreads) sample_wide_draw(const SampleArgs a) {
    const int job = blockIdx.y;
    const WideJob wj = wide_job(a, job);
    const long long t0 = (long long)blockIdx.x * kWideDraws + threadIdx.x;
    if (t0 >= wj.T) return;
    unsigned long long* tab = a.table + (long long)job * a.table_stride;
    unsigned int* slot = a.draws + (long long)job * a.draws_stride;
    const unsigned long long thr = lemire_thr((unsigned long long)a.m);
    unsigned long long mine[kWidePer], cur[kWidePer];
    unsigned h[kWidePer];
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) {                     // all draws, then all first looks at the table
        const long long t = t0 + u * kWideThreads;
        const P4 blk = philox4x64_10((unsigned long long)t, 0, 0, 0, a.seed, wj.k1);
        const unsigned r = (unsigned)uniform_below(blk, (unsigned long long)a.m, thr);
        mine[u] = ((unsigned long long)a.wgen << 51) | ((unsigned long long)r << kWideTBits) | (unsigned long long)t;
        h[u] = tab_hash(r) >> 7 & wj.mask;                   // (the multiplicative hash mixes upwards)
        cur[u] = t < wj.T ? *(const volatile unsigned long long*)(tab + h[u]) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) {
        const long long t = t0 + u * kWideThreads;
        if (t >= wj.T) break;
        bool done = false;
        // at most T <= half the slots are taken: a free one exists; a slot
        // changes hands at most once per draw, so the retries end too
        for (long long step = 0; step <= 2ll * wj.mask + 2 && !done; ++step) {
            if (cur[u] >> 51 != a.wgen) {                    // free in this generation
                const unsigned long long prev = atomicCAS(&tab[h[u]], cur[u], mine[u]);
                done = prev == cur[u];
                cur[u] = prev;
            } else if (cur[u] >> kWideTBits == mine[u] >> kWideTBits) {
                if (mine[u] < cur[u]) atomicMin(&tab[h[u]], mine[u]);    // same value: keep the least t
                done = true;
            } else {
                h[u] = (h[u] + 1u) & wj.mask;
                cur[u] = *(const volatile unsigned long long*)(tab + h[u]);
            }
        }
        if (!done) atomicOr(&a.glob->err, kErrSample);
        slot[t] = h[u];
    }
}

// Draw index of step u of this thread: warps take 128 consecutive draws.
__device__ __forceinline__ long long wide_t(int u) {
    return (long long)blockIdx.x * kWideDraws + (threadIdx.x >> 5) * (32 * kWidePer) + u * 32 + (threadIdx.x & 31);
}
__global__ void __launch_bounds__(kWideThreads) sample_wide_count(const SampleArgs a) {
    __shared__ int tot;
    const int job = blockIdx.y, lane = threadIdx.x & 31;
    const WideJob wj = wide_job(a, job);
    if ((long long)blockIdx.x * kWideDraws >= wj.T) return;
    int* cnt = a.wcnt + (long long)job * a.chunks * (1 + kWideDraws / 32);
    if (threadIdx.x == 0) tot = 0;
    __syncthreads();
    const unsigned long long* tab = a.table + (long long)job * a.table_stride;
    unsigned int* draws = a.draws + (long long)job * a.draws_stride;
    unsigned int* flags = reinterpret_cast<unsigned int*>(cnt + a.chunks) + blockIdx.x * (kWideDraws / 32);
    unsigned hs[kWidePer];
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) hs[u] = wide_t(u) < wj.T ? draws[wide_t(u)] : 0u;
    unsigned long long e[kWidePer];
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) e[u] = wide_t(u) < wj.T ? tab[hs[u] & wj.mask] : ~0ull;
    int mine = 0;
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) {
        const long long t = wide_t(u);
        const bool first = t < wj.T && (long long)(e[u] & ((1u << kWideTBits) - 1u)) == t;
        const unsigned b = __ballot_sync(0xffffffffu, first);
        if (t < wj.T) draws[t] = (unsigned)(e[u] >> kWideTBits) & 0x7fffffffu;
        if (lane == 0) flags[(threadIdx.x >> 5) * kWidePer + u] = b;
        mine += __popc(b);
    }
    if (lane == 0) atomicAdd(&tot, mine);
    __syncthreads();
    if (threadIdx.x == 0) cnt[blockIdx.x] = tot;
}

template <int NP>
__global__ void __launch_bounds__(kWideThreads) sample_wide_emit(const SampleArgs a) {
    __shared__ long long red[kWideThreads / 32 + 1];
    __shared__ unsigned rows[kWideDraws];
    const int job = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const WideJob wj = wide_job(a, job);
    const int used = (int)((wj.T + kWideDraws - 1) / kWideDraws);
    if ((int)blockIdx.x >= used && blockIdx.x > 0) return;
    const int* cnt = a.wcnt + (long long)job * a.chunks * (1 + kWideDraws / 32);
    // firsts before this chunk, and (chunk 0) in all
    long long before = 0, all = 0;
    for (int c = threadIdx.x; c < used; c += kWideThreads) {
        const int v = cnt[c];
        all += v;
        if (c < (int)blockIdx.x) before += v;
    }
    const long long p0 = block_sum<long long>(before, red);
    const long long tot = block_sum<long long>(all, red);
    __shared__ long long sh[2];
    if (threadIdx.x == 0) { sh[0] = p0; sh[1] = tot; }
    __syncthreads();
    const bool short_of = sh[1] < wj.s;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (short_of) atomicOr(&a.glob->err, kErrSample);
        if (a.job_s) a.job_s[job] = short_of ? 0 : (int)wj.s;
        if (a.mode == kSampleFinal) a.glob->s_opt = (int)wj.s;
    }
    if (short_of || sh[0] >= wj.s) return;
    const unsigned int* flags = reinterpret_cast<const unsigned int*>(cnt + a.chunks) + blockIdx.x * (kWideDraws / 32);
    const unsigned int* draws = a.draws + (long long)job * a.draws_stride;
    long long* idx = a.idx + (long long)job * a.idx_stride;
    const int have = (int)min((long long)cnt[blockIdx.x], wj.s - sh[0]);    // indices this chunk contributes
    // rank of each first in the chunk: flag words before its own
    int base = 0;
    {
        const unsigned f = flags[lane];                      // 32 words: one per lane
        int x = __popc(f);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        base = x - __popc(f);
    }
    static_assert(kWideDraws == 32 * 32, "a flag word per lane");
#pragma unroll
    for (int u = 0; u < kWidePer; ++u) {
        const int word = wid * kWidePer + u;
        const unsigned f = flags[word];
        const int at = __shfl_sync(0xffffffffu, base, word) + __popc(f & ((1u << lane) - 1u));
        if ((f >> lane & 1u) && at < have) {
            const unsigned r = draws[wide_t(u)];
            idx[sh[0] + at] = (long long)r;
            rows[at] = r;
        }
    }
    if (a.mode == kSampleStep) return;
    __syncthreads();
    float* S = a.S + (long long)job * a.S_stride;
    const int n = a.n;
    const bool vec = (n % 4) == 0 && (reinterpret_cast<uintptr_t>(a.X) & 15) == 0;
    constexpr int Q = NP / 4, RS = kWideThreads / Q, U = 4;  // pieces per row, rows per pass, passes in flight
    const int q = threadIdx.x % Q;
    for (int i0 = threadIdx.x / Q; i0 < have; i0 += U * RS) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int i = i0 + u * RS;
            if (i >= have) continue;
            const float* xr = a.X + (long long)rows[i] * n;
            if (vec) {
                if (4 * q < n) v[u] = __ldg(reinterpret_cast<const float4*>(xr) + q);
            } else {
                v[u].x = (4 * q + 0 < n) ? xr[4 * q + 0] : 0.f;
                v[u].y = (4 * q + 1 < n) ? xr[4 * q + 1] : 0.f;
                v[u].z = (4 * q + 2 < n) ? xr[4 * q + 2] : 0.f;
                v[u].w = (4 * q + 3 < n) ? xr[4 * q + 3] : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * RS < have) *reinterpret_cast<float4*>(S + tile_at<NP>(sh[0] + i0 + u * RS, 4 * q)) = v[u];
    }
}

// Rows of X by index, a thread per element (16-byte elements where rows are
// aligned): bound by the random rows.
template <typename V>
__global__ void __launch_bounds__(256) gather_kernel(const V* __restrict__ X, long long m, int per,
                                                     const long long* __restrict__ idx, long long s,
                                                     V* __restrict__ out, Globals* g) {
    for (long long e = (long long)blockIdx.x * 256 + threadIdx.x; e < s * per; e += (long long)gridDim.x * 256) {
        const long long i = e / per;
        const long long row = idx[i];
        if (row >= 0 && row < m) out[e] = X[row * per + (e - i * per)];
        else atomicOr(&g->err, kErrArgs);
    }
}
cudaError_t launch_gather(const float* X, long long m, int n, const long long* idx, long long s, float* out,
                          Globals* g, cudaStream_t st) {
    const bool vec = n % 4 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int per = vec ? n / 4 : n;
    const int grid = (int)std::min<long long>(8192, (s * per + 255) / 256);
    if (vec)
        gather_kernel<float4><<<grid, 256, 0, st>>>(reinterpret_cast<const float4*>(X), m, per, idx, s,
                                                    reinterpret_cast<float4*>(out), g);
    else
        gather_kernel<float><<<grid, 256, 0, st>>>(X, m, per, idx, s, out, g);
    return cudaGetLastError();
}

template <int NP>
__global__ void __launch_bounds__(kSampleThreads, 1) sample_kernel(const SampleArgs a) {
    __shared__ long long red64[kSampleThreads / 32 + 1];
    __shared__ int fail;
    const int job = blockIdx.x;
    const JobStream js = job_stream(a, job);
    const int purpose = js.purpose, worker = js.worker, rnd = js.rnd, pss = js.pss;
    long long s = js.s;
    if (a.mode == kSampleFinal && threadIdx.x == 0) a.glob->s_opt = (int)s;
    long long* idx = a.idx + (long long)job * a.idx_stride;
    float* S = a.S + (long long)job * a.S_stride;
    if (a.bitmap_words > 0) {
        const unsigned long long k1 = stream_k1(purpose, worker, rnd, pss);
        const long long got = s > 0 ? sample_by_bitmap(a, s, k1, a.Tcap, idx, red64) : 0;
        if (got < s) {
            if (threadIdx.x == 0) atomicOr(&a.glob->err, kErrSample);
            s = 0;
        }
        __threadfence_block();
        __syncthreads();
    } else {
        const long long m = a.m;
        unsigned int* draws = a.draws + (long long)job * a.draws_stride;
        unsigned long long* tab = a.table + (long long)job * a.table_stride;
        // table size for this job: small samples need only about 2 s draws
        const long long H = (2 * s <= m) ? min(a.H, pow2_at_least(4 * s + 2048)) : a.H;
        const unsigned int mask = (unsigned int)(H - 1);
        const long long cap = min(a.Tcap, H / 2);
        const unsigned int gen = a.gen_base + (unsigned int)job;
        const unsigned long long k1 = stream_k1(purpose, worker, rnd, pss);
        const unsigned long long thr = lemire_thr((unsigned long long)m);
        long long T_done = 0, T = min(cap, s + (s * s) / m + 64);
        if (threadIdx.x == 0) fail = 1;
        __syncthreads();
        for (int batch = 0; batch < 64 && s > 0; ++batch) {
            for (long long t = T_done + threadIdx.x; t < T; t += kSampleThreads) {
                const P4 blk = philox4x64_10((unsigned long long)t, 0, 0, 0, a.seed, k1);
                draws[t] = (unsigned int)uniform_below(blk, (unsigned long long)m, thr);
            }
            __threadfence_block();
            __syncthreads();
            bool ok = true;
            for (long long t = T_done + threadIdx.x; t < T; t += kSampleThreads)
                ok &= tab_insert(tab, mask, gen, draws[t], (unsigned int)t, draws);
            if (!ok) atomicOr(&a.glob->err, kErrSample);
            __threadfence_block();
            __syncthreads();
            const long long ch = (T + kSampleThreads - 1) / kSampleThreads;
            const long long c0 = ch * threadIdx.x, c1 = min(T, c0 + ch);
            long long mine = 0;
            for (long long t = c0; t < c1; ++t) mine += tab_is_first(tab, mask, gen, draws[t], (unsigned int)t, draws);
            long long total;
            const long long excl = block_exscan(mine, red64, &total);
            if (total >= s) {
                long long pos = excl;
                for (long long t = c0; t < c1 && pos < s; ++t) {
                    const unsigned int r = draws[t];
                    if (tab_is_first(tab, mask, gen, r, (unsigned int)t, draws)) idx[pos++] = (long long)r;
                }
                if (threadIdx.x == 0) fail = 0;
                break;
            }
            if (T >= cap) break;
            T_done = T;
            T = min(cap, 2 * T);
        }
        __syncthreads();
        if (s > 0 && fail) {
            if (threadIdx.x == 0) atomicOr(&a.glob->err, kErrSample);
            s = 0;
        }
        __threadfence_block();
        __syncthreads();
    }
    if (a.mode == kSampleStep) {
        if (threadIdx.x == 0 && a.job_s) a.job_s[job] = (int)s;
        return;
    }
    // gather (padded rows in tiles, zeros in the padding); 16-byte loads when the rows
    // of X are 16-byte aligned.  A thread takes kGatherBatch items (16-byte
    // pieces of padded rows) at a time: their row indices, then their loads,
    // are all in flight together, so that a large sample does not pay two
    // dependent memory latencies per item.
    const int n = a.n;
    const bool vec = (n % 4) == 0 && (reinterpret_cast<uintptr_t>(a.X) & 15) == 0;
    constexpr int U = kGatherBatch;
    constexpr int RS = kSampleThreads / (NP / 4);          // rows a pass of the CTA covers
    static_assert(kSampleThreads % (NP / 4) == 0, "a thread keeps its piece q of every row");
    const int q = threadIdx.x % (NP / 4);                  // this thread's 16-byte piece of a row
    for (long long i0 = threadIdx.x / (NP / 4); i0 < s; i0 += (long long)U * RS) {
        long long row[U];
#pragma unroll
        for (int u = 0; u < U; ++u) row[u] = (i0 + u * RS < s) ? idx[i0 + u * RS] : 0;
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i0 + u * RS >= s) continue;
            if (row[u] >= 0 && row[u] < a.m) {
                const float* xr = a.X + row[u] * (long long)n;
                if (vec) {
                    if (4 * q < n) v[u] = __ldg(reinterpret_cast<const float4*>(xr) + q);
                } else {
                    v[u].x = (4 * q + 0 < n) ? xr[4 * q + 0] : 0.f;
                    v[u].y = (4 * q + 1 < n) ? xr[4 * q + 1] : 0.f;
                    v[u].z = (4 * q + 2 < n) ? xr[4 * q + 2] : 0.f;
                    v[u].w = (4 * q + 3 < n) ? xr[4 * q + 3] : 0.f;
                }
            } else if (q == 0) {
                atomicOr(&a.glob->err, kErrArgs);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * RS < s) *reinterpret_cast<float4*>(S + tile_at<NP>(i0 + u * RS, 4 * q)) = v[u];
    }
    if (threadIdx.x == 0 && a.job_s) a.job_s[job] = (int)s;
}

template <int NP>
static cudaError_t launch_sample_t(const SampleArgs& a, int jobs, cudaStream_t st) {
    if (a.wide) {
        const dim3 grid((unsigned)a.chunks, (unsigned)jobs);
        sample_wide_draw<<<grid, kWideThreads, 0, st>>>(a);
        sample_wide_count<<<grid, kWideThreads, 0, st>>>(a);
        sample_wide_emit<NP><<<grid, kWideThreads, 0, st>>>(a);
        return cudaGetLastError();
    }
    const size_t smem = sample_smem_bytes(a.bitmap_words);
    // every launch goes through allow_max_smem (which raises the limit once,
    // under a lock): a launch from one host thread must not race with the
    // attribute being set from another
    const cudaError_t e = allow_max_smem((const void*)sample_kernel<NP>);
    if (e != cudaSuccess) return e;
    sample_kernel<NP><<<jobs, kSampleThreads, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_sample(int np, const SampleArgs& a, int jobs, cudaStream_t st) {
    switch (np) {
        case 4: return launch_sample_t<4>(a, jobs, st);
        case 8: return launch_sample_t<8>(a, jobs, st);
        case 16: return launch_sample_t<16>(a, jobs, st);
        case 32: return launch_sample_t<32>(a, jobs, st);
        case 64: return launch_sample_t<64>(a, jobs, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace bm
