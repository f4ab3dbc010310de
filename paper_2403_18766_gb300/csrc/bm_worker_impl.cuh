#pragma once
// Fused Big-means worker kernel (template body; instantiated per padded
// width NP in bm_worker_np*.cu): one thread-block cluster, or a group of
// clusters, per competing worker of Algorithm 1 (arXiv 2403.18766, Sec. 4.2-4.3).
//
// The samples of a round are drawn and gathered beforehand by the sampling
// kernel.  A worker's sample is split into contiguous row slices, one per CTA
// of its clusters.  Per pass they re-seed degenerate centroids with greedy
// K-means++ (a3), run Lloyd's iterations (a4-a6) and apply the incumbent rule.
// Exchange within a cluster goes through distributed shared memory and hardware
// cluster barriers (barrier.cluster); exchange within a group, and that of
// K-means++, through global memory, in a group with a counter that a CTA polls
// a bounded number of times (gsync).  All control flow that reaches a barrier
// is uniform over the CTAs that meet there: it only depends on kernel arguments
// and on values every CTA reads after a barrier from the same place, so all of
// them execute the same sequence of barriers.
#include <cstdint>
#include <map>
#include <mutex>
#include <utility>

#include "bm_device.cuh"
#include "bm_worker.cuh"

namespace bm {

template <int NP>
struct Sm {
    float* Ccur;          // k * NP  centroids of the current step
    float* Cnext;         // k * NP  next centroids, pushed by their owners
    float* CC;            // k       fl(||c||^2) FMA chain
    long long* OACC;      // owned slots * NP * kAccWords: exact coordinate sums of owned clusters
    int* ocnt;            // owned slots: member counts of owned clusters
    int* lcnt;            // k: this CTA's member counts, then bucket cursors
    int* lstart;          // k + 1: bucket starts of this CTA's rows sorted by label
    unsigned char* deg;   // k       worker's degenerate flags (identical copies)
    unsigned char* emptyall;  // k   empties of the last assignment, pushed by the owners
    Xch* x;
    ObjPart* inbox;       // kMaxCluster: objective partials of every CTA (used on rank 0)
    Decision* dec;        // rank 0's decision of the current step
    unsigned __int128* red128;    // one per warp (kMaxWarps)
    long long* red64;             // one per warp, + 1
    unsigned int* redu;           // one per warp
    CertC* cert;
    long long* bcast;             // values for the CTA: 2 K-means++ best, 3 its largest D^2, 8 deadline flag
    unsigned short* labs;         // rows_cta: label of each row of the CTA (first assignment)
    unsigned short* rowlist;      // rows_cta: the CTA's row offsets sorted by label
};

template <int NP>
__device__ inline Sm<NP> carve(int k, int cs, int rows_cta) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* p = smem_raw;
    Sm<NP> s;
    s.Ccur = (float*)p;            p += align16((size_t)k * NP * 4);
    s.Cnext = (float*)p;           p += align16((size_t)k * NP * 4);
    s.CC = (float*)p;              p += align16((size_t)k * 4);
    s.OACC = (long long*)p;        p += align16((size_t)owned_slots(k, cs) * NP * kAccWords * 8);
    s.ocnt = (int*)p;              p += align16((size_t)k * 4);
    s.lcnt = (int*)p;              p += align16((size_t)k * 4);
    s.lstart = (int*)p;            p += align16((size_t)(k + 1) * 4);
    s.deg = p;                     p += align16((size_t)k);
    s.emptyall = p;                p += align16((size_t)k);
    s.x = (Xch*)p;                 p += align16(sizeof(Xch));
    s.inbox = (ObjPart*)p;         p += align16(sizeof(ObjPart) * kMaxCluster);
    s.dec = (Decision*)p;          p += align16(sizeof(Decision));
    s.red128 = (unsigned __int128*)p; p += align16(sizeof(unsigned __int128) * kMaxWarps);
    s.red64 = (long long*)p;       p += align16(8 * (kMaxWarps + 1));
    s.redu = (unsigned int*)p;     p += align16(4 * kMaxWarps);
    s.cert = (CertC*)p;            p += align16(sizeof(CertC));
    s.bcast = (long long*)p;       p += align16(8 * 16);
    s.labs = (unsigned short*)p;
    s.rowlist = s.labs + rows_cta;
    return s;
}

template <int NP>
struct RowsPerThread { static constexpr int v = (64 / NP) > 8 ? 8 : ((64 / NP) < 1 ? 1 : 64 / NP); };

// ---------------------------------------------------------------- the CTA
// TPB: threads per CTA (256, or 512 for the largest clusters).
template <int NP, int TPB>
struct Worker {
    const WorkerArgs& a;
    cg::cluster_group cl;
    Sm<NP> sm;
    int rank, cs, w, k, n;
    int gi, G, ctaW, nW;    // cluster gi of the worker's G clusters; CTA ctaW of its nW
    int xpar = 0;           // parity of the next group exchange
    int xrot = 0;           // buffer of the next exchange of sums (0..2)
    int kpar = 0;           // parity of the next K-means++ exchange
    unsigned gepoch = 0;    // group barriers passed
    Grids g;
    float* S;               // current sample (padded rows), set per pass
    float* D2; float* Cw_mine;
    int* lab_prev;          // label of each sample row in the previous assignment

    __device__ Worker(const WorkerArgs& args, cg::cluster_group c) : a(args), cl(c) {
        cs = a.cs;
        rank = (int)cl.block_rank();
        const int ci = blockIdx.x / cs;
        if (a.ncl > 0) {
            const unsigned e = a.cmap[ci];
            w = (int)(e & 0xfffu);
            gi = (int)((e >> 16) & 0xffu);
            G = (int)(e >> 24);
        } else {
            w = a.worker_base + ci;
            gi = 0;
            G = 1;
        }
        ctaW = gi * cs + rank;
        nW = G * cs;
        k = a.k;
        n = a.n;
        sm = carve<NP>(k, cs, a.rows_cta);
        g = grids_from_maxbits(a.glob->maxbits);
        S = a.S;
        D2 = a.D2 + (long long)w * 4 * a.D2_stride;
        lab_prev = a.lab + (long long)w * a.D2_stride;
        Cw_mine = a.Cw_cta + ((long long)w * kMaxCluster + rank) * (long long)k * NP;
    }

    __device__ Xch* rx(int q) { return cl.map_shared_rank(sm.x, q); }

    // Phase trace: rank 0, thread 0 adds elapsed SM cycles to glob->trace[i].
    __device__ bool tracer() const { return gi == 0 && rank == 0 && threadIdx.x == 0; }
    __device__ void trace_add(int i, long long t0) const {
        if (tracer()) atomicAdd(&a.glob->trace[i], (unsigned long long)(clock64() - t0));
    }

    // Sample of job (worker, slot) drawn by the sampling kernel; returns its size.
    __device__ long long use_sample(int slot) {
        const long long job = (long long)w * (a.P + 1) + slot;
        S = a.S + job * a.S_stride;
        return a.job_s[job];
    }

    // Elements D0 .. D0 + DN - 1 of sample row i (D0 a multiple of 8 unless NP = 4).
    template <int D0, int DN>
    __device__ __forceinline__ void load_chunks(long long i, float4 (&v)[DN / 4]) const {
        if constexpr (NP == 4) {
            v[0] = __ldg(reinterpret_cast<const float4*>(S + i * NP));
        } else {
            const float* p = S + tile_at<NP>(i, D0);
#pragma unroll
            for (int c = 0; c < DN / 8; ++c) ld8(p + c * (NP <= 8 ? 8 : 32), v[2 * c], v[2 * c + 1]);
        }
    }

    // Rows of this CTA: its share of the worker's G * cs CTAs.
    __device__ void slice(long long s, long long& lo, long long& hi) const {
        lo = s * ctaW / nW;
        hi = s * (ctaW + 1) / nW;
    }
    __device__ bool lead() const { return gi == 0 && rank == 0; }     // records the worker's counters

    // ------------------------------------------------ group of clusters
    // Barrier among every CTA of the worker's G clusters (G > 1): a counter
    // in global memory that each CTA increments once per barrier; a CTA waits
    // until it reaches (barriers passed) x (CTAs of the group).  The wait is
    // bounded: when it runs out, or when another CTA of the group gave up,
    // the group's abort flag is raised, every later wait of the group returns
    // at once and the launch reports a timeout (results are then discarded).
    __device__ void gsync() {
        if (G == 1) return;
        ++gepoch;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(a.xbar + w, 1u);
            gwait();
        }
        __syncthreads();
    }
    // One thread: wait until every CTA of the group has passed barrier
    // `gepoch` (polls back off only once the wait is long).
    __device__ void gwait() {
        const unsigned target = gepoch * (unsigned)nW;
        const volatile unsigned* bar = a.xbar + w;
        const volatile int* ab = a.xabort + w;
        for (unsigned polls = 0; *bar < target; ++polls) {
            if (*ab) break;
            if (polls >= (1u << 22)) {
                atomicExch(a.xabort + w, 1);
                atomicOr(&a.glob->err, kErrTimeout);
                break;
            }
            if (polls > 256) __nanosleep(64);
        }
        __threadfence();
    }
    __device__ bool group_aborted() const { return G > 1 && *(const volatile int*)(a.xabort + w) != 0; }
    // Objective slot of cluster q (parity par).
    __device__ size_t xslot(int par, int q) const { return ((size_t)w * 2 + par) * kMaxGroup + q; }
    // Sums of the group in buffer `rot`: words of (cluster j, dimension d), counts.
    __device__ long long* xwords(int rot, int j, int d) const {
        return a.xpart + ((((size_t)w * 3 + rot) * k + j) * NP + d) * kAccWords;
    }
    __device__ int* xcount(int rot, int j) const { return a.xcnt + ((size_t)w * 3 + rot) * k + j; }

    // cluster barrier that also orders global-memory writes
    __device__ void csync_global() {
        __threadfence();
        cl.sync();
    }

    // ------------------------------------------------------ centroid prep
    __device__ void load_centroids(const float* src) {
        for (int e = threadIdx.x; e < k * NP; e += TPB) sm.Ccur[e] = src[e];
        __syncthreads();
    }
    __device__ void store_centroids(float* dst) {
        for (int e = threadIdx.x; e < k * NP; e += TPB) dst[e] = sm.Ccur[e];
        __syncthreads();
    }
    // fl(||c_j||^2) as an FMA chain and the certificate's upper bounds.
    __device__ void prep_centroids() {
        unsigned int mx = 0;
        for (int j = threadIdx.x; j < k; j += TPB) {
            const float* c = sm.Ccur + (size_t)j * NP;
            float acc = 0.f, up = 0.f;
#pragma unroll
            for (int d = 0; d < NP; ++d) {
                acc = __fmaf_rn(c[d], c[d], acc);
                up = __fmaf_ru(c[d], c[d], up);
            }
            sm.CC[j] = acc;
            mx = max(mx, __float_as_uint(up));
        }
        const unsigned int m = block_max_u32(mx, sm.redu);
        if (threadIdx.x == 0) {
            sm.cert->cmax2 = __uint_as_float(m);
            sm.cert->cmax = __fsqrt_ru(__uint_as_float(m));
        }
        __syncthreads();
    }

    // ------------------------------------------- exact sums at the owners
    // Additions to another CTA's shared memory are fire-and-forget reductions
    // (red, relaxed, cluster scope) on its shared::cluster address; the
    // cluster barrier that follows orders them before the owner reads.
    __device__ static unsigned cluster_addr(const void* local, int q) {
        unsigned r;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(q));
        return r;
    }
    __device__ static void red_u64(unsigned addr, unsigned long long v) {
        asm volatile("red.relaxed.cluster.shared::cluster.add.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
    }
    __device__ static void red_s32(unsigned addr, int v) {
        asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
    }
    // Words of (cluster j, dimension d) in the owner CTA's shared memory.
    __device__ unsigned owner_words(int j, int d) {
        return cluster_addr(sm.OACC + ((size_t)(j / cs) * NP + d) * kAccWords, j % cs);
    }
    __device__ unsigned owner_count(int j) { return cluster_addr(sm.ocnt + j / cs, j % cs); }
    // Add a signed 128-bit value to three int64 words (w0 + w1 2^32 + w2 2^64).
    __device__ static void add_words(unsigned wd, __int128 v) {
        if (v == 0) return;
        const unsigned long long lo = (unsigned long long)v;
        const unsigned long long w0 = lo & 0xffffffffull, w1 = lo >> 32;
        const unsigned long long w2 = (unsigned long long)(long long)(v >> 64);
        if (w0) red_u64(wd, w0);
        if (w1) red_u64(wd + 8, w1);
        if (w2) red_u64(wd + 16, w2);
    }
    // Move one row (held as m2x = -2 x) from cluster `from` (-1: none) to
    // `to` at their owners, this lane alone.
    __device__ bool move_row_lane(const float2 (&m2x)[NP / 2], int from, int to, unsigned int& inex) {
        bool ok = true;
        red_s32(owner_count(to), 1);
        if (from >= 0) red_s32(owner_count(from), -1);
#pragma unroll
        for (int d = 0; d < NP; ++d) {
            if (d < n) {
                __int128 v;
                ok &= fixed_of(-0.5f * ((d & 1) ? m2x[d >> 1].y : m2x[d >> 1].x), g.gx, inex, v);
                add_words(owner_words(to, d), v);
                if (from >= 0) add_words(owner_words(from, d), -v);
            }
        }
        return ok;
    }

    // The CTA's rows of the first assignment of a Lloyd run, summed per
    // cluster without per-element atomics: the rows are bucketed by label
    // (counting sort of 16-bit row offsets in shared memory), each warp walks
    // an equal share of the sorted rows one cluster at a time, its lanes over
    // (row, dimension), in batches whose loads are issued one batch ahead,
    // keeps the exact sum in registers and adds it to the owner's words once
    // per cluster.  Bound by issue: about 60 instructions per step of 32
    // values when every value was split in two 64-bit halves and every row's
    // label compared.  A coordinate of at least 2^(gx + 71) (2^-24 of the
    // largest |x|) is a whole number of 2^(gx + 48) and needs one half; the
    // others take the second half for their batch.
    __device__ bool bucket_sums(long long lo, long long hi, unsigned int& inex) {
        const int nrows = (int)(hi - lo);
        __syncthreads();                                   // labs and lcnt complete
        // counts to the owners; exclusive scan of the counts (warp 0)
        for (int j = threadIdx.x; j < k; j += TPB)
            if (sm.lcnt[j]) red_s32(owner_count(j), sm.lcnt[j]);
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            int run = 0;
            for (int j0 = 0; j0 < k; j0 += 32) {
                const int j = j0 + lane;
                const int c = j < k ? sm.lcnt[j] : 0;
                int x = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (j < k) sm.lstart[j] = run + x - c;
                run += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) sm.lstart[k] = run;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < k; j += TPB) sm.lcnt[j] = sm.lstart[j];   // cursors
        __syncthreads();
        for (int i = threadIdx.x; i < nrows; i += TPB)
            sm.rowlist[atomicAdd(&sm.lcnt[sm.labs[i]], 1)] = (unsigned short)i;
        __syncthreads();
        constexpr int LPR = NP < 32 ? NP : 32;             // lanes per row
        constexpr int RPS = 32 / LPR;                      // rows per warp step
        constexpr int DPL = NP / LPR;                      // dimensions per lane (2 for NP = 64)
        constexpr int U = 4;                               // steps per batch
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        const int sub = lane / LPR, d0 = lane % LPR;
        const int b0 = (int)((long long)nrows * wid / (TPB / 32));
        const int b1 = (int)((long long)nrows * (wid + 1) / (TPB / 32));
        int dof[DPL];                                      // offsets of this lane's dimensions in a tile
#pragma unroll
        for (int t = 0; t < DPL; ++t) dof[t] = (int)tile_at<NP>(0, d0 + t * LPR);
        // x 2^-(gx + 48), below 2^48, as two exact power-of-two factors
        const int eg = -(g.gx + 48);
        const int e1 = min(max(eg, -126), 127);
        const float s1 = __int_as_float((unsigned)(e1 + 127) << 23);
        const float s2 = ldexpf(1.f, eg - e1);
        // a coordinate of at least 2^(gx + 71) is a whole number of 2^(gx + 48)
        const float whole = ldexpf(1.f, max(g.gx + 71, -149));
        float top = 0.f;                                   // largest |x| 2^-(gx + 48)
        // the rows of a batch; the next batch is loaded while this one is
        // converted and added
        auto load_batch = [&](int q0, int q1, float (&xv)[U][DPL]) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = q0 + sub + u * RPS;
                const int r = p < q1 ? sm.rowlist[p] : 0;
#pragma unroll
                for (int t = 0; t < DPL; ++t)
                    xv[u][t] = (p < q1 && d0 + t * LPR < n) ? S[tile_at<NP>(lo + r, 0) + dof[t]] : 0.f;
            }
        };
        int j = 0;                                         // the cluster of sorted row b0
        if (b0 < b1)
            for (; j < k; j += 32) {
                const unsigned past = __ballot_sync(0xffffffffu, sm.lstart[min(j + lane + 1, k)] > b0);
                if (past) { j += __ffs(past) - 1; break; }
            }
        int q0 = b0, q1 = b0 < b1 ? min(b1, sm.lstart[j + 1]) : b0;      // its rows in this warp's share
        float xn[U][DPL];
        if (q0 < q1) load_batch(q0, q1, xn);
        while (q0 < q1) {                                  // one cluster at a time
            long long shi[DPL], slo[DPL];
#pragma unroll
            for (int t = 0; t < DPL; ++t) shi[t] = slo[t] = 0;
            const int jc = j;
            int nq0 = q1, nq1 = q1;                        // the next cluster with rows here
            if (q1 < b1) {
                while (sm.lstart[++j + 1] <= q1) {}
                nq1 = min(b1, sm.lstart[j + 1]);
            }
            bool low = false;                              // slo in use
            for (int p0 = q0; p0 < q1; p0 += U * RPS) {
                float xv[U][DPL];
                bool part = false;
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int t = 0; t < DPL; ++t) {
                        xv[u][t] = xn[u][t];
                        part |= fabsf(xv[u][t]) < whole && xv[u][t] != 0.f;
                    }
                if (p0 + U * RPS < q1) load_batch(p0 + U * RPS, q1, xn);
                else if (nq0 < nq1) load_batch(nq0, nq1, xn);
                const bool any_part = __any_sync(0xffffffffu, part);
                low |= any_part;
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int t = 0; t < DPL; ++t) {
                        const float y = __fmul_rn(__fmul_rn(xv[u][t], s1), s2);
                        top = fmaxf(top, fabsf(y));
                        shi[t] += __float2ll_rz(y);        // exact unless `part`: the rest below
                    }
                if (any_part) {
                    // the parts below 2^(gx + 48), whose bits below the grid
                    // are truncated (and counted): the integer fixed_of gives,
                    // split at 2^48 (x 2^-gx in two factors of its own: the
                    // remainder of a truncation at 2^48 is exact)
                    const int f1 = min(-g.gx, 127);
                    const float r1 = __int_as_float((unsigned)(f1 + 127) << 23);
                    const float r2 = __int_as_float((unsigned)(-g.gx - f1 + 127) << 23);
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int t = 0; t < DPL; ++t) {
                            const float y = __fmul_rn(__fmul_rn(xv[u][t], r1), r2);
                            const float lf = __fmaf_rn(-truncf(__fmul_rn(y, 0x1p-48f)), 0x1p48f, y);
                            const float lt = truncf(lf);
                            inex += (lf != lt) ? 1u : 0u;
                            slo[t] += __float2ll_rz(lt);
                        }
                }
            }
            // the warp's sum of the cluster: over the rows of a step, then one
            // lane per dimension adds it to the owner's words
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
                for (int t = 0; t < DPL; ++t) {
                    shi[t] += __shfl_xor_sync(0xffffffffu, shi[t], o);
                    if (low) slo[t] += __shfl_xor_sync(0xffffffffu, slo[t], o);
                }
            if (sub == 0)
#pragma unroll
                for (int t = 0; t < DPL; ++t)
                    add_words(owner_words(jc, d0 + t * LPR), ((__int128)shi[t] << 48) + (__int128)slo[t]);
            q0 = nq0;
            q1 = nq1;
        }
        return top < 0x1p48f;
    }

    // --------------------------------------------- a4/a5: assign + accumulate
    // Assign the CTA's rows against Ccur and push the CTA partial objective to
    // rank 0's inbox.  mode 0: no sums (objective only); mode 1: first
    // assignment of a Lloyd run (the owners' sums start from zero, see
    // lloyd); mode 2: incremental -- the sums are exact integers, so only rows
    // whose label changed since the previous assignment move from their old
    // cluster to the new one.
    struct Tally {                       // what the rows of a thread add up to
        unsigned __int128 f = 0;
        unsigned long long fast = 0;     // distances added in 64 bits (FastSum), at most 64 rows' worth
        int rows = 0;
        unsigned int inex = 0, resc = 0;
        bool ok = true;
        __device__ __forceinline__ void fold() { f += (unsigned __int128)fast << 40; fast = 0; rows = 0; }
    };
    // Rows row0 + 32 r + lane (r < R, below hi) of one warp; [nx0, nx1) are
    // the rows the warp takes next.
    template <int R>
    __device__ __forceinline__ void assign_rows(long long row0, long long lo, long long hi, long long nx0, long long nx1,
                                                int mode, const CertC& cc, const FastSum& fs, Tally& ty) {
        const float gB = a.gB, gp2 = a.gp2;
        const int lane = threadIdx.x & 31;
        float2 m2x[R][NP / 2];                               // -2 x, dimension pairs
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long row = row0 + 32 * r + lane;
            float4 v[NP / 4];
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < hi) load_chunks<0, NP>(row, v);
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) {
                m2x[r][2 * q + 0] = __fmul2_rn(make_float2(-2.f, -2.f), make_float2(v[q].x, v[q].y));
                m2x[r][2 * q + 1] = __fmul2_rn(make_float2(-2.f, -2.f), make_float2(v[q].z, v[q].w));
            }
        }
        int oldlab[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            oldlab[r] = (mode == 2 && row0 + 32 * r + lane < hi) ? lab_prev[row0 + 32 * r + lane] : -1;
        if (nx0 < nx1) {   // start the L2 -> L1 fetch of the warp's next rows (their tiles are contiguous)
            const char* pn = reinterpret_cast<const char*>(S + tile_at<NP>(nx0, 0));
            const int bytes = (int)(nx1 - nx0) * NP * 4;
            for (int o = lane * 128; o < bytes; o += 32 * 128) asm volatile("prefetch.global.L1 [%0];" ::"l"(pn + o));
            if (mode == 2 && lane * 32 < nx1 - nx0)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(lab_prev + nx0 + lane * 32));
        }
        float g1[R], g2[R];
        int j1[R];
#pragma unroll
        for (int r = 0; r < R; ++r) { g1[r] = __int_as_float(0x7f800000); g2[r] = g1[r]; j1[r] = 0; }
        for (int j = 0; j < k; ++j) {
            // g_j = ||c_j||^2 - 2 x.c_j as two interleaved partial sums
            // (even and odd dimensions, packed FP32 FMA), then added:
            // NP + 1 terms in another order, inside the certificate's
            // gamma_{2NP+2} bound.
            const float* cj = sm.Ccur + (size_t)j * NP;
            const float ccj = sm.CC[j];
            float2 e2[R];
#pragma unroll
            for (int r = 0; r < R; ++r) e2[r] = make_float2(ccj, 0.f);
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) {
                const float4 cv = reinterpret_cast<const float4*>(cj)[q];
                const float2 c01 = make_float2(cv.x, cv.y), c23 = make_float2(cv.z, cv.w);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    e2[r] = __ffma2_rn(m2x[r][2 * q + 0], c01, e2[r]);
                    e2[r] = __ffma2_rn(m2x[r][2 * q + 1], c23, e2[r]);
                }
            }
            float e[R];
#pragma unroll
            for (int r = 0; r < R; ++r) e[r] = __fadd_rn(e2[r].x, e2[r].y);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                g2[r] = fminf(g2[r], fmaxf(g1[r], e[r]));
                j1[r] = (e[r] < g1[r]) ? j : j1[r];
                g1[r] = fminf(g1[r], e[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long row = row0 + 32 * r + lane;
            const bool valid = row < hi;
            const float xn2 = xnorm2_up_m2x<NP>(m2x[r]);
            int lab = 0;
            float dv = 0.f;
            if (valid) {
                if (certified_quick(g1[r], g2[r], xn2, cc, gB, gp2) ||
                    certified(g1[r], g2[r], xn2, __fsqrt_ru(xn2), cc, gB, gp2)) {
                    lab = j1[r];
                    dv = d32_m2x<NP>(m2x[r], sm.Ccur + (size_t)lab * NP);
                } else {
                    ty.resc++;
                    dv = d32_m2x<NP>(m2x[r], sm.Ccur);
                    for (int j = 1; j < k; ++j) {
                        const float dj = d32_m2x<NP>(m2x[r], sm.Ccur + (size_t)j * NP);
                        if (dj < dv) { dv = dj; lab = j; }
                    }
                }
                if (dv >= fs.lim && dv < __int_as_float(0x7f800000)) ty.fast += fs.units(dv);
                else acc_obj(ty.f, dv, g.gf, ty.inex);
            }
            if (mode == 1) {
                if (valid) {
                    lab_prev[row] = lab;
                    sm.labs[row - lo] = (unsigned short)lab;
                    atomicAdd(&sm.lcnt[lab], 1);
                }
            } else if (mode == 2) {
                // Move rows whose label changed between clusters.  Many
                // movers: each lane moves its own row.  Few movers (later
                // iterations): the warp moves them one at a time, lanes
                // over dimensions, so the warp does not walk the move path
                // with one or two lanes active.
                const bool moved = valid && oldlab[r] != lab;
                const unsigned mv = __ballot_sync(0xffffffffu, moved);
                if (__popc(mv) > 8) {
                    if (moved) {
                        // the row is in registers (x = -m2x / 2, exact)
                        ty.ok &= move_row_lane(m2x[r], oldlab[r], lab, ty.inex);
                        lab_prev[row] = lab;
                    }
                } else {
                    unsigned rem = mv;
                    while (rem) {
                        const int src = __ffs(rem) - 1;
                        rem &= rem - 1u;
                        const long long srow = __shfl_sync(0xffffffffu, row, src);
                        const int snew = __shfl_sync(0xffffffffu, lab, src);
                        const int sold = __shfl_sync(0xffffffffu, oldlab[r], src);
                        if (lane == src) {
                            red_s32(owner_count(snew), 1);
                            red_s32(owner_count(sold), -1);
                            lab_prev[srow] = snew;
                        }
                        for (int d = lane; d < n; d += 32) {
                            __int128 v;
                            ty.ok &= fixed_of(S[tile_at<NP>(srow, d)], g.gx, ty.inex, v);
                            add_words(owner_words(snew, d), v);
                            add_words(owner_words(sold, d), -v);
                        }
                    }
                }
            }
        }
    }
    // The rows are taken in trips of TPB R rows, R as large as leaves no warp
    // idle: a short remainder (or a small sample's whole slice) is spread over
    // all warps instead of filling a few.
    template <int R>
    __device__ __forceinline__ void assign_trip(int want, long long t0, long long t1, int nwant, long long lo,
                                                long long hi, int mode, const CertC& cc, const FastSum& fs,
                                                Tally& ty) {
        if constexpr (R > 1)
            if (want < R) return assign_trip<R / 2>(want, t0, t1, nwant, lo, hi, mode, cc, fs, ty);
        const int wid = threadIdx.x >> 5;
        const long long row0 = t0 + (long long)wid * 32 * R, nx0 = min(hi, t1 + (long long)wid * 32 * nwant);
        if (row0 < hi)
            assign_rows<R>(row0, lo, hi, nx0, min(hi, nx0 + 32 * nwant), mode, cc, fs, ty);
    }
    __device__ static int trip_rows(long long left) {        // R for the rows that are left
        constexpr int RT = RowsPerThread<NP>::v;
        int R = RT;
        while (R > 1 && left <= (long long)TPB * (R / 2)) R >>= 1;
        return R;
    }
    __device__ void assign_slice(long long s, int mode) {
        constexpr int RT = RowsPerThread<NP>::v;
        long long lo, hi;
        slice(s, lo, hi);
        if (mode == 1)
            for (int e = threadIdx.x; e < k; e += TPB) sm.lcnt[e] = 0;
        __syncthreads();
        const long long t_loop = clock64();
        const CertC cc = *sm.cert;
        const FastSum fs(g.gf);
        Tally ty;
        const int lane = threadIdx.x & 31;
        for (long long t0 = lo; t0 < hi;) {                   // block-uniform
            const int R = trip_rows(hi - t0);
            const long long t1 = t0 + (long long)TPB * R;
            if (ty.rows + R > 64) ty.fold();
            ty.rows += R;
            assign_trip<RT>(R, t0, t1, trip_rows(hi - t1), lo, hi, mode, cc, fs, ty);
            t0 = t1;
        }
        ty.fold();
        unsigned __int128& facc = ty.f;
        unsigned int &inex = ty.inex, &resc = ty.resc;
        bool& ok = ty.ok;
        if (mode == 1) {
            if (tracer()) atomicAdd(&a.glob->trace[15], (unsigned long long)(clock64() - t_loop));
            ok &= bucket_sums(lo, hi, inex);
        }
        if (!ok) atomicOr(&a.glob->err, kErrDigits);
        const long long t_red = clock64();
        if (mode) trace_add(mode == 1 ? 14 : 8, t_loop);   // 14: first assignment of a run
        // one fused CTA reduction: objective (128-bit) and the two counters,
        // pushed into rank 0's inbox
        unsigned __int128 F = warp_sum_u128(facc);
        const unsigned long long IR = warp_sum(((unsigned long long)inex << 32) | resc);
        const int wid = threadIdx.x >> 5;
        if (lane == 0) { sm.red128[wid] = F; sm.red64[wid] = (long long)IR; }
        __syncthreads();
        if (threadIdx.x < 32) {
            F = (lane < (TPB / 32)) ? sm.red128[lane] : (unsigned __int128)0;
            unsigned long long ir = (lane < (TPB / 32)) ? (unsigned long long)sm.red64[lane] : 0ull;
            F = warp_sum_u128(F);
            ir = warp_sum(ir);
            if (lane == 0) {
                ObjPart* dst = cl.map_shared_rank(sm.inbox, 0) + rank;
                dst->f_lo = (unsigned long long)F;
                dst->f_hi = (unsigned long long)(F >> 64);
                dst->inexact = ir >> 32;
                dst->rescored = ir & 0xffffffffull;
            }
        }
        if (mode) trace_add(9, t_red);
    }

    // After a barrier, on rank 0, warp 0: the CTA partials of the inbox
    // combined into the cluster's partial (exact; valid in lane 0).
    __device__ void cluster_objective_warp(unsigned __int128& F, unsigned long long& I, unsigned long long& R) {
        const int lane = threadIdx.x & 31;
        F = 0; I = 0; R = 0;
        for (int q = lane; q < cs; q += 32) {
            const ObjPart& p = sm.inbox[q];
            F += ((unsigned __int128)p.f_hi << 64) | (unsigned __int128)p.f_lo;
            I += p.inexact;
            R += p.rescored;
        }
        F = warp_sum_u128(F);
        I = warp_sum(I);
        R = warp_sum(R);
    }
    // The worker's objective from partials (F, I, R) of every cluster: with
    // one cluster these are the partials themselves; with a group, rank 0 of
    // each cluster publishes its partial (before the group barrier) and adds
    // up all of them (after it).  f = the exact sum rounded once (lane 0);
    // the counters are recorded once per worker.
    __device__ void publish_objective(const unsigned __int128& F, unsigned long long I, unsigned long long R) {
        if (G > 1 && (threadIdx.x & 31) == 0) {
            unsigned long long* o = a.xobj + xslot(xpar, gi) * 4;
            o[0] = (unsigned long long)F;
            o[1] = (unsigned long long)(F >> 64);
            o[2] = I;
            o[3] = R;
        }
    }
    __device__ double total_objective(unsigned __int128 F, unsigned long long I, unsigned long long R) {
        if (G > 1) {                                 // a lane per cluster
            F = 0; I = 0; R = 0;
            if ((int)(threadIdx.x & 31) < G) {
                const volatile unsigned long long* o = a.xobj + xslot(xpar, threadIdx.x & 31) * 4;
                F = ((unsigned __int128)o[1] << 64) | (unsigned __int128)o[0];
                I = o[2];
                R = o[3];
            }
            F = warp_sum_u128(F);
            I = warp_sum(I);
            R = warp_sum(R);
        }
        if ((threadIdx.x & 31) == 0 && gi == 0) {
            if (I) atomicAdd(&a.glob->inexact, I);
            if (R) atomicAdd(&a.glob->rescored, R);
        }
        return u128_to_double(F, g.gf);
    }
    // Owners add their clusters' partial sums and counts to the group's (group
    // only).  Three buffers take turns: one is added to before the barrier and
    // read after it, and the one read after the barrier before is cleared
    // then, two barriers before it is added to again.  (With a slot per
    // cluster every owner read G slots one after the other.)
    __device__ void publish_sums() {
        if (G == 1) return;
        const int nOwned = (k - rank + cs - 1) / cs;
        for (int e = threadIdx.x; e < nOwned * NP; e += TPB) {
            const int slot = e / NP, d = e % NP, j = rank + slot * cs;
            const long long* wd = sm.OACC + (size_t)e * kAccWords;
            unsigned long long* o = reinterpret_cast<unsigned long long*>(xwords(xrot, j, d));
#pragma unroll
            for (int i = 0; i < kAccWords; ++i)
                if (wd[i]) atomicAdd(o + i, (unsigned long long)wd[i]);
            if (d == 0 && sm.ocnt[slot]) atomicAdd(xcount(xrot, j), sm.ocnt[slot]);
        }
    }
    // Rank 0, one thread: the decision to every CTA of the cluster.
    __device__ void push_decision(double f, int stop) {
        for (int q = 0; q < cs; ++q) {
            Decision* d = cl.map_shared_rank(sm.dec, q);
            d->f = f;
            d->stop = stop;
        }
    }

    // Zero the owned sums and counts (before a Lloyd run; a cluster barrier
    // must follow before any CTA adds to them).
    __device__ void zero_owned() {
        const int nOwned = (k - rank + cs - 1) / cs;
        for (int e = threadIdx.x; e < nOwned * NP * kAccWords; e += TPB) sm.OACC[e] = 0;
        for (int e = threadIdx.x; e < nOwned; e += TPB) sm.ocnt[e] = 0;
    }

    // a6 (owner part): new centroid of each owned cluster j (j % cs == rank):
    // float(double(exact sum) / count); an empty cluster keeps its centroid.
    // The sums are complete in this CTA's shared memory; the new centroids
    // and the empty flags are pushed into every CTA's Cnext / emptyall.
    __device__ void owner_update() {
        const int nOwned = (k - rank + cs - 1) / cs;
        const int total = nOwned * NP;
        for (int e = threadIdx.x; e < total; e += TPB) {
            const int slot = e / NP, d = e % NP;
            const int j = rank + slot * cs;
            __int128 V = 0;
            long long cntj = 0;
            if (G == 1) {
                const long long* wd = sm.OACC + (size_t)e * kAccWords;
                V = (__int128)wd[0] + ((__int128)wd[1] << 32) + ((__int128)wd[2] << 64);
                cntj = sm.ocnt[slot];
            } else {                                 // the group's sums, in global memory
                const long long* wd = xwords(xrot, j, d);
                const long long w0 = __ldcg(wd), w1 = __ldcg(wd + 1), w2 = __ldcg(wd + 2);
                cntj = __ldcg(xcount(xrot, j));
                V = (__int128)w0 + ((__int128)w1 << 32) + ((__int128)w2 << 64);
                if (gi == 0) {                       // the buffer of the exchange before: cleared for the next but one
                    const int old = xrot == 0 ? 2 : xrot - 1;
                    long long* z = xwords(old, j, d);
                    z[0] = 0; z[1] = 0; z[2] = 0;
                    if (d == 0) *xcount(old, j) = 0;
                }
            }
            float c = sm.Ccur[(size_t)j * NP + d];
            if (cntj > 0 && d < n) {
                c = __double2float_rn(__ddiv_rn(i128_to_double(V, g.gx), (double)cntj));
            }
            const unsigned char em = (cntj == 0) ? 1 : 0;
            for (int q = 0; q < cs; ++q) {
                cl.map_shared_rank(sm.Cnext, q)[(size_t)j * NP + d] = c;
                if (d == 0) cl.map_shared_rank(sm.emptyall, q)[j] = em;
            }
        }
    }

    // f(Ccur, S) without updating centroids (recompute of f_hat_w, recheck).
    __device__ double eval(long long s) {
        assign_slice(s, 0);
        cl.sync();                                       // partials in rank 0's inbox
        unsigned __int128 F = 0;
        unsigned long long I = 0, R = 0;
        if (rank == 0 && threadIdx.x < 32) {
            cluster_objective_warp(F, I, R);
            publish_objective(F, I, R);
        }
        gsync();                                         // every cluster's partial published
        if (rank == 0 && threadIdx.x < 32) {
            const double f = total_objective(F, I, R);
            if (threadIdx.x == 0) push_decision(f, 1);
        }
        xpar ^= 1;
        cl.sync();                                       // decision in every CTA
        const double f = sm.dec->f;
        if (lead() && threadIdx.x == 0) atomicAdd(&a.glob->eval_rows, (unsigned long long)s);
        return f;
    }

    // Lloyd from Ccur (Sec. 4.1; Sec. 5 stop rule).  On return Ccur holds the
    // result C_a, emptyall its empty clusters, `iters` the number of updates.
    __device__ double lloyd(long long s, int& iters) {
        zero_owned();
        cl.sync();                                       // no CTA adds before the owners cleared
        double f_prev = 0.0;
        int it = 0;
        for (;;) {
            const long long t_a = clock64();
            assign_slice(s, it == 0 ? 1 : 2);
            trace_add(1, t_a);
            if (tracer()) atomicAdd(&a.glob->trace[6], 1ull);
            const long long t_x = clock64();
            cl.sync();                                       // sums and partials at their owners
            trace_add(10, t_x);
            const long long t_o = clock64();
            unsigned __int128 F = 0;
            unsigned long long I = 0, R = 0;
            if (G > 1) {                                     // partials of every cluster of the group
                publish_sums();
                if (rank == 0 && threadIdx.x < 32) {
                    cluster_objective_warp(F, I, R);
                    publish_objective(F, I, R);
                }
                gsync();
            } else if (rank == 0 && threadIdx.x < 32) {
                cluster_objective_warp(F, I, R);
            }
            owner_update();
            if (rank == 0 && threadIdx.x < 32) {
                const double f = total_objective(F, I, R);
                if (threadIdx.x == 0) {
                    int stop;
                    if (it == 0) stop = (a.max_lloyd <= 0);
                    else stop = (__dsub_rn(f_prev, f) <= __dmul_rn(a.tol, f_prev)) || (it >= a.max_lloyd);
                    if (group_aborted()) stop = 1;
                    push_decision(f, stop);
                }
            }
            xpar ^= 1;
            xrot = xrot == 2 ? 0 : xrot + 1;
            trace_add(11, t_o);
            const long long t_b2 = clock64();
            cl.sync();                                       // updates + decision in every CTA
            trace_add(12, t_b2);
            const long long t_p = clock64();
            const double f = sm.dec->f;
            const int stop = sm.dec->stop;
            if (stop) {
                trace_add(2, t_x);
                iters = it;
                return f;
            }
            for (int e = threadIdx.x; e < k * NP; e += TPB) sm.Ccur[e] = sm.Cnext[e];
            __syncthreads();
            prep_centroids();
            trace_add(13, t_p);
            trace_add(2, t_x);
            f_prev = f;
            ++it;
        }
    }

    // ------------------------------------------------ a3: greedy K-means++
    __device__ static int frexp_exp(unsigned int mb) {   // M = f * 2^E, f in [0.5, 1)
        const unsigned ef = mb >> 23;
        if (ef) return (int)ef - 126;
        return (32 - __clz((int)(mb & 0x7fffff))) - 149;
    }
    __device__ static long long quant(float v, int E) {   // floor(v * 2^(31 - E))
        const uint32_t b = __float_as_uint(v) & 0x7fffffffu;
        if (!b) return 0;
        uint32_t mant; int e2;
        f32_parts(b, mant, e2);
        const int sh = e2 + 31 - E;
        if (sh >= 0) return (long long)mant << sh;
        if (-sh >= 32) return 0;
        return (long long)(mant >> (-sh));
    }

    __device__ void load_row(long long i, float (&x)[NP]) const {
        float4 v[NP / 4];
        load_chunks<0, NP>(i, v);
#pragma unroll
        for (int q = 0; q < NP / 4; ++q) {
            x[4 * q] = v[q].x; x[4 * q + 1] = v[q].y; x[4 * q + 2] = v[q].z; x[4 * q + 3] = v[q].w;
        }
    }

    // D^2 buffer b (0..3) of the worker: one holds D^2, the others the D^2
    // each candidate would leave, so that taking a candidate is a change of
    // buffer and no distance is computed twice.
    __device__ float* d2buf(int b) const { return D2 + (size_t)b * a.D2_stride; }

    // Rows of warp `v` of the worker's CTA `cta`: contiguous, so that prefix
    // sums over CTAs, warps and rows run in row order.
    __device__ void kpp_rows(long long s, int cta, int v, long long& w0, long long& w1) const {
        const long long lo = s * cta / nW, rows = s * (cta + 1) / nW - lo;
        w0 = lo + rows * v / (TPB / 32);
        w1 = lo + rows * (v + 1) / (TPB / 32);
    }

    // One exchange of K-means++ among every CTA of the worker: each publishes
    // NT sums of weights (per warp and in all) and maxima, then, after a
    // barrier, every CTA works out the same answer from the published words
    // alone: the array `best` with the least total (the lowest on ties), its
    // maximum M and, when M still has the exponent E (or E is kNoExp: nothing
    // to draw from) and `jdraw` < k, the `trials` candidate rows of centroid
    // jdraw: the rows at which the prefix of the weights of D^2 buffer
    // bufs[best] passes the draws.  Warp l finds candidate l by a scan over
    // the CTAs, over the warps of one CTA and over the rows of one warp, and
    // leaves the row in candbuf.  One barrier per centroid is the only time
    // the CTAs wait for one another.
    static constexpr int kNoExp = 1 << 20;
    static_assert(8 + 3 * kMaxWarps <= 64, "a CTA's slot: totals, maxima and the sums of its warps");
    __device__ float* candbuf(int par, int l) const {       // in the (idle) sums: 24 NP bytes per cluster, k >= 2
        return reinterpret_cast<float*>(sm.OACC) + (par * 3 + l) * NP;
    }
    __device__ void kpp_exchange(long long s, int NT, const long long (&sum)[3], const unsigned (&mx)[3], int E,
                                 const int (&bufs)[3], int jdraw, int trials, unsigned long long k1, int cpar) {
        constexpr int NW = TPB / 32;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        long long* wsum = reinterpret_cast<long long*>(sm.inbox);       // [3][kMaxWarps]: 384 of 512 bytes
        unsigned* wmax = reinterpret_cast<unsigned*>(sm.red128);        // [3][kMaxWarps]: 192 of 256 bytes
        for (int l = 0; l < NT; ++l) {
            const long long v = warp_sum(l == 0 ? sum[0] : l == 1 ? sum[1] : sum[2]);
            const unsigned mv = __reduce_max_sync(0xffffffffu, l == 0 ? mx[0] : l == 1 ? mx[1] : mx[2]);
            if (lane == 0) { wsum[l * kMaxWarps + wid] = v; wmax[l * kMaxWarps + wid] = mv; }
        }
        __syncthreads();
        long long* slots = a.kx + ((size_t)w * 2 + kpar) * a.kx_ctas * 64;
        kpar ^= 1;
        if (wid == 0) {
            long long* my = slots + (size_t)ctaW * 64;
            for (int e = lane; e < NT * NW; e += 32)
                my[8 + (e / NW) * kMaxWarps + e % NW] = wsum[(e / NW) * kMaxWarps + e % NW];
            if (lane < NT) {
                long long t = 0;
                unsigned mv = 0;
                for (int v = 0; v < NW; ++v) {
                    t += wsum[lane * kMaxWarps + v];
                    mv = max(mv, wmax[lane * kMaxWarps + v]);
                }
                my[lane] = t;
                my[4 + lane] = (long long)mv;
            }
            __syncwarp();
        }
        if (G == 1) {
            cl.sync();
        } else {
            ++gepoch;
            if (threadIdx.x == 0) {
                __threadfence();
                atomicAdd(a.xbar + w, 1u);
            }
            if (wid < 3) {                                  // the warps that read what the others published
                if (lane == 0) gwait();
                __syncwarp();
            }
        }
        if (wid < 3) {
            // lane's CTAs: [lane ch, (lane + 1) ch)
            const int ch = (nW + 31) / 32;
            const int q0 = lane * ch, q1 = min(nW, q0 + ch);
            long long tot[3] = {0, 0, 0};
            unsigned mm[3] = {0, 0, 0};
            for (int q = q0; q < q1; ++q)
#pragma unroll
                for (int l = 0; l < 3; ++l)
                    if (l < NT) {
                        tot[l] += __ldcg(slots + (size_t)q * 64 + l);
                        mm[l] = max(mm[l], (unsigned)__ldcg(slots + (size_t)q * 64 + 4 + l));
                    }
            int best = 0;
            long long Wtot = 0;
#pragma unroll
            for (int l = 0; l < 3; ++l)
                if (l < NT) {
                    long long t = tot[l];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    if (l == 0 || t < Wtot) { Wtot = t; best = l; }
                }
            const unsigned M = __reduce_max_sync(0xffffffffu, best == 0 ? mm[0] : best == 1 ? mm[1] : mm[2]);
            if (threadIdx.x == 0) { sm.bcast[2] = best; sm.bcast[3] = (long long)M; }
            if (jdraw < k && E != kNoExp && M != 0 && frexp_exp(M) == E && wid < trials) {
                const unsigned long long u = draw_below(a.seed, k1, (unsigned long long)wid, (unsigned long long)jdraw,
                                                        (unsigned long long)Wtot);
                long long rest = (long long)u;
                // the CTA
                const long long mine = best == 0 ? tot[0] : best == 1 ? tot[1] : tot[2];
                long long pre = warp_scan(mine);
                int src = __ffs(__ballot_sync(0xffffffffu, rest < pre)) - 1;
                bool bad = src < 0;                          // cannot happen: the prefix covers [0, Wtot)
                src = max(src, 0);
                rest -= __shfl_sync(0xffffffffu, pre - mine, src);
                int q = min(src * ch, nW - 1);
                for (; q + 1 < min(nW, src * ch + ch); ++q) {
                    const long long t = __ldcg(slots + (size_t)q * 64 + best);
                    if (rest < t) break;
                    rest -= t;
                }
                // its warp
                const long long wm = lane < NW ? __ldcg(slots + (size_t)q * 64 + 8 + best * kMaxWarps + lane) : 0;
                pre = warp_scan(wm);
                src = __ffs(__ballot_sync(0xffffffffu, rest < pre)) - 1;
                bad |= src < 0;
                src = max(src, 0);
                rest -= __shfl_sync(0xffffffffu, pre - wm, src);
                // the row: lanes over equal contiguous pieces of the warp's rows
                long long w0, w1;
                kpp_rows(s, q, src, w0, w1);
                const int bb = best == 0 ? bufs[0] : best == 1 ? bufs[1] : bufs[2];
                const float* dv = d2buf(bb);
                const long long piece = (w1 - w0 + 31) / 32;
                const long long p0 = min(w1, w0 + piece * lane), p1 = min(w1, p0 + piece);
                long long ps = 0;
                for (long long i = p0; i < p1; i += 8) {     // eight loads in flight
                    float t[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) t[e] = i + e < p1 ? __ldcg(dv + i + e) : 0.f;
#pragma unroll
                    for (int e = 0; e < 8; ++e) ps += quant(t[e], E);
                }
                pre = warp_scan(ps);
                src = __ffs(__ballot_sync(0xffffffffu, rest < pre)) - 1;
                bad |= src < 0;
                src = max(src, 0);
                rest -= __shfl_sync(0xffffffffu, pre - ps, src);
                const long long a0 = __shfl_sync(0xffffffffu, p0, src), a1 = __shfl_sync(0xffffffffu, p1, src);
                long long row = -1;
                for (long long r0 = a0; r0 < a1; r0 += 32) {     // that piece, a lane per row
                    const long long t = r0 + lane < a1 ? quant(__ldcg(dv + r0 + lane), E) : 0;
                    pre = warp_scan(t);
                    const unsigned hit = __ballot_sync(0xffffffffu, rest < pre);
                    if (hit) { row = r0 + __ffs(hit) - 1; break; }
                    rest -= __shfl_sync(0xffffffffu, pre, 31);
                }
                if (bad || row < 0 || row >= s) {
                    if (lane == 0) atomicOr(&a.glob->err, group_aborted() ? kErrTimeout : kErrArgs);
                    row = 0;
                }
                float* cb = candbuf(cpar, wid);
                for (int d = lane; d < NP; d += 32) cb[d] = S[tile_at<NP>(row, d)];
            }
        }
        __syncthreads();
    }

    // Greedy K-means++ of the degenerate centroids, by every CTA of the worker
    // (all clusters of a group).  What bounded it: cluster 0 alone computed
    // the distances of the whole sample, each centroid took four barriers with
    // serial scans between them, and the winner's distances were computed
    // again.  Now a centroid costs one pass over the CTA's rows and one
    // exchange: the candidates' potentials are at the same time the weight
    // sums of the next draw as long as the largest D^2 keeps its exponent (the
    // quantisation grid), else one more pass over D^2 and two exchanges.
    // A candidate's distances are cut short where they cannot matter: partial
    // sums of squares never decrease (each addition is rounded, the terms are
    // not negative), so once every row of a warp has reached its D^2 the
    // minimum is D^2, whatever the other dimensions hold.
    // Measured: seeding k = 50 on 64,000 x 32 by one cluster 2.38 -> 1.5 ms;
    // the worker launch of 8 workers at 10^7 x 64, k = 100 (40,000-row samples)
    // 17.8 -> 6.7 ms, of which the smaller shared memory (owned_slots) 6 ms.
    __device__ void kmeanspp(long long s, unsigned long long k1) {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        long long w0, w1;
        kpp_rows(s, ctaW, wid, w0, w1);
        const int trials = a.trials < 1 ? 1 : (a.trials > 3 ? 3 : a.trials);
        auto next_deg = [&](int j) { ++j; while (j < k && !sm.deg[j]) ++j; return j; };
        auto count = [&] { if (lead() && threadIdx.x == 0) atomicAdd(&a.glob->reseeded, 1ull); };
        bool any_live = false;
        for (int j = 0; j < k; ++j) any_live |= (sm.deg[j] == 0);
        int j = next_deg(-1);
        int cur = 0;
        if (!any_live) {                                     // the first centroid: uniform
            const long long pick = (long long)draw_below(a.seed, k1, 0, (unsigned long long)j, (unsigned long long)s);
            count();
            for (int d = threadIdx.x; d < NP; d += TPB) sm.Ccur[(size_t)j * NP + d] = S[tile_at<NP>(pick, d)];
            __syncthreads();
            for (long long i = w0 + lane; i < w1; i += 32) {
                float x[NP];
                load_row(i, x);
                d2buf(cur)[i] = d32<NP>(x, sm.Ccur + (size_t)j * NP);
            }
            j = next_deg(j);
        } else {
            for (long long i = w0 + lane; i < w1; i += 32) {
                float x[NP];
                load_row(i, x);
                float dm = __int_as_float(0x7f800000);
                for (int c = 0; c < k; ++c)
                    if (!sm.deg[c]) dm = fminf(dm, d32<NP>(x, sm.Ccur + (size_t)c * NP));
                d2buf(cur)[i] = dm;
            }
        }
        bool drawn = false;                                  // candidates of centroid j are in candbuf(cpar, .)
        int cpar = 0, E = kNoExp;
        while (j < k) {
            if (!drawn) {                                    // the grid's exponent, then the weights on it
                long long ws[3] = {0, 0, 0};
                unsigned mx[3] = {0, 0, 0};
                const int bf[3] = {cur, cur, cur};
                for (long long i = w0 + lane; i < w1; i += 32) mx[0] = max(mx[0], __float_as_uint(d2buf(cur)[i]));
                kpp_exchange(s, 1, ws, mx, kNoExp, bf, k, trials, k1, cpar);
                const unsigned M = (unsigned)sm.bcast[3];
                if (M == 0) {                                // every row sits on a centroid: uniform picks
                    for (; j < k; j = next_deg(j)) {
                        const long long pick = (long long)draw_below(a.seed, k1, 0, (unsigned long long)j,
                                                                     (unsigned long long)s);
                        count();
                        for (int d = threadIdx.x; d < NP; d += TPB) sm.Ccur[(size_t)j * NP + d] = S[tile_at<NP>(pick, d)];
                    }
                    break;
                }
                E = frexp_exp(M);
                for (long long i = w0 + lane; i < w1; i += 32) ws[0] += quant(d2buf(cur)[i], E);
                kpp_exchange(s, 1, ws, mx, E, bf, j, trials, k1, cpar);
            }
            // potentials of the candidates, and the D^2 each would leave.  The
            // next row is on its way while this one is scored: all of it, or
            // for NP = 64 its first 16 dimensions (the others are asked for
            // 16 dimensions ahead).
            constexpr int H = NP <= 8 ? NP : (NP == 64 ? 16 : 8);    // dimensions between cuts
            constexpr int PF = NP == 64 ? 16 : NP;                   // dimensions fetched a row ahead
            const float* c0 = candbuf(cpar, 0);
            const float* dcur = d2buf(cur);
            float* dn[3] = {d2buf((cur + 1) & 3), d2buf((cur + 2) & 3), d2buf((cur + 3) & 3)};
            const int bf[3] = {(cur + 1) & 3, (cur + 2) & 3, (cur + 3) & 3};
            long long pot[3] = {0, 0, 0};
            unsigned mx[3] = {0, 0, 0};
            float4 xn[PF / 4];
            float d2n = 0.f;
            auto fetch = [&](long long i) {
                if (i < w1) {
                    d2n = dcur[i];
                    load_chunks<0, PF>(i, xn);
                }
            };
#pragma unroll
            for (int q = 0; q < PF / 4; ++q) xn[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            fetch(w0 + lane);
            for (long long b = w0; b < w1; b += 32) {        // warp-uniform trips
                const long long i = b + lane;
                const bool valid = i < w1;
                float4 x[PF / 4];
#pragma unroll
                for (int q = 0; q < PF / 4; ++q) x[q] = xn[q];
                const float d2 = d2n;
                fetch(i + 32);
                const float* rest = S + tile_at<NP>(valid ? i : w0, 0);
                float4 v[2][H / 4];                          // NP = 64: the chunk in hand and the next one
                float acc[3] = {0.f, 0.f, 0.f};
                auto add = [&](int l, const float4& xv, int q) {
                    const float4 c = *reinterpret_cast<const float4*>(c0 + l * NP + 4 * q);
                    float2 t0 = __fadd2_rn(make_float2(xv.x, xv.y), make_float2(-c.x, -c.y));
                    float2 t1 = __fadd2_rn(make_float2(xv.z, xv.w), make_float2(-c.z, -c.w));
                    t0 = __fmul2_rn(t0, t0);
                    t1 = __fmul2_rn(t1, t1);
                    acc[l] = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc[l], t0.x), t0.y), t1.x), t1.y);
                };
                bool go[3] = {true, trials > 1, trials > 2};
#pragma unroll
                for (int h = 0; h < NP / H; ++h) {
                    if (h > 0) {
#pragma unroll
                        for (int l = 0; l < 3; ++l)
                            go[l] = go[l] && __any_sync(0xffffffffu, valid && acc[l] < d2);
                        if (!(go[0] || go[1] || go[2])) break;
                    }
                    if (PF < NP && h + 1 < NP / H)
#pragma unroll
                        for (int c = 0; c < H / 8; ++c)
                            ld8(rest + ((h + 1) * (H / 8) + c) * 32, v[(h + 1) & 1][2 * c], v[(h + 1) & 1][2 * c + 1]);
#pragma unroll
                    for (int l = 0; l < 3; ++l)
                        if (go[l])
#pragma unroll
                            for (int q = 0; q < H / 4; ++q)
                                add(l, (PF == NP || h == 0) ? x[((PF == NP ? h : 0) * (H / 4) + q)] : v[h & 1][q],
                                    h * (H / 4) + q);
                }
                if (valid) {
#pragma unroll
                    for (int l = 0; l < 3; ++l)
                        if (l < trials) {
                            const float m = fminf(d2, acc[l]);
                            dn[l][i] = m;
                            pot[l] += quant(m, E);
                            mx[l] = max(mx[l], __float_as_uint(m));
                        }
                }
            }
            const int jn = next_deg(j);
            kpp_exchange(s, trials, pot, mx, E, bf, jn, trials, k1, cpar ^ 1);
            const int best = (int)sm.bcast[2];
            const unsigned M = (unsigned)sm.bcast[3];
            count();
            for (int d = threadIdx.x; d < NP; d += TPB) sm.Ccur[(size_t)j * NP + d] = candbuf(cpar, best)[d];
            cur = bf[best];
            drawn = M != 0 && frexp_exp(M) == E;
            cpar ^= 1;
            j = jn;
        }
        __syncthreads();
    }
};

// BATCH: a launch for several fits, whose arguments are read from device
// memory (p.batch[fit of the cluster]); otherwise the kernel parameter itself.
template <int NP, int TPB, bool BATCH>
__global__ void __launch_bounds__(TPB, 512 / TPB) worker_kernel(const __grid_constant__ WorkerArgs p) {
    // The launch must have the cluster shape and grid the arguments describe
    // (every exchange addresses the other CTAs of the cluster by rank): if
    // not, record the error and leave before any barrier or remote access.
    if (cg::this_cluster().num_blocks() != (unsigned)p.cs || gridDim.x % (unsigned)p.cs != 0 ||
        (p.ncl > 0 && gridDim.x != (unsigned)(p.ncl * p.cs))) {
        if (threadIdx.x == 0) atomicOr(&p.glob->err, kErrArgs);
        return;
    }
    const WorkerArgs& a = BATCH ? p.batch[(p.cmap[blockIdx.x / p.cs] >> 12) & 0xfu] : p;
    Worker<NP, TPB> W(a, cg::this_cluster());
    if (a.glob->nonfinite) return;            // uniform: read before any barrier
    const int w = W.w;

    if (a.mode == kModeStepKpp || a.mode == kModeStepLloyd) {
        // S (padded) and C (padded, in a.Cw) were staged by the host.
        W.load_centroids(a.Cw);
        for (int j = threadIdx.x; j < W.k; j += TPB) W.sm.deg[j] = a.deg[j];
        __syncthreads();
        W.cl.sync();
        if (a.mode == kModeStepKpp) {
            W.kmeanspp(a.step_s, stream_k1(kPurposeKpp, a.step_worker, a.step_round, a.step_pass));
        } else {
            W.prep_centroids();
            int iters = 0;
            const double f = W.lloyd(a.step_s, iters);
            if (W.lead() && threadIdx.x == 0) { *a.step_f = f; *a.step_iters = iters; }
            if (W.lead())
                for (int j = threadIdx.x; j < W.k; j += TPB) a.step_empty[j] = W.sm.emptyall[j];
        }
        if (W.lead()) W.store_centroids(a.Cw);
        W.csync_global();
        return;
    }

    // worker state for this launch
    const long long t_kernel = clock64();
    for (int j = threadIdx.x; j < W.k; j += TPB) W.sm.deg[j] = a.deg[(long long)w * W.k + j];
    for (int e = threadIdx.x; e < W.k * NP; e += TPB)
        W.Cw_mine[e] = a.Cw[(long long)w * W.k * NP + e];
    __syncthreads();
    double fhat = a.fhat[w];

    if (a.mode == kModeFinalEval) {
        // the common sample S (job 0 of the final sampling launch)
        W.S = a.S;
        const long long s_opt = a.job_s[0];
        W.load_centroids(W.Cw_mine);
        W.prep_centroids();
        const double f = W.eval(s_opt);
        if (W.lead() && threadIdx.x == 0) a.f_final[w] = f;
        W.cl.sync();
        return;
    }

    // ---------------------------------------------------- Algorithm 1 round
    // Samples of this round were drawn and gathered by the sampling kernel:
    // slots 0..P-1 are the passes, slot P the f_hat recompute sample.
    bool failed = false, out_of_time = false;
    int rounds_completed = 0;
    for (int t = a.round_begin; t < a.round_end && !failed && !out_of_time; ++t) {
        const long long s_w = W.use_sample(a.P);
        if (s_w <= 0) { failed = true; break; }
        bool all_deg = true;
        for (int j = 0; j < W.k; ++j) all_deg &= (W.sm.deg[j] != 0);
        if (!all_deg) {                                  // recompute f_hat_w with the new s_w
            const long long t_e = clock64();
            W.load_centroids(W.Cw_mine);
            W.prep_centroids();
            fhat = W.eval(s_w);
            W.trace_add(3, t_e);
        }
        for (int p = 0; p < a.P; ++p) {
            if (a.deadline_ns) {
                // the lead CTA reads the clock; its decision reaches every CTA
                // of the cluster (and, for a group, every cluster)
                if (W.lead() && threadIdx.x == 0) {
                    unsigned long long now;
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                    const int late = (now >= a.deadline_ns) ? 1 : 0;
                    W.sm.x->flag = late;
                    if (W.G > 1) a.xflag[(size_t)w * 2 + W.xpar] = late;
                }
                if (W.G > 1) {
                    W.gsync();
                    if (threadIdx.x == 0) W.sm.bcast[8] = *(const volatile int*)(a.xflag + (size_t)w * 2 + W.xpar);
                    W.xpar ^= 1;
                } else {
                    W.cl.sync();
                    if (threadIdx.x == 0) W.sm.bcast[8] = W.rx(0)->flag;
                }
                __syncthreads();
                const bool late = W.sm.bcast[8] != 0;
                W.cl.sync();
                if (late) { out_of_time = true; break; }
            }
            W.use_sample(p);
            W.load_centroids(W.Cw_mine);
            bool any_deg = false;
            for (int j = 0; j < W.k; ++j) any_deg |= (W.sm.deg[j] != 0);
            if (any_deg) {
                // re-seeding is in place (Alg. 1)
                const long long t_k = clock64();
                W.kmeanspp(s_w, stream_k1(kPurposeKpp, w, t, p));
                W.store_centroids(W.Cw_mine);
                W.trace_add(0, t_k);
            }
            W.prep_centroids();
            int iters = 0;
            const double f = W.lloyd(s_w, iters);
            if (f < fhat) {                              // incumbent rule
                fhat = f;
                for (int j = threadIdx.x; j < W.k; j += TPB) W.sm.deg[j] = W.sm.emptyall[j];
                W.store_centroids(W.Cw_mine);
                if (W.lead() && threadIdx.x == 0) {
                    const unsigned long long pos = atomicAdd(&a.glob->accepts, 1ull);
                    atomicAdd(&a.glob->L_sum, (unsigned long long)s_w);
                    if ((long long)pos < a.L_cap) a.L_buf[pos] = s_w;
                }
            }
            __syncthreads();
            if (W.lead() && threadIdx.x == 0) {
                atomicAdd(&a.glob->passes, 1ull);
                atomicAdd(&a.glob->lloyd_iters, (unsigned long long)iters);
                atomicAdd(&a.glob->assign_rows, (unsigned long long)(s_w * (iters + 1)));
            }
        }
        if (!failed && !out_of_time) ++rounds_completed;
    }
    if (failed && W.lead() && threadIdx.x == 0) atomicOr(&a.glob->err, kErrSample);
    // persist worker state
    if (W.lead()) {
        for (int e = threadIdx.x; e < W.k * NP; e += TPB)
            a.Cw[(long long)w * W.k * NP + e] = W.Cw_mine[e];
        for (int j = threadIdx.x; j < W.k; j += TPB) a.deg[(long long)w * W.k + j] = W.sm.deg[j];
        if (threadIdx.x == 0) {
            a.fhat[w] = fhat;
            atomicMin(&a.glob->rounds_done, a.round_begin + rounds_completed);
            const unsigned long long dt = (unsigned long long)(clock64() - t_kernel);
            atomicAdd(&a.glob->trace[4], dt);
            atomicMax(&a.glob->trace[5], dt);
            atomicAdd(&a.glob->trace[7], 1ull);
        }
    }
    W.csync_global();
}

template <int NP>
int worker_max_cluster_t(int k) {
    const size_t smem = worker_smem_bytes<NP>(k, 1);
    if (allow_max_smem((const void*)worker_kernel<NP, 256, false>) != cudaSuccess ||
        allow_max_smem((const void*)worker_kernel<NP, 512, false>) != cudaSuccess ||
        cudaFuncSetAttribute(worker_kernel<NP, 256, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(worker_kernel<NP, 512, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return 8;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 16;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, worker_kernel<NP, 256, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 8;
    }
    return nclusters > 0 ? 16 : 8;
}

template <int NP>
int worker_active_clusters_t(int cs, size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<int, size_t>, int> memo;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(cs, smem);
    const auto it = memo.find(key);
    if (it != memo.end()) return it->second;
    if (allow_max_smem((const void*)worker_kernel<NP, 256, false>) != cudaSuccess ||
        (cs > 8 && cudaFuncSetAttribute(worker_kernel<NP, 256, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                       cudaSuccess)) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, worker_kernel<NP, 256, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        ncl = 0;
    }
    memo[key] = ncl;
    return ncl;
}

template <int NP, int TPB, bool BATCH>
cudaError_t launch_worker_tpb(const WorkerArgs& a, int clusters, cudaStream_t st) {
    const size_t smem = worker_smem_bytes<NP>(a.k_smem > 0 ? a.k_smem : a.k, a.cs) + bucket_smem_bytes(a.rows_cta);
    cudaError_t e = allow_max_smem((const void*)worker_kernel<NP, TPB, BATCH>);
    if (e != cudaSuccess) return e;
    if (a.cs > 8) {
        e = cudaFuncSetAttribute(worker_kernel<NP, TPB, BATCH>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * a.cs), 1, 1);
    cfg.blockDim = dim3(TPB, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.coop ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, worker_kernel<NP, TPB, BATCH>, a);
}

// a.tpb = 512 runs the worker with 512-thread CTAs (one per SM), else 256.
template <int NP>
cudaError_t launch_worker_t(const WorkerArgs& a, int clusters, cudaStream_t st) {
    if (a.batch) return launch_worker_tpb<NP, 256, true>(a, clusters, st);
    return a.tpb == 512 ? launch_worker_tpb<NP, 512, false>(a, clusters, st)
                        : launch_worker_tpb<NP, 256, false>(a, clusters, st);
}

}  // namespace bm
