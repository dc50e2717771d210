// k_select.cu -- the selection phase (Sec. "Selection phase": cluster_threshold,
// numb_cluster_lower / numb_cluster_upper, max_selection; Sec. "Selection":
// explored CVs are clustered and the values with high model deviation are
// collected by the trust levels; Sec. "CV selection": per-CV clustering
// weights and the angular mask).
//
//   k_sel_count / k_sel_scan / k_sel_scatter
//                     frames with trust_lo <= eps < trust_hi, compacted in
//                     frame order over the whole grid (counts per block of
//                     1024 frames, their prefix sums, then the scatter), the
//                     CVs transposed to [C][candidate]
//   k_sel_leaders     leader clustering in candidate order: a candidate joins
//                     the first leader within the threshold, else it becomes a
//                     leader.  One trial of the threshold search is one
//                     thread-block cluster; the trials the search may ask for
//                     next run side by side in one launch
// The distance test decides integers, so it is taken in FP32 with explicitly
// rounded operations in a fixed order:
//   delta = a - b; periodic: delta -= 2 pi floor(delta / (2 pi) + 1/2);
//   d2 += w (delta delta); join iff d2 <= t^2 (t^2 rounded to FP32 once).
// The threshold search runs on the host (double), one clustering per trial.
#include <algorithm>
#include <cmath>
#include <vector>

#include "rid_internal.cuh"

namespace {

constexpr int SEL_T = 1024;
constexpr float SEL_TWO_PI = 6.28318530717959f;
constexpr float SEL_INV_2PI = 0.159154943091895f;

// Distance of the leader a [C] and the candidate whose CV c is at b[c * cap].
__device__ __forceinline__ float sel_d2(const float* a, const float* __restrict__ b, long long cap, const float* w,
                                        const int* per, int C) {
    float acc = 0.0f;
#pragma unroll 4
    for (int c = 0; c < C; ++c) {
        float d = __fsub_rn(a[c], __ldg(b + c * cap));
        if (per[c]) {
            const float k = floorf(__fadd_rn(__fmul_rn(d, SEL_INV_2PI), 0.5f));
            d = __fsub_rn(d, __fmul_rn(SEL_TWO_PI, k));
        }
        acc = __fadd_rn(acc, __fmul_rn(w[c], __fmul_rn(d, d)));
    }
    return acc;
}

// Exclusive block scan of counts over SEL_T threads; returns the prefix and
// writes the block total to *tot.
__device__ int block_excl_scan(int f, int* warp_sums, int* tot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int v = f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) warp_sums[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int s = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;   // inclusive over warps
        if (lane == 31) *tot = s;
    }
    __syncthreads();
    const int before = (wid ? warp_sums[wid - 1] : 0) + v - f;
    __syncthreads();
    return before;
}

// Trust window of one frame (compared in FP32, as eps is).
__device__ __forceinline__ int sel_in(const float* __restrict__ eps, int n, long long k, float lo, float hi) {
    return (k < n && eps[k] >= lo && eps[k] < hi) ? 1 : 0;
}

// Candidates in each block of SEL_T frames.
__global__ void __launch_bounds__(SEL_T) k_sel_count(const float* __restrict__ eps, int n, float lo, float hi,
                                                     int* __restrict__ blk) {
    const long long k = (long long)blockIdx.x * SEL_T + threadIdx.x;
    const int c = __syncthreads_count(sel_in(eps, n, k, lo, hi));
    if (threadIdx.x == 0) blk[blockIdx.x] = c;
}

// Exclusive prefix sums of blk[nb] in place; the total into *n_cand.  Clears
// the word that the trials of each later launch share.
constexpr int SEL_LAUNCHES = 66;   // 64 trials at most, then the clustering kept
__global__ void __launch_bounds__(SEL_T) k_sel_scan(int* __restrict__ blk, int nb, int* __restrict__ n_cand,
                                                    unsigned* __restrict__ out_words) {
    __shared__ int warp_sums[32];
    __shared__ int tot;
    int base = 0;
    if (threadIdx.x < SEL_LAUNCHES) out_words[threadIdx.x] = 0;
    for (int b0 = 0; b0 < nb; b0 += SEL_T) {
        const int b = b0 + threadIdx.x;
        const int v = b < nb ? blk[b] : 0;
        const int pos = block_excl_scan(v, warp_sums, &tot);
        if (b < nb) blk[b] = base + pos;
        base += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_cand = base;
}

// Candidate frame indices cand[pos] and their CVs x[c][pos] (row length cap):
// transposed, so that consecutive candidates are consecutive addresses in
// every distance.
__global__ void __launch_bounds__(SEL_T) k_sel_scatter(const float* __restrict__ cv, const float* __restrict__ eps,
                                                       int n, int C, float lo, float hi, const int* __restrict__ blk,
                                                       int* __restrict__ cand, float* __restrict__ x, long long cap) {
    __shared__ int warp_sums[32];
    __shared__ int tot;
    __shared__ int list[SEL_T];
    const long long k = (long long)blockIdx.x * SEL_T + threadIdx.x;
    const int base = blk[blockIdx.x];
    const int f = sel_in(eps, n, k, lo, hi);
    const int pos = block_excl_scan(f, warp_sums, &tot);
    if (f) {
        list[pos] = (int)k;
        cand[base + pos] = (int)k;
    }
    __syncthreads();
    const int m = tot;
    for (int e = threadIdx.x; e < m * C; e += SEL_T) {
        const int c = e / m, r = e - c * m;
        x[c * cap + base + r] = cv[(long long)list[r] * C + c];
    }
}

__device__ __forceinline__ uint32_t sel_peer(const void* local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(local))), "r"(rank));
    return r;
}
__device__ __forceinline__ void sel_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The trials of one launch: thresholds (squared, FP32), where a trial stops
// (0: runs to the end), its leader list at lead + trial * lcap, and the trials
// (bits) that the search no longer visits once this one has found more than
// `upper` clusters, fewer than `lower`, or a count between them.
constexpr int SEL_TRIALS = 7;
constexpr int SEL_CLUSTER = 16;
struct SelTrials {
    float t2[SEL_TRIALS];
    int stop, lower, upper;
    unsigned many_out[SEL_TRIALS], few_out[SEL_TRIALS], hit_out[SEL_TRIALS];
};

// One trial per cluster of P CTAs (CTAs trial * P ..).  Candidate k belongs to
// thread k mod (1024 P) of the cluster, which keeps one bit per candidate: not
// yet in a cluster.  A round takes the smallest such candidate of the whole
// cluster as the next leader (warp minimum, block minimum, one word per CTA
// through distributed shared memory, one cluster barrier) and every thread
// strikes its candidates within the threshold of it.  The smallest unassigned
// candidate is exactly the next one that the sequential rule makes a leader,
// and a candidate is struck by the first leader that covers it, so the leaders
// and their order are the sequential rule's.
// A round is bound by latency (the leader's CVs from L2, two block barriers and
// a cluster barrier), its distances being spread over 16 SMs.  102400 frames x
// 20 CVs searched into 30-45 clusters: 14.9 ms a call with one CTA settling
// 1024 candidates at a time and the trials one after another, 0.71 ms now.
// A trial that ends sets the bits of those it makes needless in *out, and these
// leave: the first CTA of a cluster reads the word every eighth round, uses it
// four rounds later (a read takes longer than a short round) and sends 0 in its
// next message, so that the cluster leaves together.  (Without it a
// search whose first trial is already in a wide window, 10 clusters in 1 to
// 20000, waited for trials that count to 20001: 48.9 ms at 102400 frames of 20
// CVs, 2.6 ms now, 25.8 ms with one trial at a time in one CTA.)
// Candidates past the first 32 of a thread keep their bits in alive_g
// [trial][word - 1][1024 P].
__global__ void __launch_bounds__(SEL_T) k_sel_leaders(const float* __restrict__ x, long long cap,
                                                       const int* __restrict__ n_cand_p, int C,
                                                       const float* __restrict__ w, const int* __restrict__ per,
                                                       SelTrials T, int P, int* __restrict__ lead, long long lcap,
                                                       int* __restrict__ n_lead, unsigned* out,
                                                       unsigned* __restrict__ alive_g, long long alive_stride) {
    __shared__ float lc[RID_MAX_CV], ws[RID_MAX_CV];
    __shared__ int ps[RID_MAX_CV];
    __shared__ unsigned wmin[32];
    __shared__ unsigned cmin[2][SEL_CLUSTER];
    constexpr unsigned NONE = 0xffffffffu;
    const int trial = blockIdx.x / P, rank = blockIdx.x - trial * P;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned n = (unsigned)*n_cand_p, G = (unsigned)P * SEL_T, g = (unsigned)rank * SEL_T + tid;
    const unsigned mine = g < n ? (n - g + G - 1) / G : 0;      // candidates of this thread
    const unsigned words = ((n + G - 1) / G + 31) / 32;         // the same for every thread
    const float t2 = T.t2[trial];
    unsigned* alive = alive_g + trial * alive_stride + g;
    if (tid < C) {
        ws[tid] = w[tid];
        ps[tid] = per[tid];
    }
    auto full_word = [&](unsigned q) {
        const unsigned left = mine > 32 * q ? mine - 32 * q : 0;
        return left >= 32 ? NONE : (1u << left) - 1u;
    };
    unsigned word0 = full_word(0);
    for (unsigned q = 1; q < words; ++q) alive[(long long)(q - 1) * G] = full_word(q);
    unsigned first = mine ? g + 1 : NONE;                       // 1 + this thread's smallest candidate left
    unsigned gone = 0, seen = 0;                                // *out, in the cluster's first thread
    int nl = 0, par = 0;
    // every CTA of the cluster runs before a peer writes to its shared memory
    if (P > 1) sel_cluster_sync();
    for (;;) {
        unsigned v = __reduce_min_sync(0xffffffffu, first);
        if (lane == 0) wmin[warp] = v;
        __syncthreads();
        if (warp == 0) {
            // the message: 1 + the candidate, NONE, or 0 to leave
            v = __reduce_min_sync(0xffffffffu, gone >> trial & 1u ? 0u : wmin[lane]);
            if (P == 1) {
                if (lane == 0) cmin[par][0] = v;
            } else if (lane < P) {
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(sel_peer(&cmin[par][rank], (uint32_t)lane)), "r"(v)
                             : "memory");
            }
        }
        if (P > 1) sel_cluster_sync();
        else __syncthreads();
        unsigned L = NONE;
        for (int q = 0; q < P; ++q) L = min(L, cmin[par][q]);
        par ^= 1;                     // this parity is written again only after the next barrier
        if (L == NONE) break;
        if (L == 0) return;           // the same in every thread of the cluster, after its barrier
        --L;
        if (rank == 0 && tid == 0 && nl < lcap) lead[trial * lcap + nl] = (int)L;
        ++nl;
        if (T.stop > 0 && nl > T.stop) break;
        if (tid < C) lc[tid] = x[tid * cap + L];
        __syncthreads();
        if (rank == 0 && tid == 0) {
            if (nl % 8 == 0) seen = *reinterpret_cast<const volatile unsigned*>(out);
            else if (nl % 8 == 4) gone = seen;
        }
        first = NONE;
        for (unsigned q = 0; q < words; ++q) {
            unsigned a = q == 0 ? word0 : alive[(long long)(q - 1) * G];
            const unsigned was = a;
            for (unsigned any = __reduce_or_sync(0xffffffffu, a); any; any &= any - 1) {
                const unsigned b = __ffs(any) - 1;
                if (!(a >> b & 1u)) continue;
                const unsigned k = g + G * (32 * q + b);
                if (k == L || sel_d2(lc, x + k, cap, ws, ps, C) <= t2) a &= ~(1u << b);
            }
            if (a && first == NONE) first = g + G * (32 * q + __ffs(a) - 1) + 1;
            if (q == 0) word0 = a;
            else if (a != was) alive[(long long)(q - 1) * G] = a;
        }
    }
    if (rank == 0 && tid == 0) {
        n_lead[trial] = nl;
        const unsigned rest = nl > T.upper ? T.many_out[trial] : nl < T.lower ? T.few_out[trial] : T.hit_out[trial];
        if (rest) atomicOr(out, rest);
    }
}

// selected[i] = frame index of leader i (leaders hold candidate rows)
__global__ void k_sel_map(const int* __restrict__ lead, const int* __restrict__ cand, int n, int* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = cand[lead[i]];
}

int sel_cuda(cudaError_t e, const char* what) {
    return rid_fail(RID_ERR_CUDA, "select: %s: %s", what, cudaGetErrorString(e));
}

struct SelBuf {
    void* p = nullptr;
    ~SelBuf() {
        if (p) cudaFree(p);
    }
};

}  // namespace

extern "C" RID_API int rid_select(const rid_select_desc* d, int32_t n, const float* cv, const float* eps,
                                  int32_t* selected, int32_t* n_selected, int32_t* n_clusters, double* threshold_out,
                                  int32_t mem, void* stream) {
    NvtxScope nvtx_("rid_select");
    if (!d || !cv || !eps) return rid_fail(RID_ERR_ARG, "select: NULL argument");
    if (mem != RID_MEM_HOST && mem != RID_MEM_DEVICE) return rid_fail(RID_ERR_ARG, "select: bad mem");
    const int C = d->n_cv;
    if (C < 1 || C > RID_MAX_CV || n < 0 || !(d->cluster_threshold > 0) || d->max_selection < 0 ||
        (d->max_selection > 0 && !selected) ||
        (d->adapt && (d->numb_cluster_lower < 1 || d->numb_cluster_upper < d->numb_cluster_lower)))
        return rid_fail(RID_ERR_ARG, "select: parameters out of range");
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<float> hw(C, 1.0f);
    std::vector<int> hp(C, 1);
    for (int c = 0; c < C; ++c) {
        if (d->weights) hw[c] = d->weights[c];
        if (d->periodic) hp[c] = d->periodic[c] != 0;
    }
    const long long nn = n > 0 ? n : 1;
    const int nb = (int)((nn + SEL_T - 1) / SEL_T);
    // One CTA up to 4096 frames, where a cluster's barrier costs more than its
    // SMs save; else a cluster of 16.
    const int P = nn <= 4 * SEL_T ? 1 : SEL_CLUSTER;
    const long long G = (long long)P * SEL_T;
    // Trials of a search run SEL_TRIALS to a launch; very long traces (where a
    // trial fills the launch's time by itself) keep the scratch of one.
    const int trials = d->adapt && nn <= (1 << 22) ? SEL_TRIALS : 1;
    // a trial of the search stops once its count passes `upper`
    const int upper = d->adapt ? d->numb_cluster_upper : 0;
    const long long lcap = d->adapt && upper < nn ? (long long)upper + 1 : nn;
    const long long nlead = std::max(nn, trials * lcap);   // the final clustering may need nn
    const long long awords = ((nn + G - 1) / G + 31) / 32 - 1;
    const long long ncv = mem == RID_MEM_HOST ? nn * C : 0, neps = mem == RID_MEM_HOST ? nn : 0;
    const size_t bytes = sizeof(float) * (size_t)(ncv + neps + nn * C + C) +
                         sizeof(int) * (size_t)(nn + nlead + nb + C + 1 + trials + SEL_LAUNCHES + trials * awords * G + nn);
    SelBuf buf;
    if (cudaMalloc(&buf.p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return rid_fail(RID_ERR_OOM, "select: device allocation of %zu bytes failed", bytes);
    }
    float* x = reinterpret_cast<float*>(buf.p);      // [C][nn] candidates
    float* dw = x + nn * C;
    float* hcv = dw + C;                             // host calls: the uploaded frames
    float* heps = hcv + ncv;
    int* cand = reinterpret_cast<int*>(heps + neps);
    int* lead = cand + nn;
    int* blk = lead + nlead;
    int* dper = blk + nb;
    int* dncand = dper + C;                          // then the leader counts of a launch's trials
    int* dnl = dncand + 1;
    unsigned* out_words = reinterpret_cast<unsigned*>(dnl + trials);   // one per launch
    unsigned* alive = out_words + SEL_LAUNCHES;
    int* dsel_buf = reinterpret_cast<int*>(alive + trials * awords * G);   // [nn] frame indices of the selection
    cudaError_t e;
    const float* dcv = cv;
    const float* deps = eps;
    if (mem == RID_MEM_HOST && n > 0) {
        if ((e = cudaMemcpyAsync(hcv, cv, sizeof(float) * (size_t)n * C, cudaMemcpyHostToDevice, st)) != cudaSuccess)
            return sel_cuda(e, "cv");
        if ((e = cudaMemcpyAsync(heps, eps, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, st)) != cudaSuccess)
            return sel_cuda(e, "eps");
        dcv = hcv;
        deps = heps;
    }
    if ((e = cudaMemcpyAsync(dw, hw.data(), sizeof(float) * C, cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return sel_cuda(e, "weights");
    if ((e = cudaMemcpyAsync(dper, hp.data(), sizeof(int) * C, cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return sel_cuda(e, "mask");
    // trust window: eps in [lo, hi), compared in FP32 (the eps values are FP32)
    const float lo = (float)d->trust_lo, hi = (float)d->trust_hi;
    k_sel_count<<<nb, SEL_T, 0, st>>>(deps, n, lo, hi, blk);
    k_sel_scan<<<1, SEL_T, 0, st>>>(blk, nb, dncand, out_words);
    k_sel_scatter<<<nb, SEL_T, 0, st>>>(dcv, deps, n, C, lo, hi, blk, cand, x, nn);
    static RidOnce once;
    if ((e = rid_on_device(once, [](int) {
             return cudaFuncSetAttribute(k_sel_leaders, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
         })) != cudaSuccess)
        return sel_cuda(e, "cluster size");
    int hn[1 + SEL_TRIALS] = {};
    // nt clusterings side by side; their counts into hn[1 ..], the candidate count into hn[0]
    int n_launch = 0;
    auto cluster = [&](SelTrials T, const double* t, int nt, int stop, long long cap_l) -> int {
        for (int k = 0; k < nt; ++k) T.t2[k] = (float)(t[k] * t[k]);
        T.stop = stop;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(nt * P), 1, 1);
        cfg.blockDim = dim3(SEL_T, 1, 1);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)P;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cudaError_t e2 = cudaLaunchKernelEx(&cfg, k_sel_leaders, (const float*)x, nn, (const int*)dncand, C,
                                            (const float*)dw, (const int*)dper, T, P, lead, cap_l, dnl,
                                            out_words + n_launch++, alive, awords * G);
        if (e2 != cudaSuccess) return sel_cuda(e2, "launch");
        if ((e2 = cudaMemcpyAsync(hn, dncand, sizeof(int) * (1 + nt), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
            return sel_cuda(e2, "count");
        if ((e2 = cudaStreamSynchronize(st)) != cudaSuccess) return sel_cuda(e2, "synchronize");
        return RID_OK;
    };
    double t = d->cluster_threshold;
    int count = 0;
    const int* leaders = lead;
    if (!d->adapt) {
        if (int rc = cluster({}, &t, 1, 0, lcap)) return rc;
        count = hn[1];
    } else {
        // The search: t doubles or halves until the count is bracketed, then
        // geometric bisection, 64 trials at most.  What a trial's outcome (too
        // many clusters or too few) makes of the bracket does not depend on its
        // count, so the next levels of that decision tree are known beforehand:
        // each launch runs the first `trials` nodes of the tree below the
        // current trial (three levels of seven) and the walk then follows the
        // counts, launching again where it leaves them.
        struct Node {
            double t, lo, hi;
            int many, few;
        };
        const int lower = d->numb_cluster_lower;
        auto step = [](const Node& a, bool many) {
            Node b{a.t, a.lo, a.hi, -1, -1};
            if (many) {
                b.lo = a.t;
                b.t = std::isinf(a.hi) ? 2.0 * a.t : std::sqrt(a.t * a.hi);
            } else {
                b.hi = a.t;
                b.t = a.lo == 0.0 ? 0.5 * a.t : std::sqrt(a.lo * a.t);
            }
            return b;
        };
        Node cur{t, 0.0, INFINITY, -1, -1};
        int it = 0, at = -1;
        bool done = false;
        while (!done) {
            Node tree[SEL_TRIALS];
            double tt[SEL_TRIALS];
            int nt = 0;
            tree[nt++] = cur;
            for (int k = 0; k < nt; ++k)
                for (int many = 1; many >= 0; --many)
                    if (nt < trials) {
                        (many ? tree[k].many : tree[k].few) = nt;
                        tree[nt++] = step(tree[k], many != 0);
                    }
            SelTrials T{};
            T.lower = lower;
            T.upper = upper;
            unsigned below[SEL_TRIALS];          // a node and all after it (children follow their parents)
            for (int k = nt - 1; k >= 0; --k) {
                T.few_out[k] = tree[k].many < 0 ? 0u : below[tree[k].many];
                T.many_out[k] = tree[k].few < 0 ? 0u : below[tree[k].few];
                T.hit_out[k] = T.few_out[k] | T.many_out[k];
                below[k] = 1u << k | T.hit_out[k];
                tt[k] = tree[k].t;
            }
            if (int rc = cluster(T, tt, nt, upper, lcap)) return rc;
            for (at = 0;;) {
                t = tree[at].t;
                count = hn[1 + at];
                if (hn[0] == 0 || (count >= lower && count <= upper) || it == 63) {
                    done = true;
                    break;
                }
                ++it;
                const bool many = count > upper;
                const int next = many ? tree[at].many : tree[at].few;
                if (next < 0) {
                    cur = step(tree[at], many);
                    break;
                }
                at = next;
            }
        }
        leaders = lead + at * lcap;
        if (count > upper) {   // the clustering finally kept had stopped early
            if (int rc = cluster({}, &t, 1, 0, nn)) return rc;
            count = hn[1];
            leaders = lead;
        }
    }
    const int nsel = count < d->max_selection ? count : d->max_selection;
    if (nsel > 0) {
        int* dsel = mem == RID_MEM_DEVICE ? selected : dsel_buf;
        k_sel_map<<<(nsel + 255) / 256, 256, 0, st>>>(leaders, cand, nsel, dsel);
        if ((e = cudaGetLastError()) != cudaSuccess) return sel_cuda(e, "map");
        if (mem == RID_MEM_HOST &&
            (e = cudaMemcpyAsync(selected, dsel, sizeof(int) * nsel, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
            return sel_cuda(e, "selected");
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return sel_cuda(e, "synchronize");
    }
    if (n_selected) *n_selected = nsel;
    if (n_clusters) *n_clusters = count;
    if (threshold_out) *threshold_out = t;
    return RID_OK;
}
