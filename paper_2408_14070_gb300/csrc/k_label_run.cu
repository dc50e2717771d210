// k_label_run.cu -- restrained label runs, one CTA per run with all of its
// steps in one launch: rid_label_batch for chains whose bonded slots fit in
// shared memory (RID_BONDED_SMEM_MAX beads), rid_label for chains below 768
// beads.
//
// The same step as k_label_fused, term for term and in the same order (so the
// same bits as there and as through the per-step kernels), arranged for the
// latency of one run.  The chain stays in shared memory; a step is two phases
// between block barriers:
//   beads   all threads, a bead each: bonded slots + LJ row + chain rule -> f,
//           closing B of the step before, B A O A of this one (Langevin noise
//           drawn beforehand), the cluster boxes by shuffles
//   terms   tasks that the warps take from a counter, the longest first: the
//           bonded terms of 32 beads (once per term, into shared slots), 32 CVs
//           with their restraint forces and label samples, the LJ rows of 32
//           beads over their neighbour lists (rebuilt by the same task when a
//           bead has moved half the skin), the noise of 32 beads' next step
// k_label_fused does these one after another on a thread per bead, with every
// angle evaluated by its three beads.
// Bound by latency: a step is two barriers and the longest task (a row's list,
// the bonded terms of 32 beads), 1.2 us of beads and 2 to 3 of terms at 200 beads,
// a rebuild every ten steps or so.  30 runs x 100 steps of 200 beads: 1.14 ms with
// k_label_fused, 0.58 now; 512 uneven runs of 50 to 500 beads x 250 steps, the
// call in C: 6.4 ms and 4.6 (k_label_fused's CTA size chosen by timing, the
// longest chain's shared memory for all).
#include <cmath>

#include "rid_batch.cuh"
#include "rid_forces.cuh"

namespace {

// 225 KB of the 227 a CTA may have: a few hundred bytes are static.
constexpr int RUN_SMEM_MAX = 225 * 1024;

// Shared memory of a chain of N beads and C CVs.
struct LrLayout {
    int N8, nclus;
    int NP, cap;                           // beads of a list row, longest list
    size_t xs, cbox, vs, fs, J, dsum, dsum2, dbp, zs, xr, fB, fA, fD, Fs, acv, off, over, nl, bytes;
};
__host__ __device__ inline LrLayout lr_layout(int N, int C) {
    LrLayout L{};
    L.nclus = (N + LJ_CLUSTER - 1) / LJ_CLUSTER;
    L.N8 = L.nclus * LJ_CLUSTER;
    size_t o = 0;
    L.xs = o;    o += 16 * (size_t)L.N8;
    L.cbox = o;  o += 32 * (size_t)L.nclus;
    L.vs = o;    o += 16 * (size_t)N;
    L.fs = o;    o += 16 * (size_t)N;
    L.J = o;     o += 64 * (size_t)C;
    L.dsum = o;  o += 8 * (size_t)C;
    L.dsum2 = o; o += 8 * (size_t)C;
    L.dbp = o;   o += 8 * (size_t)C;
    L.acv = o;   o += 8 * 4 * (size_t)C;
    L.zs = o;    o += 12 * (size_t)N;
    L.xr = o;    o += 12 * (size_t)N;
    L.fB = o;    o += 12 * (size_t)N;
    L.fA = o;    o += 36 * (size_t)N;
    L.fD = o;    o += 48 * (size_t)N;
    L.Fs = o;    o += 4 * (size_t)C;
    L.off = o;   o += 4 * (size_t)(N + 1);
    L.over = o;  o += 4 * (size_t)((N + 31) / 32);
    L.NP = (N + 1) / 2 * 2;
    // collapsed chains reach 50 beads within 1.2 rc (with 32 to 40 entries, the rows that
    // overflowed set the step: 30 runs of 200 beads 12 us a step, 5.7 with 64); the longest
    // chains keep what there is room for, 16 at least
    L.nl = o;
    const size_t room = o < (size_t)RUN_SMEM_MAX ? ((size_t)RUN_SMEM_MAX - o) / (2 * (size_t)L.NP) : 0;
    L.cap = room > 65 ? 64 : room > 17 ? (int)room - 1 : 16;
    o += 2 * (size_t)L.NP * (L.cap + 1);
    L.bytes = (o + 15) & ~(size_t)15;
    return L;
}

// Block of label sample k (of K) among B blocks.
__device__ __forceinline__ int lr_block(long long k, int B, long long K) { return (int)((k * B) / K); }

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_label_run(FusedArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ FusedJob J;
    __shared__ int s_item, s_task;
    __shared__ unsigned keep_s[NT / 32][(RID_BONDED_SMEM_MAX / LJ_CLUSTER + 31) / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(A.next, 1);
        __syncthreads();
        if (tid == 0 && s_item < A.n_items) J = A.jobs[A.items[s_item].job];
        __syncthreads();
        const int it = s_item;
        if (it >= A.n_items) break;
        const int r = A.items[it].run;
        const SysDev& S = J.S;
        const int N = S.N, C = S.C;
        const LrLayout L = lr_layout(N, C);
        float4* xs = reinterpret_cast<float4*>(smem + L.xs);
        float4* cbox = reinterpret_cast<float4*>(smem + L.cbox);
        float4* vs = reinterpret_cast<float4*>(smem + L.vs);
        float4* fs = reinterpret_cast<float4*>(smem + L.fs);   // LJ row sums, at the end of a launch the force
        float4* Jm = reinterpret_cast<float4*>(smem + L.J);
        double* lsum = reinterpret_cast<double*>(smem + L.dsum);
        double* lsum2 = reinterpret_cast<double*>(smem + L.dsum2);
        double* lbp = reinterpret_cast<double*>(smem + L.dbp);
        int2* acv = reinterpret_cast<int2*>(smem + L.acv);
        float3* zs = reinterpret_cast<float3*>(smem + L.zs);
        float3* fB = reinterpret_cast<float3*>(smem + L.fB);
        float3* fA = reinterpret_cast<float3*>(smem + L.fA);
        float3* fD = reinterpret_cast<float3*>(smem + L.fD);
        float* Fs = reinterpret_cast<float*>(smem + L.Fs);
        int* off = reinterpret_cast<int*>(smem + L.off);
        float3* xr = reinterpret_cast<float3*>(smem + L.xr);   // positions of the neighbour lists
        int* over = reinterpret_cast<int*>(smem + L.over);
        unsigned short* nl = reinterpret_cast<unsigned short*>(smem + L.nl);
        const long long base = (long long)r * N;
        const float kick = S.half_dt * S.inv_mass;
        const float lj_s = -S.lj_eps24;
        const bool sig1 = S.sig2 == 1.0f;
        const long long t0 = J.t0, t1 = J.t1;
        const int nb = (N + 31) / 32, nc = (C + 31) / 32;
        const int ntask = 3 * nb + nc;
        int bad = 0;

        // ---- stage the run
        for (int i = tid; i < L.N8; i += NT) {
            if (i < N) {
                xs[i] = J.x[base + i];
                if (J.init && J.mb) {
                    const float3 z = rid_normals3(rid_philox(make_uint4(i, r, J.step0, 1u), S.key0, S.key1));
                    vs[i] = make_float4(S.sd_mb * z.x, S.sd_mb * z.y, S.sd_mb * z.z, 0.0f);
                } else {
                    vs[i] = J.v[base + i];
                }
                if (!J.init) fs[i] = J.f[base + i];
            } else {
                xs[i] = make_float4(1.0e30f, 1.0e30f, 1.0e30f, 0.0f);
            }
        }
        for (int i = tid; i <= N; i += NT) off[i] = S.acv_off[i];
        for (int i = tid; i < 4 * C; i += NT) acv[i] = S.acv[i];
        // block of the last sample before step t (block 0 before the first)
        auto block_before = [&](long long t) {
            const long long k = t - 1 - J.n_equil;
            return k >= 0 ? lr_block(k, J.B, J.K) : 0;
        };
        // label accumulators; lbp holds the partial sum of the current block
        for (int j = tid; j < C; j += NT) {
            const long long o = (long long)r * C + j;
            lsum[j] = J.sum[o];
            lsum2[j] = J.sum2[o];
            lbp[j] = J.bsum[o * J.B + block_before(t0)];
        }
        auto noise = [&](long long t, int i) {
            if (i < N && S.c2 != 0.0f)
                zs[i] = rid_normals3(rid_philox(make_uint4(i, r, J.step0 + (uint32_t)t, 0u), S.key0, S.key1));
        };
        // (a launch that resumes a run starts from the stored force)
        if (!J.init)
            for (int i = tid; i < N; i += NT) noise(t0, i);
        if (tid == 0) s_task = 0;
        __syncthreads();

        // Terms at the current positions: bonded slots, CVs with restraint forces
        // and the label sample of step ts (ts < n_equil: none), LJ rows into fs; the
        // noise of step ts + 1.
        auto terms = [&](long long ts, bool build) {
            for (;;) {
                int k = 0;
                if (lane == 0) k = atomicAdd(&s_task, 1);
                k = __shfl_sync(0xffffffffu, k, 0);
                if (k >= ntask) break;
                if (k < nb) {
                    const int t = 32 * k + lane;
                    if (t < N) bonded_terms_to_smem(S, xs, t, fB, fA, fD);
                } else if ((k -= nb) < nc) {
                    const int j = 32 * k + lane;
                    if (j < C) {
                        const int4 q = S.cv[j];
                        float3 g[4];
                        const float sj = rid_cv(q, xs, g);
#pragma unroll
                        for (int a = 0; a < 4; ++a) Jm[4 * j + a] = make_float4(g[a].x, g[a].y, g[a].z, 0.0f);
                        const long long o = (long long)r * C + j;
                        const double d = rid_cv_offset(q, (double)sj, J.s0[o]);
                        Fs[j] = (float)(-J.kappa[o] * d);
                        if (ts >= J.n_equil) {
                            const int b = lr_block(ts - J.n_equil, J.B, J.K), b0 = block_before(ts);
                            if (b != b0) {
                                J.bsum[o * J.B + b0] = lbp[j];
                                lbp[j] = 0.0;
                            }
                            lsum[j] += d;
                            lsum2[j] = fma(d, d, lsum2[j]);
                            lbp[j] += d;
                        }
                    }
                } else if ((k -= nc) < nb) {
                    const int i = 32 * k + lane;
                    float fx = 0.f, fy = 0.f, fz = 0.f;
                    if (build) {
                        lj_list_build(S, xs, cbox, L.nclus, 32 * k, nl, L.NP, L.cap, over);
                        if (i < N) xr[i] = f3(xs[i]);
                    }
                    if (over[k]) {
                        float el = 0.f;
                        const float3 xi = f3(xs[i < N ? i : N - 1]);
                        lj_warp_keep_masks(S, cbox, L.nclus, xi, keep_s[warp]);
                        const int b0 = max(32 * k - 2, 0) / LJ_CLUSTER, b1 = min(32 * k + 33, N - 1) / LJ_CLUSTER;
                        const int nwords = (L.nclus + 31) / 32;
                        if (sig1) lj_row_culled<true, false, true>(S, xs, cbox, keep_s[warp], nwords, xi, i, b0, b1, fx, fy, fz, el);
                        else lj_row_culled<false, false, true>(S, xs, cbox, keep_s[warp], nwords, xi, i, b0, b1, fx, fy, fz, el);
                        __syncwarp();
                    } else if (sig1) {
                        lj_list_row<true>(S, xs, nl, L.NP, i, fx, fy, fz);
                    } else {
                        lj_list_row<false>(S, xs, nl, L.NP, i, fx, fy, fz);
                    }
                    if (i < N) fs[i] = make_float4(fx, fy, fz, 0.0f);
                } else if (ts + 1 < t1) {
                    noise(ts + 1, 32 * (k - nb) + lane);
                }
            }
            __syncthreads();
        };
        // The force on bead i from the terms.
        auto force = [&](int i) {
            const float3 fb = bonded_gather(S, i, fB, fA, fD);
            const float4 lj = fs[i];
            float4 f = make_float4(fmaf(lj_s, lj.x, fb.x), fmaf(lj_s, lj.y, fb.y), fmaf(lj_s, lj.z, fb.z), 0.0f);
            for (int e = off[i]; e < off[i + 1]; ++e) {
                const int2 ja = acv[e];
                const float4 g = Jm[4 * ja.x + ja.y];
                const float fsj = Fs[ja.x];
                f.x = fmaf(fsj, g.x, f.x);
                f.y = fmaf(fsj, g.y, f.y);
                f.z = fmaf(fsj, g.z, f.z);
            }
            bad |= !(isfinite(f.x) && isfinite(f.y) && isfinite(f.z));
            return f;
        };
        // The closing kick of a step.
        auto close = [&](float4& v, const float4& f) {
            v.x = fmaf(kick, f.x, v.x);
            v.y = fmaf(kick, f.y, v.y);
            v.z = fmaf(kick, f.z, v.z);
            bad |= !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z));
        };

        if (J.init) {                      // t0 = 0: the force at x0, no sample, the noise of step 0
            for (int w0 = 32 * warp; w0 < N; w0 += NT) {
                const int i = w0 + lane;
                lj_lane_boxes(f3(xs[i < N ? i : N - 1]), i < N, i, cbox);
            }
            __syncthreads();
            terms(-1, true);
        }
        for (long long t = t0; t < t1; ++t) {
            if (tid == 0) s_task = 0;
            int moved = t == t0 && !J.init;    // (a launch that resumes a run has no lists yet)
            for (int w0 = 32 * warp; w0 < N; w0 += NT) {
                const int i = w0 + lane;
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < N) {
                    x = xs[i];
                    float4 v = vs[i];
                    const float4 f = (t == t0 && !J.init) ? fs[i] : force(i);
                    if (t > t0) close(v, f);                    // B of step t - 1
                    v.x = fmaf(kick, f.x, v.x);                 // B
                    v.y = fmaf(kick, f.y, v.y);
                    v.z = fmaf(kick, f.z, v.z);
                    x.x = fmaf(S.half_dt, v.x, x.x);            // A
                    x.y = fmaf(S.half_dt, v.y, x.y);
                    x.z = fmaf(S.half_dt, v.z, x.z);
                    if (S.c2 != 0.0f) {                         // O
                        const float3 z = zs[i];
                        v.x = fmaf(S.c1, v.x, S.c2 * z.x);
                        v.y = fmaf(S.c1, v.y, S.c2 * z.y);
                        v.z = fmaf(S.c1, v.z, S.c2 * z.z);
                    }
                    x.x = fmaf(S.half_dt, v.x, x.x);            // A
                    x.y = fmaf(S.half_dt, v.y, x.y);
                    x.z = fmaf(S.half_dt, v.z, x.z);
                    xs[i] = make_float4(x.x, x.y, x.z, 0.0f);
                    vs[i] = v;
                    if (!moved) {
                        const float3 d = f3(x) - xr[i];
                        moved = !(dot3(d, d) <= LJ_MOVED2 * S.rc2);
                    }
                }
                lj_lane_boxes(f3(x), i < N, i, cbox);
            }
            terms(t, __syncthreads_or(moved));
        }

        // ---- the last closing kick, and the run back to memory
        for (int i = tid; i < N; i += NT) {
            const float4 f = (t0 == t1 && !J.init) ? fs[i] : force(i);
            float4 v = vs[i];
            if (t1 > t0) close(v, f);
            J.x[base + i] = xs[i];
            J.v[base + i] = v;
            J.f[base + i] = f;
        }
        const int last_b = block_before(t1);
        for (int j = tid; j < C; j += NT) {
            const long long o = (long long)r * C + j;
            J.sum[o] = lsum[j];
            J.sum2[o] = lsum2[j];
            J.bsum[o * J.B + last_b] = lbp[j];
            if (t1 == J.n_steps)
                label_stats(J.sum + o, J.sum2 + o, J.bsum + o * J.B, J.kappa[o], J.K, J.B, J.mf[o], J.se[o], J.sd[o]);
        }
        bad = __syncthreads_or(bad);
        if (tid == 0 && bad) J.flags[r] = 1;
        __syncthreads();   // J and s_item are rewritten by the next item
    }
}

// Runs that an SM holds at once.
template <int NT>
cudaError_t runs_per_sm(size_t smem, int& occ) {
    static RidOnce once;
    cudaError_t e = rid_opt_in(once, RUN_SMEM_MAX, k_label_run<NT>);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_label_run<NT>, NT, smem);
    return e;
}

template <int NT>
cudaError_t launch_run(const FusedArgs& A, int n_sm, size_t smem, cudaStream_t s) {
    int occ = 0;
    if (const cudaError_t e = runs_per_sm<NT>(smem, occ)) return e;
    const long long most = (long long)(occ > 0 ? occ : 1) * n_sm;
    k_label_run<NT><<<(unsigned)(A.n_items < most ? A.n_items : most), NT, smem, s>>>(A);
    return cudaGetLastError();
}

}  // namespace

size_t rid_label_run_smem(int N, int C) {
    const size_t b = N <= RID_BONDED_SMEM_MAX ? lr_layout(N, C).bytes : 0;
    return b <= (size_t)RUN_SMEM_MAX ? b : 0;
}

// The sizes' times of a wave, in twentieths of the largest's, are those of 80 to 200 beads with every SM full
// (60 steps of 80 beads, us: 445 for 2 runs an SM at 512 threads, 559 for 4 at 256, 886 for 8 at 128).  By chain
// length alone -> with the runs, the call's time (and through k_label_fused): 1216 runs of 66 beads 1230 -> 716 us
// (1061), 4096 of 80 beads 3773 -> 2323 (3570), 1024 of 200 beads 1547 -> 1512 (2280).  608 of 200 beads stay
// at 512 threads (1056 us, 1128 at 256).
int rid_label_run_threads(int N, size_t smem, double runs, int n_sm) {
    const int most = N <= 32 ? 128 : N <= 64 ? 256 : 512;
    int best = most;
    double cost = INFINITY;
    for (int nt = most; nt >= 128; nt /= 2) {
        int occ = 0;
        const cudaError_t e = nt == 512 ? runs_per_sm<512>(smem, occ) : nt == 256 ? runs_per_sm<256>(smem, occ)
                                                                                  : runs_per_sm<128>(smem, occ);
        if (e != cudaSuccess || occ < 1) continue;
        const double waves = std::ceil(runs / ((double)occ * n_sm));
        const double c = waves * (nt == 512 ? 20.0 : nt == 256 ? 25.0 : 39.0);
        if (c < cost) {
            cost = c;
            best = nt;
        }
        if (waves <= 1.0) break;   // a smaller size takes longer
    }
    return best;
}

cudaError_t rid_launch_label_run(const FusedArgs& A, int threads, int n_sm, size_t smem, cudaStream_t s) {
    switch (threads) {
        case 128: return launch_run<128>(A, n_sm, smem, s);
        case 256: return launch_run<256>(A, n_sm, smem, s);
        case 512: return launch_run<512>(A, n_sm, smem, s);
        default: return cudaErrorInvalidValue;
    }
}
