// rid_gemm.cuh -- the batched FP32 GEMMs with fused per-pass epilogues of the
// training chain (k_train.cu).  Members of the ensemble run on grid z;
// activations are [M][rows][ld] row-major and weights [rows][ld] with ld a
// multiple of 4 floats and 16-byte aligned starts, zero past the columns.
#pragma once

#include "rid_internal.cuh"

namespace {

enum Epi { EPI_FWD = 1, EPI_BWD = 2, EPI_ADJ = 3, EPI_BACK = 4, EPI_LOSS = 5 };

// C[i][j] = sum_k A(i, k) B(k, j) of member z (member offsets z * sm): A
// row-major along K; B the rows j of W (K contiguous: forward, adjoint) or the
// rows k of W (columns contiguous: input gradient, back).
struct GemmArgs {
    const float* A;
    long long a_sm;
    int lda;
    const float* B;
    long long b_sm;
    int ldb;
    int K, rows, cols;
};

// What the epilogues read and write, [M][rows][ld] with member stride sm
// unless said otherwise.
struct EpiArgs {
    int ld;
    long long sm;
    // forward: bias b_l, T_l out, h_l out, h_{l-1} in (residual), w_out (last layer: G, D out)
    const float* bias; const float* wout; long long w_sm;
    float* T; float* Hout; const float* Hin;
    float* Gout; float* Dout;
    // backward / adjoint / back: residual input, T of the layer, second outputs
    float* out; const float* res; const float* Tl; const float* Gl; float* out2; const float* tb; float* out3;
    // dropout scales dq of the layer whose tanh the epilogue forms or reads
    // (forward, adjoint: layer l; backward, back: layer l - 1); NULL: dq = 1
    const float* Q;
    int resid;         // r_l
    int last;          // forward / adjoint on the last layer
    // loss (input gradient of layer 0): inputs u, labels and residuals [M][rows][C]
    const float* U; const float* MF; float* R; const int* dist;
    float scale;       // 2 / (rows C)
};

__device__ __forceinline__ void cp_async4(float* dst, const float* src, int src_bytes) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
// 16-byte copy global -> shared, past src_bytes zeros.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int src_bytes) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// At most n (0..7) of this thread's copy groups in flight.
__device__ __forceinline__ void cp_async_wait_n(int n) {
    switch (n) {
        case 0: cp_async_wait<0>(); break;
        case 1: cp_async_wait<1>(); break;
        case 2: cp_async_wait<2>(); break;
        case 3: cp_async_wait<3>(); break;
        case 4: cp_async_wait<4>(); break;
        case 5: cp_async_wait<5>(); break;
        case 6: cp_async_wait<6>(); break;
        default: cp_async_wait<7>(); break;
    }
}
// Bytes of a 4-float copy of which `left` floats exist.
__device__ __forceinline__ int bytes4(int left) { return left <= 0 ? 0 : (left >= 4 ? 16 : 4 * left); }

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may be scheduled before its predecessor on the stream has
// finished; pdl_wait() returns once the predecessor has completed and its
// memory is visible (at once for a normal launch).  pdl_trigger() lets the
// next such kernel be scheduled.  The GEMMs trigger after their K loop, so at
// most the next grid waits resident during their epilogue (a trigger at kernel
// entry let the whole chain of grids sit resident: 244 -> 327 us a step).
// A GEMM reads its weights before pdl_wait(): they were last written by the
// update of the step before, which the batch gather waits for before it
// triggers, and no kernel of the chain starts before its predecessor's trigger.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Launch with programmatic stream serialization when pdl is set.
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                     Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// The epilogue's inputs for output (i, j), loaded before the sums are ready.
// (__ldcg: written by kernels this one may overlap with.)
struct EpiIn {
    float a, b, c, d;
};
template <int EPI>
__device__ __forceinline__ EpiIn epi_load(const EpiArgs& e, int z, int i, int j) {
    const long long o = (long long)z * e.sm + (long long)i * e.ld + j;
    EpiIn v{0.0f, 0.0f, 0.0f, 0.0f};
    if (EPI == EPI_FWD) {
        v.a = __ldcg(e.bias + (long long)z * e.w_sm + j);
        v.b = e.Q ? __ldcg(e.Q + o) : 1.0f;
        if (e.resid) v.c = __ldcg(e.Hin + o);
        if (e.last) v.d = __ldcg(e.wout + (long long)z * e.w_sm + j);
    } else if (EPI == EPI_BWD || EPI == EPI_BACK) {
        if (e.resid) v.a = __ldcg(e.res + o);
        if (e.Tl) v.b = __ldcg(e.Tl + o);
        v.c = e.Q ? __ldcg(e.Q + o) : 1.0f;
        if (EPI == EPI_BACK) v.d = __ldcg(e.tb + o);
    } else if (EPI == EPI_ADJ) {
        v.a = __ldcg(e.Tl + o);
        v.b = e.Q ? __ldcg(e.Q + o) : 1.0f;
        v.c = __ldcg(e.Gl + o);
        if (e.resid) v.d = __ldcg(e.res + o);
    }
    return v;
}
template <int EPI>
__device__ __forceinline__ void epi_store(const EpiArgs& e, int z, int i, int j, float a, const EpiIn& v) {
    const long long o = (long long)z * e.sm + (long long)i * e.ld + j;
    if (EPI == EPI_FWD) {
        // t_l = tanh(z_l); h_l = dq t_l + r h_{l-1}; last: g = w_out, d = g dq (1 - t^2)
        const float t = tanhf(a + v.a), dq = v.b;
        e.T[o] = t;
        if (e.Hout != e.T) e.Hout[o] = e.resid ? fmaf(dq, t, v.c) : dq * t;
        if (e.last) {
            e.Gout[o] = v.d;
            e.Dout[o] = v.d * (dq * (1.0f - t * t));
        }
    } else if (EPI == EPI_BWD) {
        // g_{l-1} = d_l W_l + r_l g_l; d_{l-1} = g_{l-1} dq (1 - t_{l-1}^2)
        const float gv = e.resid ? a + v.a : a;
        e.out[o] = gv;
        if (e.Dout) e.Dout[o] = gv * (v.c * (1.0f - v.b * v.b));
    } else if (EPI == EPI_ADJ) {
        // dbar = acc; gbar_l = dbar dq (1 - t^2) + r gbar_{l-1}; tbar = -2 dq t g dbar
        const float t = v.a, dq = v.b;
        const float sp = 1.0f - t * t, spq = dq * sp;
        e.out[o] = e.resid ? a * spq + v.d : a * spq;
        const float tb = -2.0f * (dq * t) * v.c * a;
        e.out2[o] = tb;
        if (e.last) e.out3[o] = tb * sp;      // zbar_{L-1} (hbar_{L-1} = 0)
    } else if (EPI == EPI_BACK) {
        // hbar_{l-1} = zbar_l W_l + r hbar_l; zbar_{l-1} = (tbar + dq hbar)(1 - t^2)
        const float hb = e.resid ? a + v.a : a;
        e.out[o] = hb;
        e.out3[o] = fmaf(v.c, hb, v.d) * (1.0f - v.b * v.b);
    }
}

// Residual of one (sample, CV) and the loss's adjoint gbar_{-1} = d loss /
// d(dA/du), from g_{-1} = (g0, g1) of its input pair.  cs, sn: the pair u.
__device__ __forceinline__ void epi_loss(const EpiArgs& e, int z, int i, int c, int C, int rows, float g0, float g1,
                                         float cs, float sn, float mf) {
    // a distance CV (input (s, 0)): dA/ds = dA/du_2j; a torsion: through (cos, sin)
    const bool dj = e.dist && e.dist[c];
    const float dads = dj ? g0 : fmaf(cs, g1, -sn * g0);
    const float r = dads - mf;
    e.R[((long long)z * rows + i) * C + c] = r;
    const float v = e.scale * r;
    float* gb = e.out + (long long)z * e.sm + (long long)i * e.ld + 2 * c;
    gb[0] = dj ? v : -sn * v;
    gb[1] = dj ? 0.0f : cs * v;
}

// One 32 x 32 output tile per CTA, all of K (at most 512) resident: at the
// training sizes (128 rows, 256 columns, 4 members: 128 CTAs) a pass is a chain
// of latencies, so the weights are fetched before the wait on the predecessor
// (see pdl_wait), the activations all at once behind it in chunks of 64 K, and
// the epilogue's inputs beside them.  256 threads in two K groups of 128: group
// q multiplies the K tiles of 32 with index q, q + 2, .., each output in
// increasing k, and the two sums are added in group order (each group finishes
// one of a thread's two rows).  KB: B is K contiguous (a thread's columns tx +
// 8 q), else column contiguous (4 tx + q).
// A step of 4 members 40-256x4-1, 128 rows each, dropout 0.1: 233 us with 4-byte
// copies through a ring behind the wait and the loss, column sums and Adam in
// launches of their own, 125 us now (calls of 20 steps).
constexpr int TT = 256;
constexpr int TBP = 36;    // row pitch of a column-contiguous B
__host__ __device__ inline size_t tile_floats(int K, bool KB) {
    const int Kr = (K + 31) / 32 * 32;
    return (size_t)32 * (Kr + 4) + (KB ? (size_t)32 * (Kr + 4) : (size_t)Kr * TBP) + 8 * 128;
}
template <int EPI, bool KB>
__global__ void __launch_bounds__(TT) k_tr_tile(GemmArgs g, EpiArgs e) {
    extern __shared__ __align__(16) float gsm[];
    const int z = blockIdx.z, i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    const int K = g.K, Kr = (K + 31) / 32 * 32, LDK = Kr + 4;
    float* As = gsm;                                 // [32][LDK]
    float* Bs = As + 32 * LDK;                       // KB: [32][LDK], else [Kr][TBP]
    float* red = Bs + (KB ? 32 * LDK : Kr * TBP);    // [2][4][128]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = tid >> 7, gt = tid & 127, tx = gt & 7, ty = gt >> 3;   // rows 2 ty, 2 ty + 1
    {
        const float* pb = g.B + (long long)z * g.b_sm;
        if (KB) {
            for (int j = warp; j < 32; j += 8)
                for (int k = 4 * lane; k < Kr; k += 128) {
                    const int left = j0 + j < g.cols ? K - k : 0;
                    cp_async16(Bs + j * LDK + k, left > 0 ? pb + (long long)(j0 + j) * g.ldb + k : pb, bytes4(left));
                }
        } else {
            for (int q = tid; q < Kr * 8; q += TT) {
                const int k = q >> 3, c = 4 * (q & 7);
                const int left = k < K ? g.cols - (j0 + c) : 0;
                cp_async16(Bs + k * TBP + c, left > 0 ? pb + (long long)k * g.ldb + j0 + c : pb, bytes4(left));
            }
        }
        cp_async_commit();
    }
    pdl_wait();
    const int nr = (K + 63) / 64;                    // at most 8
    {
        const float* pa = g.A + (long long)z * g.a_sm;
        for (int c = 0; c < nr; ++c) {
            for (int q = tid; q < 32 * 16; q += TT) {
                const int i = q >> 4, k = 64 * c + 4 * (q & 15);
                if (k < Kr) {
                    const int left = i0 + i < g.rows ? K - k : 0;
                    cp_async16(As + i * LDK + k, left > 0 ? pa + (long long)(i0 + i) * g.lda + k : pa, bytes4(left));
                }
            }
            cp_async_commit();
        }
    }
    // this thread finishes row 2 ty + grp
    const int row = i0 + 2 * ty + grp;
    int col[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) col[q] = j0 + (KB ? tx + 8 * q : 4 * tx + q);
    EpiIn in[4];
    float u[4], mf[2];                               // EPI_LOSS: the pairs' inputs and labels
    const int C = g.cols >> 1;
    if (EPI == EPI_LOSS) {
        if (row < g.rows) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                u[q] = col[q] < g.cols ? __ldcg(e.U + (long long)z * e.sm + (long long)row * e.ld + col[q]) : 0.0f;
#pragma unroll
            for (int q = 0; q < 2; ++q)
                mf[q] = col[2 * q] < g.cols ? __ldcg(e.MF + ((long long)z * g.rows + row) * C + (col[2 * q] >> 1)) : 0.0f;
        }
    } else if (row < g.rows) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (col[q] < g.cols) in[q] = epi_load<EPI>(e, z, row, col[q]);
    }
    float acc[2][4] = {};
    for (int c = 0; c < nr; ++c) {
        cp_async_wait_n(nr - 1 - c);
        __syncthreads();
        const int k0 = 64 * c + 32 * grp;
        if (k0 < K) {
            const float* a0 = As + (2 * ty) * LDK + k0;
#pragma unroll
            for (int kk = 0; kk < 32; kk += 4) {
                const float4 av0 = *reinterpret_cast<const float4*>(a0 + kk);
                const float4 av1 = *reinterpret_cast<const float4*>(a0 + LDK + kk);
                const float x0[4] = {av0.x, av0.y, av0.z, av0.w}, x1[4] = {av1.x, av1.y, av1.z, av1.w};
                if (KB) {
                    float y[4][4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 b = *reinterpret_cast<const float4*>(Bs + (tx + 8 * q) * LDK + k0 + kk);
                        y[q][0] = b.x, y[q][1] = b.y, y[q][2] = b.z, y[q][3] = b.w;
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            acc[0][q] = fmaf(x0[s], y[q][s], acc[0][q]);
                            acc[1][q] = fmaf(x1[s], y[q][s], acc[1][q]);
                        }
                } else {
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const float4 b = *reinterpret_cast<const float4*>(Bs + (k0 + kk + s) * TBP + 4 * tx);
                        const float y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            acc[0][q] = fmaf(x0[s], y[q], acc[0][q]);
                            acc[1][q] = fmaf(x1[s], y[q], acc[1][q]);
                        }
                    }
                }
            }
        }
    }
    pdl_trigger();                     // the next kernel may be scheduled during the epilogue
#pragma unroll
    for (int q = 0; q < 4; ++q) red[(grp * 4 + q) * 128 + gt] = grp ? acc[0][q] : acc[1][q];
    __syncthreads();
    float sum[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float other = red[((grp ^ 1) * 4 + q) * 128 + gt];
        sum[q] = grp ? other + acc[1][q] : acc[0][q] + other;
    }
    if (row >= g.rows) return;
    if (EPI == EPI_LOSS) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (col[2 * q] < g.cols)
                epi_loss(e, z, row, col[2 * q] >> 1, C, g.rows, sum[2 * q], sum[2 * q + 1], u[2 * q], u[2 * q + 1], mf[q]);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (col[q] < g.cols) epi_store<EPI>(e, z, row, col[q], sum[q], in[q]);
    }
}

// Large batches (from 1024 rows, 64 columns): 64 x 64 tiles of 256 threads (4 x
// 4 outputs), K tiles of 32 through a ring of shared-memory stages, every output
// one chain over increasing k.
constexpr int GK = 32, BT = 64, BLD = BT + 4, BNS = 3;
constexpr size_t BIG_SMEM = sizeof(float) * 2 * BNS * GK * BLD;
template <int EPI, bool KB>
__global__ void __launch_bounds__(TT) k_tr_big(GemmArgs g, EpiArgs e) {
    extern __shared__ __align__(16) float gsm[];
    pdl_wait();
    float* As = gsm;                     // [BNS][GK][BLD]
    float* Bs = gsm + BNS * GK * BLD;
    const int z = blockIdx.z, i0 = blockIdx.y * BT, j0 = blockIdx.x * BT;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[4][4] = {};
    const int nt = (g.K + GK - 1) / GK;
    const float* pa = g.A + (long long)z * g.a_sm;
    const float* pb = g.B + (long long)z * g.b_sm;
    auto issue_tile = [&](int t) {
        if (t < nt) {
            const int k0 = t * GK;
            float* as = As + (t % BNS) * GK * BLD;
            float* bs = Bs + (t % BNS) * GK * BLD;
#pragma unroll
            for (int r = 0; r < BT * GK / TT; ++r) {
                const int idx = tid + TT * r;
                const int ii = idx / GK, kk = idx % GK, gi = i0 + ii, gk = k0 + kk;
                const bool ia = gi < g.rows && gk < g.K;
                cp_async4(as + kk * BLD + ii, ia ? pa + (long long)gi * g.lda + gk : pa, ia ? 4 : 0);
                const int jj = KB ? idx / GK : idx % BT, kb = KB ? idx % GK : idx / BT;
                const int gj = j0 + jj, gkb = k0 + kb;
                const bool ib = gj < g.cols && gkb < g.K;
                cp_async4(bs + kb * BLD + jj,
                          ib ? pb + (KB ? (long long)gj * g.ldb + gkb : (long long)gkb * g.ldb + gj) : pb, ib ? 4 : 0);
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int t = 0; t < BNS - 1; ++t) issue_tile(t);
    for (int t = 0; t < nt; ++t) {
        cp_async_wait<BNS - 2>();      // this thread's copies of tile t have landed
        __syncthreads();               // everyone's have, and everyone is done with tile t - 1
        issue_tile(t + BNS - 1);
        const float* as = As + (t % BNS) * GK * BLD;
        const float* bs = Bs + (t % BNS) * GK * BLD;
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            const float4 a = *reinterpret_cast<const float4*>(&as[kk * BLD + 4 * ty]);
            const float4 b = *reinterpret_cast<const float4*>(&bs[kk * BLD + 4 * tx]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
        }
    }
    pdl_trigger();
    cp_async_wait<0>();
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int i = i0 + 4 * ty + p;
        if (i >= g.rows) continue;
        if (EPI == EPI_LOSS) {
            const int C = g.cols >> 1;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int j = j0 + 4 * tx + 2 * q;
                if (j >= g.cols) continue;
                const float* up = e.U + (long long)z * e.sm + (long long)i * e.ld + j;
                epi_loss(e, z, i, j >> 1, C, g.rows, acc[p][2 * q], acc[p][2 * q + 1], __ldcg(up), __ldcg(up + 1),
                         __ldcg(e.MF + ((long long)z * g.rows + i) * C + (j >> 1)));
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + 4 * tx + q;
                if (j < g.cols) epi_store<EPI>(e, z, i, j, acc[p][q], epi_load<EPI>(e, z, i, j));
            }
        }
    }
}

// pdl: launch as a programmatic dependent of the previous kernel on st.
template <int EPI, bool KB>
void launch_gemm(const GemmArgs& g, const EpiArgs& e, int M, cudaStream_t st, bool pdl) {
    if (g.rows >= 1024 && g.cols >= 64) {
        static RidOnce once;
        rid_opt_in(once, BIG_SMEM, k_tr_big<EPI, KB>);
        launch_k(k_tr_big<EPI, KB>, dim3((g.cols + BT - 1) / BT, (g.rows + BT - 1) / BT, M), dim3(TT), BIG_SMEM, st, pdl,
                 g, e);
        return;
    }
    static RidOnce once;
    rid_opt_in(once, sizeof(float) * tile_floats(RID_MAX_WIDTH, KB), k_tr_tile<EPI, KB>);
    launch_k(k_tr_tile<EPI, KB>, dim3((g.cols + 31) / 32, (g.rows + 31) / 32, M), dim3(TT),
             sizeof(float) * tile_floats(g.K, KB), st, pdl, g, e);
}

}  // namespace
