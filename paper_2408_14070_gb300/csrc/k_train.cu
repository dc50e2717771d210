// k_train.cu -- training the ensemble on mean-force labels (Sec. "Training
// phase": numb_models, neurons, resnet, batch_size, init_lr, decay_steps,
// decay_rate; Sec. "Training": the models are fitted to the labelled mean
// forces, the derivatives of the free energy).
//
// Each member i is fitted on its own batches: the loss is the mean squared
// difference between its CV gradient dA_i/ds and the label MF over the batch
// and the C components, and the weights take one Adam step per batch with the
// learning rate init_lr * decay_rate^(t / decay_steps).
//
// One training step is a chain of batched FP32 GEMMs (members on grid z) with
// the elementwise work of each pass fused into the GEMM that produces its
// input (notation of the per-layer recurrences; r_l = 1 for residual layers):
//   forward    l = 0..L-1:  t_l = tanh(h_{l-1} W_l^T + b_l), h_l = t_l + r_l h_{l-1}
//                           (last layer: g_{L-1} = w_out, d_{L-1} = g (1 - t^2))
//   input grad l = L-1..0:  g_{l-1} = d_l W_l + r_l g_l, d_{l-1} = g_{l-1} (1 - t_{l-1}^2)
//   loss:                   dA/ds_j = -sin s_j g[2j] + cos s_j g[2j+1], its adjoint gbar_{-1}
//   adjoint    l = 0..L-1:  dbar = gbar_{l-1} W_l^T, gbar_l = dbar (1 - t^2) + r_l gbar_{l-1},
//                           tbar_l = -2 t_l g_l dbar  (last layer: zbar = tbar (1 - t^2))
//   back       l = L-1..1:  hbar_{l-1} = zbar_l W_l + r_l hbar_l,
//                           zbar_{l-1} = (tbar_{l-1} + hbar_{l-1}) (1 - t_{l-1}^2)
//   weights:   dW_l = d_l^T gbar_{l-1} + zbar_l^T h_{l-1} (one GEMM over 2B rows),
//              db_l = sum_b zbar_l, dw_out = sum_b gbar_{L-1}, db_out = 0,
//              and Adam (Kingma & Ba) on every parameter, in one launch.
// A step is 4L + 1 launches.
// Dropout (drop_out_rate) scales each hidden unit's tanh by q in {0, 1/(1-p)}:
// h_l = q t_l + r_l h_{l-1}, and every (1 - t^2) above that belongs to a
// layer's activation derivative becomes q (1 - t^2), tbar_l gains the factor
// q, and zbar_{l-1} = (tbar + q hbar)(1 - t^2).  The masks come from Philox,
// one counter per four units, drawn by the batch gather of each step.
// Every sum is taken in a fixed order, so a run is reproducible bit for bit.
#include <algorithm>
#include <cmath>
#include <vector>

#include "rid_gemm.cuh"

namespace {

// Dropout scales of one step (one Philox block per four units):
// Q[l][m][b][j] = 1/(1-p) iff word j % 4 of Philox(j / 4 + nw (l + L m), b,
// step, 4) >= thr, else 0 (nw = ceil(H / 4)).
struct MaskArgs {
    float* Q;                  // NULL: no dropout
    int L, H, ld;              // ld: floats of a row of H
    uint32_t step, thr, k0, k1;
    float scale;
};
__device__ __forceinline__ void tr_mask_block(const MaskArgs& a, int M, int B, long long e) {
    const int nw = (a.H + 3) / 4;
    const int k = (int)(e % nw);
    const long long r = e / nw;                       // (l, m, b)
    const int b = (int)(r % B);
    const long long lm = r / B;                       // l M + m
    const int m = (int)(lm % M), l = (int)(lm / M);
    const uint4 x = rid_philox(make_uint4((uint32_t)(k + nw * (l + a.L * m)), (uint32_t)b, a.step, 4u), a.k0, a.k1);
    const uint32_t wd[4] = {x.x, x.y, x.z, x.w};
    float* q = a.Q + r * a.ld + 4 * k;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (4 * k + c < a.H) q[c] = wd[c] >= a.thr ? a.scale : 0.0f;
}

// u = (cos s, sin s) of each member's batch ((s, 0) for a distance CV:
// dist[j] != 0; rows of ldu floats), plus the batch's labels and the step's
// dropout scales.  idx is checked; an index outside [0, n) reads sample 0 and
// sets *bad.  Triggers its dependents only after its own wait: they read the
// weights before theirs.
__global__ void k_tr_gather(const int* __restrict__ idx, const float* __restrict__ s, const float* __restrict__ mf,
                            int n, int M, int B, int C, float* __restrict__ U, int ldu, float* __restrict__ MFB,
                            int* bad, MaskArgs mk, const int* __restrict__ dist) {
    pdl_wait();
    pdl_trigger();
    if (mk.Q) {
        const long long nm = (long long)mk.L * M * B * ((mk.H + 3) / 4);
        for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nm; e += (long long)gridDim.x * blockDim.x)
            tr_mask_block(mk, M, B, e);
    }
    const long long tot = (long long)M * B * C;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const long long mb = e / C;
        const int j = (int)(e - mb * C);
        int k = idx[mb];
        if (k < 0 || k >= n) {
            atomicOr(bad, 1);
            k = 0;
        }
        const float sv = s[(long long)k * C + j];
        float cs = sv, sn = 0.0f;
        if (!(dist && dist[j])) sincosf(sv, &sn, &cs);
        U[mb * ldu + 2 * j] = cs;
        U[mb * ldu + 2 * j + 1] = sn;
        MFB[e] = mf[(long long)k * C + j];
    }
}

// Where a member's parameters lie inside the trainer: every matrix row, vector
// and member starts on 16 bytes (the packed layout of the interface has odd
// strides), padded with zeros that stay zero.
struct ParamMap {
    int L, H, D, ldh, ldd;
    long long Pp, w[RID_MAX_LAYERS], b[RID_MAX_LAYERS], wo;   // floats per member; offsets
    long long P;                                              // packed floats per member
};
// Padded offset of packed parameter p.
__host__ __device__ inline long long param_at(const ParamMap& m, long long p) {
    for (int l = 0; l < m.L; ++l) {
        const int fin = l == 0 ? m.D : m.H, ld = l == 0 ? m.ldd : m.ldh;
        const long long n = (long long)m.H * fin;
        if (p < n) return m.w[l] + p / fin * ld + p % fin;
        p -= n;
        if (p < m.H) return m.b[l] + p;
        p -= m.H;
    }
    return m.wo + p;   // w_out, then b_out
}
__global__ void k_tr_unpad(const float* __restrict__ src, float* __restrict__ dst, int M, ParamMap m) {
    const long long n = (long long)M * m.P;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long i = e / m.P;
        dst[e] = src[i * m.Pp + param_at(m, e - i * m.P)];
    }
}

// One step's update: weight gradients, column sums, the loss and Adam.
struct UpdateArgs {
    ParamMap m;
    int M, B, C;
    const float *Dl[RID_MAX_LAYERS], *GBin[RID_MAX_LAYERS], *ZB[RID_MAX_LAYERS], *Hin[RID_MAX_LAYERS];
    const float* GBlast;
    const float* R;            // [M][B C] residuals
    double* lpart;             // [M][ceil(B C / 256)]
    float* loss;               // [M]
    float *grad, *w, *am, *av; // grad NULL: Adam in place, else the gradient alone
    float lr, b1, b2, eps, c1, c2;
    int tile0[RID_MAX_LAYERS + 1];   // first block of each layer's tiles (per member), then their total
    int sums;                        // blocks of the column sums per member
};

__device__ __forceinline__ void tr_apply(const UpdateArgs& A, long long e, float gv) {
    if (A.grad) {
        A.grad[e] = gv;
        return;
    }
    const float m = fmaf(A.b1, A.am[e], (1.0f - A.b1) * gv);
    const float v = fmaf(A.b2, A.av[e], (1.0f - A.b2) * gv * gv);
    A.am[e] = m;
    A.av[e] = v;
    A.w[e] -= A.lr * (m / A.c1) / (sqrtf(v / A.c2) + A.eps);
}

// Grid (blocks per member, M).  A block is one of
//   a 64 x 64 tile of dW_l = d_l^T gbar_{l-1} + zbar_l^T h_{l-1}: K tiles of 32
//     batch rows of the two products in one sequence through a ring of stages
//     (both operands row-contiguous, 16-byte copies), even and odd tiles summed
//     apart and added, every output in increasing k;
//   256 columns of one of the column sums (rows in increasing order);
//   the loss of the member: chunks of 256 squared residuals, each by a
//     fixed tree (one warp), added in order.
// Parameters are read and written once, in the epilogue: the gradient never
// goes to memory unless it is asked for.
constexpr int UK = 32, UT = 64, ULD = UT + 4, UNS = 3;
constexpr size_t UPD_SMEM = sizeof(float) * 2 * UNS * UK * ULD;
__global__ void __launch_bounds__(256) k_tr_update(UpdateArgs A) {
    extern __shared__ __align__(16) float gsm[];
    pdl_wait();
    pdl_trigger();
    const int z = blockIdx.y, tid = threadIdx.x;
    const int B = A.B, H = A.m.H, L = A.m.L;
    int blk = blockIdx.x;
    if (blk < A.tile0[L]) {
        int l = 0;
        while (blk >= A.tile0[l + 1]) ++l;
        blk -= A.tile0[l];
        const int fin = l == 0 ? A.m.D : H, ldf = l == 0 ? A.m.ldd : A.m.ldh, ldh = A.m.ldh;
        const int nx = (fin + UT - 1) / UT, i0 = blk / nx * UT, j0 = blk % nx * UT;
        const float* pa[2] = {A.Dl[l] + (long long)z * B * ldh, A.ZB[l] + (long long)z * B * ldh};
        const float* pb[2] = {A.GBin[l] + (long long)z * B * ldf, A.Hin[l] + (long long)z * B * ldf};
        const int nt0 = (B + UK - 1) / UK, nt = 2 * nt0;
        float* As = gsm;
        float* Bs = gsm + UNS * UK * ULD;
        auto issue = [&](int t) {
            if (t < nt) {
                const int seg = t >= nt0, k0 = (t - (seg ? nt0 : 0)) * UK;
                const float* a = seg ? pa[1] : pa[0];
                const float* b = seg ? pb[1] : pb[0];
                float* as = As + (t % UNS) * UK * ULD;
                float* bs = Bs + (t % UNS) * UK * ULD;
#pragma unroll
                for (int r = 0; r < UK * UT / 4 / 256; ++r) {
                    const int q = tid + 256 * r, kk = q >> 4, c = 4 * (q & 15), k = k0 + kk;
                    const int la = k < B ? H - (i0 + c) : 0, lb = k < B ? fin - (j0 + c) : 0;
                    cp_async16(as + kk * ULD + c, la > 0 ? a + (long long)k * ldh + i0 + c : a, bytes4(la));
                    cp_async16(bs + kk * ULD + c, lb > 0 ? b + (long long)k * ldf + j0 + c : b, bytes4(lb));
                }
            }
            cp_async_commit();
        };
        const int tx = tid & 15, ty = tid >> 4;
        float acc[2][4][4] = {};
        auto mul = [&](int t, float(&c)[4][4]) {
            const float* as = As + (t % UNS) * UK * ULD + 4 * ty;
            const float* bs = Bs + (t % UNS) * UK * ULD + 4 * tx;
#pragma unroll
            for (int kk = 0; kk < UK; ++kk) {
                const float4 a = *reinterpret_cast<const float4*>(as + kk * ULD);
                const float4 b = *reinterpret_cast<const float4*>(bs + kk * ULD);
                const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[p][q] = fmaf(x[p], y[q], c[p][q]);
            }
        };
#pragma unroll
        for (int t = 0; t < UNS - 1; ++t) issue(t);
        for (int t = 0; t < nt; ++t) {
            cp_async_wait<UNS - 2>();
            __syncthreads();
            issue(t + UNS - 1);
            if (t & 1) mul(t, acc[1]);
            else mul(t, acc[0]);
        }
        cp_async_wait<0>();
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const int i = i0 + 4 * ty + p;
            if (i >= H) continue;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + 4 * tx + q;
                if (j < fin)
                    tr_apply(A, (long long)z * A.m.Pp + A.m.w[l] + (long long)i * ldf + j, acc[0][p][q] + acc[1][p][q]);
            }
        }
        return;
    }
    blk -= A.tile0[L];
    if (blk < A.sums) {
        const int nb = (H + 255) / 256, v = blk / nb, j = blk % nb * 256 + tid;
        if (j >= H) return;
        const int ld = A.m.ldh;
        const float* src = (v < L ? A.ZB[v] : A.GBlast) + (long long)z * B * ld + j;
        // rows in increasing order; eight loads are issued ahead of their adds
        float a = 0.0f;
        int b = 0;
        for (; b + 8 <= B; b += 8) {
            float x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = __ldcg(src + (long long)(b + k) * ld);
#pragma unroll
            for (int k = 0; k < 8; ++k) a += x[k];
        }
        for (; b < B; ++b) a += __ldcg(src + (long long)b * ld);
        tr_apply(A, (long long)z * A.m.Pp + (v < L ? A.m.b[v] : A.m.wo) + j, a);
        return;
    }
    // loss[m] = sum over chunks of (the chunk's tree sum) / (B C): element t of a
    // chunk adds element t + w for w = 128, 64, 32 (within a lane), then 16 .. 1
    const long long n = (long long)B * A.C, nchunk = (n + 255) / 256;
    const int warp = tid >> 5, lane = tid & 31;
    for (long long c = warp; c < nchunk; c += 8) {
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long e = c * 256 + 32 * k + lane;
            const float r = e < n ? __ldcg(A.R + (long long)z * n + e) : 0.0f;
            x[k] = (double)r * r;
        }
#pragma unroll
        for (int w = 4; w > 0; w >>= 1)
#pragma unroll
            for (int k = 0; k < w; ++k) x[k] += x[k + w];
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) x[0] += __shfl_down_sync(0xffffffffu, x[0], w);
        if (lane == 0) A.lpart[z * nchunk + c] = x[0];
    }
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (long long c = 0; c < nchunk; ++c) t += A.lpart[z * nchunk + c];
        A.loss[z] = (float)(t / (double)n);
    }
}

}  // namespace

// ---------------------------------------------------------------------------
struct rid_trainer {
    rid_train_desc d{};
    int D = 0, P = 0;
    ParamMap pm{};
    int64_t steps = 0;
    int n_data = 0, cap_data = 0;
    float* w = nullptr;      // [M][Pp] padded parameters, then Adam m, v and the gradient
    float* am = nullptr;
    float* av = nullptr;
    float* grad = nullptr;
    float* ds = nullptr;     // data s [n][C], mf [n][C]
    float* dmf = nullptr;
    float* act = nullptr;    // activations (see carve)
    int* didx = nullptr;     // [cap_idx] batch indices
    long long cap_idx = 0;
    float* dloss = nullptr;  // [cap_loss]
    long long cap_loss = 0;
    int* dbad = nullptr;
    int* ddist = nullptr;     // [C] 1 for a distance CV, or NULL (all torsions)
    double* lpart = nullptr;  // [M][ceil(B C / 256)] loss chunk sums
    float* packed = nullptr;  // [M][P] staging of host reads (on first use)
    // carve of act, [M][B][ld] (MFB, R: [M][B][C])
    float *U, *MFB, *GB0, *R;
    float* Q[RID_MAX_LAYERS] = {};   // dropout scales [M][B][H] per layer (NULL: no dropout)
    uint32_t dthr = 0;               // keep iff the Philox word >= dthr
    float dscale = 1.0f;             // 1 / (1 - rate)
    float *T[RID_MAX_LAYERS], *Hh[RID_MAX_LAYERS], *G[RID_MAX_LAYERS], *Dl[RID_MAX_LAYERS], *GB[RID_MAX_LAYERS],
        *TB[RID_MAX_LAYERS], *ZB[RID_MAX_LAYERS], *HB[RID_MAX_LAYERS];
};

namespace {

int tr_fail_cuda(cudaError_t e, const char* what) {
    return rid_fail(RID_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}
#define TCK(x)                                          \
    do {                                                \
        cudaError_t e_ = (x);                           \
        if (e_ != cudaSuccess) return tr_fail_cuda(e_, #x); \
    } while (0)

int grow(void** p, long long* cap, long long need, size_t elem) {
    if (need <= *cap) return RID_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    if (cudaMalloc(p, (size_t)need * elem) != cudaSuccess) {
        cudaGetLastError();
        return rid_fail(RID_ERR_OOM, "trainer: cudaMalloc of %lld bytes failed", need * (long long)elem);
    }
    *cap = need;
    return RID_OK;
}

// One step for the batch indices idx [M][B] (device) at training step `step`
// (the step index of the dropout masks): the per-member loss into loss[M], and
// the Adam update `up` or (up NULL) the gradient into tr->grad.  Every kernel
// after the first is a programmatic dependent of its predecessor; the first is
// one too unless `after_copy` (it then follows a memory copy).
struct AdamStep {
    float lr, c1, c2;
};
int tr_step(rid_trainer* tr, const int* idx, float* loss, int64_t step, const AdamStep* up, bool after_copy,
            cudaStream_t st) {
    const rid_train_desc& d = tr->d;
    const ParamMap& pm = tr->pm;
    const int M = d.n_models, B = d.batch_size, C = d.n_cv, D = tr->D, L = d.n_layers, H = d.width;
    const int ldh = pm.ldh, ldd = pm.ldd;
    const long long smH = (long long)B * ldh, smD = (long long)B * ldd;
    {
        MaskArgs mk{tr->Q[0], L, H, ldh, (uint32_t)step, tr->dthr, (uint32_t)d.dropout_seed,
                    (uint32_t)(d.dropout_seed >> 32), tr->dscale};
        long long tot = (long long)M * B * C;
        if (mk.Q && (long long)L * M * B * ((H + 3) / 4) > tot) tot = (long long)L * M * B * ((H + 3) / 4);
        const int blocks = (int)((tot + 255) / 256 < 1024 ? (tot + 255) / 256 : 1024);
        TCK(launch_k(k_tr_gather, dim3(blocks), dim3(256), 0, st, !after_copy, idx, (const float*)tr->ds,
                     (const float*)tr->dmf, tr->n_data, M, B, C, tr->U, ldd, tr->MFB, tr->dbad, mk,
                     (const int*)tr->ddist));
    }
    auto gemm = [&](const float* A, int fin, int l, int cols) {
        GemmArgs g{};
        g.A = A;
        g.lda = fin == D && l < 0 ? ldd : ldh;
        g.a_sm = (long long)B * g.lda;
        g.K = fin;
        g.rows = B;
        g.cols = cols;
        g.b_sm = pm.Pp;
        return g;
    };
    auto epi = [&](bool wide) {
        EpiArgs e{};
        e.ld = wide ? ldd : ldh;
        e.sm = wide ? smD : smH;
        e.w_sm = pm.Pp;
        return e;
    };
    // forward
    for (int l = 0; l < L; ++l) {
        GemmArgs g = gemm(l == 0 ? tr->U : tr->Hh[l - 1], l == 0 ? D : H, l == 0 ? -1 : l, H);
        g.B = tr->w + pm.w[l];                      // (k, j) -> W_l[j][k]
        g.ldb = l == 0 ? ldd : ldh;
        EpiArgs e = epi(false);
        e.bias = tr->w + pm.b[l];
        e.T = tr->T[l];
        e.Hout = tr->Hh[l];
        e.Hin = l == 0 ? nullptr : tr->Hh[l - 1];
        e.resid = d.resnet && l >= 1;
        e.last = l == L - 1;
        e.wout = tr->w + pm.wo;
        e.Gout = tr->G[L - 1];
        e.Dout = tr->Dl[L - 1];
        e.Q = tr->Q[l];
        launch_gemm<EPI_FWD, true>(g, e, M, st, true);
    }
    // input gradient, decreasing l: g_{l-1} = d_l W_l (+ r g_l); layer 0 ends in the loss
    for (int l = L - 1; l >= 0; --l) {
        GemmArgs g = gemm(tr->Dl[l], H, l, l == 0 ? D : H);
        g.B = tr->w + pm.w[l];                      // (k, j) -> W_l[k][j]
        g.ldb = l == 0 ? ldd : ldh;
        EpiArgs e = epi(l == 0);
        if (l == 0) {
            e.out = tr->GB0;
            e.U = tr->U;
            e.MF = tr->MFB;
            e.R = tr->R;
            e.dist = tr->ddist;
            e.scale = 2.0f / (float)((long long)B * C);
            launch_gemm<EPI_LOSS, false>(g, e, M, st, true);
        } else {
            e.out = tr->G[l - 1];
            e.resid = d.resnet;
            e.res = tr->G[l];
            e.Tl = tr->T[l - 1];
            e.Dout = tr->Dl[l - 1];
            e.Q = tr->Q[l - 1];
            launch_gemm<EPI_BWD, false>(g, e, M, st, true);
        }
    }
    // adjoint of the input-gradient pass, increasing l
    for (int l = 0; l < L; ++l) {
        GemmArgs g = gemm(l == 0 ? tr->GB0 : tr->GB[l - 1], l == 0 ? D : H, l == 0 ? -1 : l, H);
        g.B = tr->w + pm.w[l];                      // W_l^T
        g.ldb = l == 0 ? ldd : ldh;
        EpiArgs e = epi(false);
        e.out = tr->GB[l];
        e.resid = d.resnet && l >= 1;
        e.res = l == 0 ? nullptr : tr->GB[l - 1];
        e.Tl = tr->T[l];
        e.Gl = tr->G[l];
        e.out2 = tr->TB[l];
        e.last = l == L - 1;
        e.out3 = tr->ZB[L - 1];
        e.Q = tr->Q[l];
        launch_gemm<EPI_ADJ, true>(g, e, M, st, true);
    }
    // back through the forward pass, decreasing l (hbar_{L-1} = 0)
    for (int l = L - 1; l >= 1; --l) {
        GemmArgs g = gemm(tr->ZB[l], H, l, H);
        g.B = tr->w + pm.w[l];                      // W_l
        g.ldb = ldh;
        EpiArgs e = epi(false);
        e.out = tr->HB[l - 1];
        e.resid = d.resnet && l < L - 1;            // hbar_{L-1} = 0
        e.res = tr->HB[l];
        e.Tl = tr->T[l - 1];
        e.tb = tr->TB[l - 1];
        e.out3 = tr->ZB[l - 1];
        e.Q = tr->Q[l - 1];
        launch_gemm<EPI_BACK, false>(g, e, M, st, true);
    }
    UpdateArgs u{};
    u.m = pm;
    u.M = M;
    u.B = B;
    u.C = C;
    for (int l = 0; l < L; ++l) {
        u.Dl[l] = tr->Dl[l];
        u.ZB[l] = tr->ZB[l];
        u.GBin[l] = l == 0 ? tr->GB0 : tr->GB[l - 1];
        u.Hin[l] = l == 0 ? tr->U : tr->Hh[l - 1];
        u.tile0[l + 1] = u.tile0[l] + (H + UT - 1) / UT * (((l == 0 ? D : H) + UT - 1) / UT);
    }
    u.GBlast = tr->GB[L - 1];
    u.R = tr->R;
    u.lpart = tr->lpart;
    u.loss = loss;
    u.w = tr->w;
    u.am = tr->am;
    u.av = tr->av;
    u.grad = up ? nullptr : tr->grad;
    if (up) {
        u.lr = up->lr;
        u.c1 = up->c1;
        u.c2 = up->c2;
        u.b1 = (float)d.beta1;
        u.b2 = (float)d.beta2;
        u.eps = (float)d.adam_eps;
    }
    u.sums = (L + 1) * ((H + 255) / 256);
    static RidOnce once;
    TCK(rid_opt_in(once, UPD_SMEM, k_tr_update));
    TCK(launch_k(k_tr_update, dim3(u.tile0[L] + u.sums + 1, M), dim3(256), UPD_SMEM, st, true, u));
    return RID_OK;
}

// The padded parameters src to the caller's packed [M][P].
int tr_unpad_out(rid_trainer* tr, const float* src, float* dst, int mem, cudaStream_t st) {
    const long long n = (long long)tr->d.n_models * tr->P;
    const int blocks = (int)((n + 255) / 256 < 2048 ? (n + 255) / 256 : 2048);
    if (mem == RID_MEM_DEVICE) {
        k_tr_unpad<<<blocks, 256, 0, st>>>(src, dst, tr->d.n_models, tr->pm);
        TCK(cudaGetLastError());
        return RID_OK;
    }
    if (!tr->packed && cudaMalloc(&tr->packed, sizeof(float) * n) != cudaSuccess) {
        cudaGetLastError();
        tr->packed = nullptr;
        return rid_fail(RID_ERR_OOM, "trainer: device allocation failed");
    }
    k_tr_unpad<<<blocks, 256, 0, st>>>(src, tr->packed, tr->d.n_models, tr->pm);
    TCK(cudaGetLastError());
    TCK(cudaMemcpyAsync(dst, tr->packed, sizeof(float) * n, cudaMemcpyDeviceToHost, st));
    return RID_OK;
}

int tr_check_desc(const rid_train_desc* d) {
    if (!d) return rid_fail(RID_ERR_ARG, "trainer: desc is NULL");
    if (d->n_models < 1 || d->n_models > RID_MAX_MODELS) return rid_fail(RID_ERR_ARG, "trainer: n_models out of range");
    if (d->n_cv < 1 || d->n_cv > RID_MAX_CV) return rid_fail(RID_ERR_ARG, "trainer: n_cv out of range");
    if (d->n_layers < 1 || d->n_layers > RID_MAX_LAYERS) return rid_fail(RID_ERR_ARG, "trainer: n_layers out of range");
    if (d->width < 1 || d->width > RID_MAX_WIDTH) return rid_fail(RID_ERR_ARG, "trainer: width out of range");
    if (d->batch_size < 1 || d->batch_size > 65536) return rid_fail(RID_ERR_ARG, "trainer: batch_size out of range");
    if (!(d->init_lr > 0) || !(d->decay_rate > 0) || d->decay_steps < 1)
        return rid_fail(RID_ERR_ARG, "trainer: learning-rate schedule out of range");
    if (!(d->beta1 >= 0 && d->beta1 < 1) || !(d->beta2 >= 0 && d->beta2 < 1) || !(d->adam_eps > 0))
        return rid_fail(RID_ERR_ARG, "trainer: Adam parameters out of range");
    if (!(d->dropout_rate >= 0 && d->dropout_rate < 1)) return rid_fail(RID_ERR_ARG, "trainer: dropout_rate outside [0, 1)");
    return RID_OK;
}

int tr_copy_in(void* dst, const void* src, size_t bytes, int mem, cudaStream_t st) {
    TCK(cudaMemcpyAsync(dst, src, bytes, mem == RID_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st));
    return RID_OK;
}
int tr_copy_out(void* dst, const void* src, size_t bytes, int mem, cudaStream_t st) {
    TCK(cudaMemcpyAsync(dst, src, bytes, mem == RID_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
    return RID_OK;
}

int tr_finish(rid_trainer* tr, cudaStream_t st) {
    int bad = 0;
    TCK(cudaMemcpyAsync(&bad, tr->dbad, sizeof(int), cudaMemcpyDeviceToHost, st));
    TCK(cudaStreamSynchronize(st));
    TCK(cudaGetLastError());
    if (bad) {
        TCK(cudaMemsetAsync(tr->dbad, 0, sizeof(int), st));
        TCK(cudaStreamSynchronize(st));
        return rid_fail(RID_ERR_ARG, "trainer: a batch index is outside [0, n_data)");
    }
    return RID_OK;
}

}  // namespace

extern "C" {

RID_API int rid_trainer_create(const rid_train_desc* desc, const float* weights, rid_trainer** out) {
    if (!out || !weights) return rid_fail(RID_ERR_ARG, "trainer: NULL argument");
    *out = nullptr;
    if (int rc = tr_check_desc(desc)) return rc;
    rid_trainer* tr = new rid_trainer();
    tr->d = *desc;
    const int M = desc->n_models, C = desc->n_cv, L = desc->n_layers, H = desc->width, B = desc->batch_size;
    const int D = 2 * C;
    tr->D = D;
    auto round4 = [](long long n) { return (n + 3) / 4 * 4; };
    ParamMap& pm = tr->pm;
    pm.L = L;
    pm.H = H;
    pm.D = D;
    pm.ldh = (int)round4(H);
    pm.ldd = (int)round4(D);
    for (int l = 0; l < L; ++l) {
        pm.w[l] = pm.Pp;
        pm.Pp += (long long)H * (l == 0 ? pm.ldd : pm.ldh);
        pm.b[l] = pm.Pp;
        pm.Pp += pm.ldh;
        pm.P += (long long)H * (l == 0 ? D : H) + H;
    }
    pm.wo = pm.Pp;
    pm.Pp += round4(H + 1);
    pm.P += H + 1;
    tr->P = (int)pm.P;
    const long long nP = (long long)M * pm.Pp;
    const long long smH = (long long)B * pm.ldh, smD = (long long)B * pm.ldd, smC = (long long)B * C;
    // activations: U, GB0 [M][B][ldd]; MFB, R [M][B][C] (each member start on 16 bytes); per layer T, Hh
    // (resnet or dropout), G, Dl, GB, TB, ZB, HB, and Q (dropout)
    const bool drop = desc->dropout_rate > 0;
    const long long per_layer = ((desc->resnet || drop ? 8 : 7) + (drop ? 1 : 0)) * smH;
    const long long nact = (long long)M * (2 * smD + L * per_layer) + 2 * round4(M * smC);
    bool ok = cudaMalloc(&tr->w, sizeof(float) * 4 * nP) == cudaSuccess;
    ok = ok && cudaMalloc(&tr->act, sizeof(float) * nact) == cudaSuccess;
    ok = ok && cudaMalloc(&tr->dbad, sizeof(int)) == cudaSuccess;
    ok = ok && cudaMalloc(&tr->lpart, sizeof(double) * M * (((long long)B * C + 255) / 256)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        rid_trainer_destroy(tr);
        return rid_fail(RID_ERR_OOM, "trainer: device allocation failed");
    }
    tr->am = tr->w + nP;
    tr->av = tr->am + nP;
    tr->grad = tr->av + nP;
    float* p = tr->act;
    auto take = [&](long long per_member) { float* r = p; p += M * per_member; return r; };
    tr->U = take(smD);
    tr->GB0 = take(smD);
    for (int l = 0; l < L; ++l) {
        tr->T[l] = take(smH);
        tr->Hh[l] = desc->resnet || drop ? take(smH) : tr->T[l];
        tr->G[l] = take(smH);
        tr->Dl[l] = take(smH);
        tr->GB[l] = take(smH);
        tr->TB[l] = take(smH);
        tr->ZB[l] = take(smH);
        tr->HB[l] = take(smH);
    }
    if (drop) {   // the scales of all layers are contiguous: the gather writes them in one launch
        for (int l = 0; l < L; ++l) tr->Q[l] = take(smH);
        tr->dthr = (uint32_t)std::floor(desc->dropout_rate * 4294967296.0);
        tr->dscale = (float)(1.0 / (1.0 - desc->dropout_rate));
    }
    tr->MFB = p;
    tr->R = p + round4(M * smC);
    bool any_dist = false;
    for (int j = 0; desc->cv_dist && j < C; ++j) any_dist |= desc->cv_dist[j] != 0;
    if (any_dist) {
        std::vector<int> h(C);
        for (int j = 0; j < C; ++j) h[j] = desc->cv_dist[j] ? 1 : 0;
        if (cudaMalloc(&tr->ddist, sizeof(int) * C) != cudaSuccess ||
            cudaMemcpy(tr->ddist, h.data(), sizeof(int) * C, cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaGetLastError();
            rid_trainer_destroy(tr);
            return rid_fail(RID_ERR_OOM, "trainer: device allocation failed");
        }
    }
    tr->d.cv_dist = nullptr;   // the caller's array is not kept
    std::vector<float> padded((size_t)nP, 0.0f);
    for (int m = 0; m < M; ++m) {
        const float* src = weights + (size_t)m * pm.P;
        float* dst = padded.data() + (size_t)m * pm.Pp;
        for (int l = 0; l < L; ++l) {
            const int fin = l == 0 ? D : H, ld = l == 0 ? pm.ldd : pm.ldh;
            for (int i = 0; i < H; ++i, src += fin) std::copy(src, src + fin, dst + pm.w[l] + (size_t)i * ld);
            std::copy(src, src + H, dst + pm.b[l]);
            src += H;
        }
        std::copy(src, src + H + 1, dst + pm.wo);
    }
    if (cudaMemcpy(tr->w, padded.data(), sizeof(float) * nP, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(tr->am, 0, sizeof(float) * 3 * nP) != cudaSuccess || cudaMemset(tr->act, 0, sizeof(float) * nact) != cudaSuccess ||
        cudaMemset(tr->dbad, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        rid_trainer_destroy(tr);
        return rid_fail(RID_ERR_CUDA, "trainer: initial copy failed");
    }
    *out = tr;
    return RID_OK;
}

RID_API int rid_trainer_destroy(rid_trainer* tr) {
    if (!tr) return RID_OK;
    cudaFree(tr->w);
    cudaFree(tr->act);
    cudaFree(tr->dbad);
    cudaFree(tr->ddist);
    cudaFree(tr->lpart);
    cudaFree(tr->packed);
    cudaFree(tr->ds);
    cudaFree(tr->didx);
    cudaFree(tr->dloss);
    delete tr;
    return RID_OK;
}

RID_API int rid_trainer_set_data(rid_trainer* tr, int32_t n, const float* s, const float* mf, int32_t mem, void* stream) {
    if (!tr || !s || !mf || n < 1) return rid_fail(RID_ERR_ARG, "trainer: bad data arguments");
    if (mem != RID_MEM_HOST && mem != RID_MEM_DEVICE) return rid_fail(RID_ERR_ARG, "trainer: bad mem");
    cudaStream_t st = (cudaStream_t)stream;
    const int C = tr->d.n_cv;
    if (n > tr->cap_data) {
        cudaFree(tr->ds);
        tr->ds = nullptr;
        tr->cap_data = 0;
        if (cudaMalloc(&tr->ds, sizeof(float) * 2 * (size_t)n * C) != cudaSuccess) {
            cudaGetLastError();
            return rid_fail(RID_ERR_OOM, "trainer: data allocation failed");
        }
        tr->cap_data = n;
    }
    tr->dmf = tr->ds + (size_t)tr->cap_data * C;
    tr->n_data = n;
    if (int rc = tr_copy_in(tr->ds, s, sizeof(float) * (size_t)n * C, mem, st)) return rc;
    if (int rc = tr_copy_in(tr->dmf, mf, sizeof(float) * (size_t)n * C, mem, st)) return rc;
    TCK(cudaStreamSynchronize(st));
    return RID_OK;
}

RID_API int rid_trainer_grad(rid_trainer* tr, const int32_t* idx, float* loss_out, float* grad_out, int32_t mem,
                             void* stream) {
    NvtxScope nvtx_("rid_trainer_grad");
    if (!tr || !idx) return rid_fail(RID_ERR_ARG, "trainer: NULL argument");
    if (mem != RID_MEM_HOST && mem != RID_MEM_DEVICE) return rid_fail(RID_ERR_ARG, "trainer: bad mem");
    if (tr->n_data < 1) return rid_fail(RID_ERR_STATE, "trainer: no data set");
    cudaStream_t st = (cudaStream_t)stream;
    const int M = tr->d.n_models, B = tr->d.batch_size;
    if (int rc = grow((void**)&tr->didx, &tr->cap_idx, (long long)M * B, sizeof(int))) return rc;
    if (int rc = grow((void**)&tr->dloss, &tr->cap_loss, M, sizeof(float))) return rc;
    if (int rc = tr_copy_in(tr->didx, idx, sizeof(int) * (size_t)M * B, mem, st)) return rc;
    if (int rc = tr_step(tr, tr->didx, tr->dloss, tr->steps, nullptr, true, st)) return rc;
    TCK(cudaGetLastError());
    if (loss_out)
        if (int rc = tr_copy_out(loss_out, tr->dloss, sizeof(float) * M, mem, st)) return rc;
    if (grad_out)
        if (int rc = tr_unpad_out(tr, tr->grad, grad_out, mem, st)) return rc;
    return tr_finish(tr, st);
}

RID_API int rid_trainer_run(rid_trainer* tr, int32_t n_steps, const int32_t* idx, float* loss_out, int32_t mem,
                            void* stream) {
    NvtxScope nvtx_("rid_trainer_run");
    if (!tr || !idx || n_steps < 0) return rid_fail(RID_ERR_ARG, "trainer: bad run arguments");
    if (mem != RID_MEM_HOST && mem != RID_MEM_DEVICE) return rid_fail(RID_ERR_ARG, "trainer: bad mem");
    if (tr->n_data < 1) return rid_fail(RID_ERR_STATE, "trainer: no data set");
    if (n_steps == 0) return RID_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const rid_train_desc& d = tr->d;
    const int M = d.n_models, B = d.batch_size;
    const long long per = (long long)M * B;
    if (int rc = grow((void**)&tr->didx, &tr->cap_idx, per * n_steps, sizeof(int))) return rc;
    if (int rc = grow((void**)&tr->dloss, &tr->cap_loss, (long long)M * n_steps, sizeof(float))) return rc;
    if (int rc = tr_copy_in(tr->didx, idx, sizeof(int) * (size_t)(per * n_steps), mem, st)) return rc;
    for (int k = 0; k < n_steps; ++k) {
        const int64_t t = tr->steps + k;
        const double lr = d.init_lr * std::pow(d.decay_rate, (double)t / (double)d.decay_steps);
        const double c1 = 1.0 - std::pow(d.beta1, (double)(t + 1)), c2 = 1.0 - std::pow(d.beta2, (double)(t + 1));
        const AdamStep up{(float)lr, (float)c1, (float)c2};
        if (int rc = tr_step(tr, tr->didx + per * k, tr->dloss + (long long)M * k, t, &up, k == 0, st)) return rc;
    }
    TCK(cudaGetLastError());
    if (loss_out)
        if (int rc = tr_copy_out(loss_out, tr->dloss, sizeof(float) * (size_t)M * n_steps, mem, st)) return rc;
    const int rc = tr_finish(tr, st);
    if (rc == RID_OK) tr->steps += n_steps;
    return rc;
}

RID_API int rid_trainer_weights(rid_trainer* tr, float* weights_out, int64_t* steps_done, int32_t mem, void* stream) {
    if (!tr) return rid_fail(RID_ERR_ARG, "trainer: NULL argument");
    if (mem != RID_MEM_HOST && mem != RID_MEM_DEVICE) return rid_fail(RID_ERR_ARG, "trainer: bad mem");
    cudaStream_t st = (cudaStream_t)stream;
    if (weights_out)
        if (int rc = tr_unpad_out(tr, tr->w, weights_out, mem, st)) return rc;
    if (steps_done) *steps_done = tr->steps;
    TCK(cudaStreamSynchronize(st));
    return RID_OK;
}

}  // extern "C"
