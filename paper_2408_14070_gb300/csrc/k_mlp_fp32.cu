// k_mlp_fp32.cu -- plain FP32 (SIMT) ensemble MLP: forward pass and
// reverse-mode input gradient, or the member values alone, for every member on
// a tile of R walkers.
//
// Grid (ceil(W / R), M), 256 threads: 8 / WCN warp rows x WCN warp columns of
// 128 output neurons, WCN = 1, 2 or 4 by width, so a layer is one pass over
// its inputs.  In a warp, half (lane / 16) takes one group of RPT walkers and
// lane % 16 the columns 4 lc .. + 3 and 64 + 4 lc .. + 3, so a thread keeps an
// RPT x 8 register tile, accumulated by fma.rn.f32x2 (two neighbouring columns
// an instruction; each half rounds as fmaf does).  (Member values of widths to 64
// and 32 take CPT = 4 and 2 columns a thread, 16 CPT a warp.)  Activations live in shared
// memory transposed as [neuron][walker] rows of LD floats, one group of RPT
// walkers in GS slots (RPT rounded up to a power of two), so a thread's walkers
// are one or two 16-byte loads; a layer's outputs go back over its inputs once
// every warp has read them.
// Weight rows (forward: W^T [in][out], backward: W [out][in]) stream from L2
// into a ring of NSW stages of KC rows in shared memory by cp.async, shared by
// the eight warps, the first stages of a layer during the epilogue of the one
// before it.
// tanh(z_l) of every layer is kept in a global scratch [M][tile][L][H][walkers of
// the tile] (L2-resident at the sizes used) for the backward pass:
//   g_L = w_out,  delta_l = g_l * (1 - tanh^2 z_l),
//   g_{l-1} = W_l^T delta_l (+ g_l for a residual layer),
//   dA/ds_j = -sin s_j g_0[2j] + cos s_j g_0[2j+1].
//
// Bound by the FP32 pipe at RPT >= 4 (one CTA an SM, two warps a scheduler; a K
// row is 16 RPT cycles of FMAs and 40 to 48 of shared loads), by the shared loads
// at RPT = 2.  The walker count of a tile follows the call (choose_rpt).
// 1024 walkers x 4 members 40-256x4-1 (128 tiles of 32): 238 us with a 256-thread
// CTA of 8 x 4 register tiles, scalar FMAs and 8-row stages, 115 us now (29.5 of
// 69.8 TFLOP/s); a force evaluation of them 353 -> 237 us.
#include <algorithm>

#include "rid_internal.cuh"

namespace {

constexpr int NT = 256;   // threads per CTA
constexpr int F32_SMEM_MAX = 227 * 1024;

// Walkers of a member in the scratch, but for groups of seven (choose_rpt).
__host__ __device__ inline size_t f32_walkers(int W) { return ((size_t)W + 31) / 32 * 32; }

__device__ __forceinline__ void cpa4(float* dst, const float* src, int bytes) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cpa16(float* dst, const float* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Two FP32 values in one 64-bit register pair, and their fused multiply-add.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// Tile shape: RPT walkers and CPT columns a thread, WCN warp columns.
template <int RPT, int WCN, int CPT>
struct Shape {
    static constexpr int GS = RPT > 4 ? 8 : RPT > 2 ? 4 : RPT;   // slots of a walker group
    static constexpr int GROUPS = 2 * (8 / WCN);                 // walker groups of a CTA
    static constexpr int R = GROUPS * RPT;                       // walkers of a CTA
    static constexpr int SLOTS = GROUPS * GS;
    static constexpr int LD = SLOTS + 4;                         // floats of a shared row
    static constexpr int COLS = 16 * CPT * WCN;                  // output neurons
    // weight rows per ring stage: 32 KB a stage (16 rows of 256 columns cost 84 us where 32 cost
    // 78, for twice the block barriers); short tiles, whose rows are consumed faster than one
    // stage ahead arrives, keep more stages
    static constexpr int KC = WCN == 4 ? 16 : 32;
    static constexpr int NSW = RPT <= 2 ? 4 : 2;
};
__host__ __device__ constexpr int shape_gs(int rpt) { return rpt > 4 ? 8 : rpt > 2 ? 4 : rpt; }

// Shared memory of a tile, bytes: activations (and, for a residual gradient, g_l
// beside them), the inputs, the weight ring.
size_t tile_smem(int rpt, int wcn, int cpt, int D, int H, int resnet, bool bwd) {
    const int slots = 2 * (8 / wcn) * shape_gs(rpt), ld = slots + 4;
    const int kc = wcn == 4 ? 16 : 32, nsw = rpt <= 2 ? 4 : 2;
    return sizeof(float) * ((size_t)(bwd && resnet ? 2 : 1) * H * ld + (size_t)D * ld + (size_t)nsw * kc * 16 * cpt * wcn);
}

// Where a thread's outputs lie: walker group, column base of its warp.
struct Lane {
    int rg, lc, wc;
};
template <int WCN>
__device__ __forceinline__ Lane lane_of() {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    return Lane{(warp / WCN) * 2 + (lane >> 4), lane & 15, warp % WCN};
}
// Column j (0 .. CPT - 1) of a thread within a pass.
template <int CPT>
__device__ __forceinline__ int col_of(const Lane& t, int j) {
    if (CPT == 2) return 32 * t.wc + 2 * t.lc + j;
    return 16 * CPT * t.wc + (j < 4 ? 4 * t.lc + j : 64 + 4 * t.lc + j - 4);
}

// The RPT values of a walker group at p (GS slots, aligned to them).
template <int RPT>
__device__ __forceinline__ void load_group(const float* p, float (&v)[RPT]) {
    constexpr int GS = shape_gs(RPT);
    float t[GS];
    if constexpr (GS >= 4) {
#pragma unroll
        for (int q = 0; q < GS / 4; ++q) {
            const float4 a = *reinterpret_cast<const float4*>(p + 4 * q);
            t[4 * q] = a.x, t[4 * q + 1] = a.y, t[4 * q + 2] = a.z, t[4 * q + 3] = a.w;
        }
    } else if constexpr (GS == 2) {
        const float2 a = *reinterpret_cast<const float2*>(p);
        t[0] = a.x, t[1] = a.y;
    } else {
        t[0] = *p;
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) v[i] = t[i];
}
template <int RPT>
__device__ __forceinline__ void store_group(float* p, const float (&v)[RPT]) {
    constexpr int GS = shape_gs(RPT);
    float t[GS];
#pragma unroll
    for (int i = 0; i < GS; ++i) t[i] = i < RPT ? v[i < RPT ? i : 0] : 0.0f;
    if constexpr (GS >= 4) {
#pragma unroll
        for (int q = 0; q < GS / 4; ++q)
            *reinterpret_cast<float4*>(p + 4 * q) = make_float4(t[4 * q], t[4 * q + 1], t[4 * q + 2], t[4 * q + 3]);
    } else if constexpr (GS == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(t[0], t[1]);
    } else {
        *p = t[0];
    }
}

// The weight rows of one pass: K rows of ldw floats from W on, whose first
// `ncol` columns are loaded (vec: a multiple of 4 with 16-byte aligned rows) and
// whose first `nuse` are wanted.
struct Stream {
    const float* W;
    int K, ldw, ncol, nuse;
    bool vec;
};
template <typename S>
__device__ __forceinline__ void ring_issue(const Stream& q, int st, float* ws) {
    constexpr int KC = S::KC, COLS = S::COLS, NSW = S::NSW;
    const int kn = q.K - st * KC < KC ? q.K - st * KC : KC;
    if (kn > 0) {
        float* dst = ws + (st % NSW) * KC * COLS;
        const float* src = q.W + (size_t)st * KC * q.ldw;
        if (q.vec) {
#pragma unroll
            for (int e = threadIdx.x; e < KC * COLS / 4; e += NT) {
                const int r = e / (COLS / 4), c = 4 * (e % (COLS / 4));
                if (r < kn && c < q.ncol) cpa16(dst + r * COLS + c, src + (size_t)r * q.ldw + c);
            }
        } else {
            for (int e = threadIdx.x; e < KC * COLS; e += NT) {
                const int r = e / COLS, c = e % COLS;
                if (r < kn && c < q.ncol) cpa4(dst + r * COLS + c, src + (size_t)r * q.ldw + c, 4);
            }
        }
    }
    cpa_commit();
}
// The first stages of a pass; the ring must be free.
template <typename S>
__device__ __forceinline__ void ring_prime(const Stream& q, float* ws) {
#pragma unroll
    for (int st = 0; st < S::NSW - 1; ++st) ring_issue<S>(q, st, ws);
}

// acc[i][j] += sum_k in[k][walker i] * W[k][column j] for a primed pass, every
// accumulator over k in increasing order.  SPLIT sums the K tiles of 32 with
// even and odd index in acc and acc1.  Ends with every warp past its last read
// of `in` and of the ring.
template <int RPT, int WCN, int CPT, bool SPLIT>
__device__ __forceinline__ void tile_gemm(const float* in, const Stream& q, const Lane& t, f32x2 (&acc)[RPT][CPT / 2],
                                          f32x2 (&acc1)[SPLIT ? RPT : 1][CPT / 2], float* ws) {
    using S = Shape<RPT, WCN, CPT>;
    constexpr int KC = S::KC, COLS = S::COLS, NSW = S::NSW;
    const int nst = (q.K + KC - 1) / KC;
    const bool use = 16 * CPT * t.wc < q.nuse;    // warp-uniform: some column of this warp is wanted
    auto stage = [&](int st, f32x2(&a)[RPT][CPT / 2]) {
        const float* wsr = ws + (st % NSW) * KC * COLS + 16 * CPT * t.wc + (CPT == 2 ? 2 : 4) * t.lc;
        const float* ar = in + (size_t)st * KC * S::LD + t.rg * S::GS;
        const int kn = q.K - st * KC < KC ? q.K - st * KC : KC;
        auto row = [&](int r) {
            float av[RPT];
            load_group<RPT>(ar + r * S::LD, av);
            f32x2 w[CPT / 2];
            if constexpr (CPT == 2) {
                w[0] = *reinterpret_cast<const f32x2*>(wsr + r * COLS);
            } else {
#pragma unroll
                for (int h = 0; h < CPT / 4; ++h) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wsr + r * COLS + 64 * h);
                    w[2 * h] = v.x;
                    w[2 * h + 1] = v.y;
                }
            }
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const f32x2 d = pack2(av[i], av[i]);
#pragma unroll
                for (int h = 0; h < CPT / 2; ++h) fma2(a[i][h], d, w[h]);
            }
        };
        if (kn == KC) {
#pragma unroll
            for (int r = 0; r < KC; ++r) row(r);
        } else {
            for (int r = 0; r < kn; ++r) row(r);
        }
    };
    for (int st = 0; st < nst; ++st) {
        cpa_wait<NSW - 2>();
        __syncthreads();
        ring_issue<S>(q, st + NSW - 1, ws);
        if (use) {
            if constexpr (SPLIT) {
                if ((st * KC / 32) & 1) stage(st, acc1);
                else stage(st, acc);
            } else {
                stage(st, acc);
            }
        }
    }
    cpa_wait<0>();
    __syncthreads();
}

// BWD: the input gradient as well; else the member values alone.
template <int RPT, int WCN, int CPT, bool BWD, bool SPLIT>
__global__ void __launch_bounds__(NT, RPT >= 4 && CPT == 8 ? 1 : 2) k_mlp_fp32(MlpF32 E) {
    static_assert(CPT == 8 || !BWD, "the input gradient takes eight columns a thread");
    using S = Shape<RPT, WCN, CPT>;
    constexpr int GS = S::GS, LD = S::LD, R = S::R;
    extern __shared__ __align__(16) float sm[];
    const int D = E.D, L = E.L, H = E.H, W = E.W;
    float* X = sm;                                      // current activations, then delta_l  [H][LD]
    float* Y = X + (size_t)(BWD && E.resnet ? H : 0) * LD;   // g_l (residual gradient)          [H][LD]
    float* ubuf = Y + (size_t)H * LD;
    float* ws = ubuf + (size_t)D * LD;                  // weight ring [NSW][KC][COLS]
    const int m = blockIdx.y, w0 = blockIdx.x * R;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Lane t = lane_of<WCN>();
    const int own = t.rg * GS;                          // this thread's slots of a row
    // saved tanh: rows of the tile's slots; a last tile of 64 that holds 32 walkers or fewer keeps half of them
    constexpr bool halves = RPT == 8 && R == 64;
    const int tw = halves && W - w0 <= 32 ? 32 : S::SLOTS;
    const bool keep = !halves || own < tw;
    const size_t wst = RPT == 7 ? (size_t)gridDim.x * S::SLOTS : f32_walkers(W);
    float* hs = BWD ? E.hs + (m * wst + (size_t)blockIdx.x * S::SLOTS) * (size_t)L * H + own : nullptr;

    // the passes in order: forward layers, then (BWD) gradient layers L - 1 .. 0
    const int npass = BWD ? 2 * L : L;
    auto stream = [&](int p) {
        Stream q{};
        if (p >= npass) return q;
        if (p < L) {
            q.W = E.WT + (long long)m * E.wt_st + E.toff[p];
            q.K = p == 0 ? D : H;
            q.ldw = q.ncol = E.ldt;
            q.nuse = H;
            q.vec = true;
        } else {
            const int l = 2 * L - 1 - p;
            q.W = E.Wb + (long long)m * E.wb_st + E.woff[l];   // [H][fin] row-major = [K][Nout]
            q.K = H;
            q.ldw = q.ncol = q.nuse = l == 0 ? D : H;
            q.vec = (q.ldw & 3) == 0 && (reinterpret_cast<uintptr_t>(q.W) & 15) == 0;
        }
        return q;
    };
    int pass = 0;
    Stream cur = stream(0);
    ring_prime<S>(cur, ws);
    auto next_pass = [&]() {
        cur = stream(++pass);
        ring_prime<S>(cur, ws);
    };

    for (int idx = threadIdx.x; idx < D * R; idx += NT) {
        const int r = idx / D, k = idx - r * D;
        ubuf[k * LD + (r / RPT) * GS + r % RPT] = (w0 + r < W) ? E.u[(size_t)(w0 + r) * D + k] : 0.0f;
    }
    __syncthreads();

    f32x2 acc1[SPLIT ? RPT : 1][CPT / 2];
    // value (i, j) of an accumulator set
    auto value = [](const f32x2(&a)[RPT][CPT / 2], int i, int j) {
        float lo, hi;
        unpack2(a[i][j >> 1], lo, hi);
        return (j & 1) ? hi : lo;
    };
    // ---------------- forward
    for (int l = 0; l < L; ++l) {
        const float* bias = E.b + (long long)m * E.b_st + E.boff[l];
        f32x2 acc[RPT][CPT / 2];
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
            for (int j = 0; j < CPT / 2; ++j) acc[i][j] = 0ull;
        if constexpr (SPLIT)
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int j = 0; j < CPT / 2; ++j) acc1[i][j] = 0ull;
        tile_gemm<RPT, WCN, CPT, SPLIT>(l == 0 ? ubuf : X, cur, t, acc, acc1, ws);
        next_pass();
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int n = col_of<CPT>(t, j);
            if (n < H) {
                const float bn = bias[n];
                float tv[RPT], h[RPT];
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    float z = value(acc, i, j);
                    if constexpr (SPLIT) z += value(acc1, i, j);
                    tv[i] = tanhf(z + bn);
                }
                if (BWD && keep) store_group<RPT>(hs + ((size_t)l * H + n) * tw, tv);
                if (E.resnet && l > 0) {
                    load_group<RPT>(X + (size_t)n * LD + own, h);
#pragma unroll
                    for (int i = 0; i < RPT; ++i) h[i] = tv[i] + h[i];
                    store_group<RPT>(X + (size_t)n * LD + own, h);
                } else {
                    store_group<RPT>(X + (size_t)n * LD + own, tv);
                }
            }
        }
        __syncthreads();
    }
    // value A = w_out . h_L + b_out: lane-strided partial sums, then the butterfly
    const float* wo = E.wout + (long long)m * E.wo_st;
    for (int r = warp; r < R; r += NT / 32) {
        if (w0 + r >= W) break;
        const float* hr = X + (r / RPT) * GS + r % RPT;
        float part = 0.0f;
        for (int n = lane; n < H; n += 32) part = fmaf(wo[n], hr[(size_t)n * LD], part);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) E.Aval[(size_t)m * W + w0 + r] = part + E.bout[(long long)m * E.bo_st];
    }
    if constexpr (BWD) {
        auto load_kept = [&](const float* p, float(&v)[RPT]) {
            if (keep) {
                load_group<RPT>(p, v);
            } else {
#pragma unroll
                for (int i = 0; i < RPT; ++i) v[i] = 0.0f;
            }
        };
        // ---------------- backward: X holds delta_l, Y g_l of this thread's own columns
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int n = col_of<8>(t, j);
            if (n < H) {
                const float wn = wo[n];
                float tv[RPT], g[RPT];
                load_kept(hs + ((size_t)(L - 1) * H + n) * tw, tv);
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    g[i] = wn;
                    tv[i] = wn * (1.0f - tv[i] * tv[i]);
                }
                store_group<RPT>(X + (size_t)n * LD + own, tv);
                if (E.resnet) store_group<RPT>(Y + (size_t)n * LD + own, g);
            }
        }
        __syncthreads();
        for (int l = L - 1; l >= 0; --l) {
            const bool res = E.resnet && l > 0;
            f32x2 acc[RPT][4];
            float g[RPT][8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int n = col_of<8>(t, j);
                float v[RPT];
                if (res && n < H) load_group<RPT>(Y + (size_t)n * LD + own, v);
#pragma unroll
                for (int i = 0; i < RPT; ++i) g[i][j] = res && n < H ? v[i] : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = pack2(g[i][2 * j], g[i][2 * j + 1]);
            tile_gemm<RPT, WCN, CPT, false>(X, cur, t, acc, acc1, ws);
            next_pass();
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) g[i][j] = value(acc, i, j);
            if (l > 0) {
                // g_{l-1}, and its delta over delta_l
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = col_of<8>(t, j);
                    if (n >= H) continue;
                    float v[RPT], tv[RPT];
                    load_kept(hs + ((size_t)(l - 1) * H + n) * tw, tv);
#pragma unroll
                    for (int i = 0; i < RPT; ++i) v[i] = g[i][j];
                    if (E.resnet) store_group<RPT>(Y + (size_t)n * LD + own, v);
#pragma unroll
                    for (int i = 0; i < RPT; ++i) v[i] = v[i] * (1.0f - tv[i] * tv[i]);
                    store_group<RPT>(X + (size_t)n * LD + own, v);
                }
                __syncthreads();
            } else {
                // dA/ds_j = -sin s_j g0[2j] + cos s_j g0[2j+1] (torsion), g0[2j] (distance: input (s, 0))
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int n = col_of<8>(t, 2 * q), j = n >> 1;
                    if (n >= D) continue;
                    const bool dist = E.cvdist && __ldg(E.cvdist + j);
                    float cs[RPT], sn[RPT];
                    load_group<RPT>(ubuf + (size_t)n * LD + own, cs);
                    load_group<RPT>(ubuf + (size_t)(n + 1) * LD + own, sn);
#pragma unroll
                    for (int i = 0; i < RPT; ++i) {
                        const int wg = w0 + t.rg * RPT + i;
                        const float G0 = g[i][2 * q], G1 = g[i][2 * q + 1];
                        const float gr = dist ? G0 : -sn[i] * G0 + cs[i] * G1;
                        if (wg < W) E.gradA[((size_t)m * W + wg) * E.C + j] = gr;
                    }
                }
            }
        }
    }
}

// Walkers per thread: the tile whose waves of CTAs over the SMs cost least,
// counting a K row at the larger of its FMA cycles (16 RPT) and its shared loads
// (40), plus 8 for what does not overlap; of those that fit in shared memory.
// Two walkers always fit.  compact: not seven, whose rows of saved tanh are an
// eighth padding: a server's jobs, whose scratch counts against its budget.  (Rows
// of seven without padding cost everyone: 4200 -> 4330 us for 20 steps of 1500
// walkers with 16-, 8- and 4-byte accesses, 4716 with 4-byte ones.)
int choose_rpt(int wcn, int cpt, int W, int M, int D, int H, int resnet, bool bwd, bool compact) {
    static int nsm[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
    int& n = nsm[dev & 63];
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 152;
    int best = 2;
    long long cost = -1;
    for (int rpt : {2, 4, 7, 8}) {
        if (compact && rpt == 7) continue;
        if (tile_smem(rpt, wcn, cpt, D, H, resnet, bwd) > (size_t)F32_SMEM_MAX) continue;
        const int R = 2 * (8 / wcn) * rpt;
        const long long ctas = (long long)((W + R - 1) / R) * M;
        const long long c = (ctas + n - 1) / n * (std::max(2 * cpt * rpt, 40) + 8);
        if (cost < 0 || c <= cost) {
            cost = c;
            best = rpt;
        }
    }
    return best;
}

template <int RPT, int WCN, int CPT, bool BWD, bool SPLIT>
void launch_f32(const MlpF32& E, int M, cudaStream_t s) {
    static RidOnce once;
    auto k = k_mlp_fp32<RPT, WCN, CPT, BWD, SPLIT>;
    rid_opt_in(once, F32_SMEM_MAX, k);
    constexpr int R = Shape<RPT, WCN, CPT>::R;
    k<<<dim3((E.W + R - 1) / R, M), NT, tile_smem(RPT, WCN, CPT, E.D, E.H, E.resnet, BWD), s>>>(E);
}

// Small ensembles (every layer of a member fits in shared memory at once, as
// for widths up to about 96): one CTA per (tile of 32 walkers, member) loads
// the member's weights once -- rows of W_l [H][fin] padded to fin + 1 floats,
// so the lanes of a warp (consecutive output neurons) read distinct banks --
// and runs every layer from shared memory, with no weight ring to wait on.
// The operations are those of k_mlp_fp32 in the same order: each forward
// output is the FMA chain over its K inputs in increasing order from zero,
// then + b and tanh; each input-gradient output starts from the residual term
// (or zero) and chains over the H outputs of the layer in increasing order;
// the member value is the same lane-strided partial sums and butterfly.
constexpr int SM_MAX_FLOATS = 50 * 1024;   // 200 KB of shared memory
constexpr int SM_MAX_WIDTH = 128;          // at least two walker groups per neuron
constexpr int SR_MAX = 32 / (NT / SM_MAX_WIDTH);   // walkers per thread at the widest layer: 16

struct SmallLayout {
    int woff[RID_MAX_LAYERS + 1];
    int bias, wout, u, t, h0, h1, G0, G1, total;
};
__host__ __device__ inline SmallLayout small_layout(int D, int L, int H, int resnet, int TW) {
    SmallLayout S{};
    int o = 0;
    for (int l = 0; l < L; ++l) {
        S.woff[l] = o;
        o += H * ((l == 0 ? D : H) + 1);
    }
    S.woff[L] = o;
    S.bias = o; o += L * H;
    S.wout = o; o += H;
    S.u = o;    o += TW * D;
    S.t = o;    o += L * TW * H;
    S.h0 = o;   o += resnet ? TW * H : 0;
    S.h1 = o;   o += resnet ? TW * H : 0;
    const int gw = H > D ? H : D;
    S.G0 = o;   o += TW * gw;
    S.G1 = o;   o += TW * gw;
    S.total = o;
    return S;
}

// Offset of layer l's padded weight rows (the same as SmallLayout::woff, in registers).
__device__ __forceinline__ int small_woff(int D, int H, int l) { return l == 0 ? 0 : H * (D + 1) + (l - 1) * H * (H + 1); }

// TW: walkers per CTA (1 .. 32), chosen by the launcher so that small walker
// counts still spread over many SMs; SR: a power of two bounding the walkers
// one thread carries (ceil(TW / (NT / H)) at most).
template <int SR>
__global__ void __launch_bounds__(NT) k_mlp_fp32_small(EnsDev E, StateDev st, int W, int C, int TW) {
    extern __shared__ __align__(16) float sm[];
    const int D = E.D, L = E.L, H = E.H;
    const SmallLayout Y = small_layout(D, L, H, E.resnet, TW);
    const int m = blockIdx.y, w0 = blockIdx.x * TW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float* Wm = E.W + (size_t)m * E.wstride;
    // the member's weights: every copy in flight at once, one wait
    for (int l = 0; l < L; ++l) {
        const int fin = l == 0 ? D : H;
        const float* Wl = Wm + E.loff[l];
        for (int idx = threadIdx.x; idx < H * fin; idx += NT) {
            const int n = idx / fin, k = idx - n * fin;
            cpa4(sm + small_woff(D, H, l) + n * (fin + 1) + k, Wl + idx, 4);
        }
    }
    cpa_commit();
    for (int idx = threadIdx.x; idx < L * H; idx += NT) sm[Y.bias + idx] = __ldg(E.b + (size_t)m * L * H + idx);
    for (int idx = threadIdx.x; idx < H; idx += NT) sm[Y.wout + idx] = __ldg(E.wout + (size_t)m * H + idx);
    for (int idx = threadIdx.x; idx < TW * D; idx += NT) {
        const int wl = idx / D, k = idx - wl * D;
        sm[Y.u + idx] = (w0 + wl < W) ? st.u[(size_t)(w0 + wl) * D + k] : 0.0f;
    }
    cpa_wait<0>();
    __syncthreads();
    // forward: t_l = tanh(in W_l^T + b_l), h_l = t_l (+ h_{l-1} for a residual layer)
    const float* in = sm + Y.u;
    for (int l = 0; l < L; ++l) {
        const int K = l == 0 ? D : H;
        const float* Wl = sm + small_woff(D, H, l);
        float* tl = sm + Y.t + l * TW * H;
        const bool res = E.resnet && l > 0;
        float* hout = E.resnet ? sm + ((l & 1) ? Y.h1 : Y.h0) : tl;
        // thread -> neuron n and walkers g, g + P, ...: one weight read per k
        // serves SR independent chains
        const int P = NT / H, n = threadIdx.x % H, g = threadIdx.x / H;
        if (g < P) {
            float acc[SR];
#pragma unroll
            for (int r = 0; r < SR; ++r) acc[r] = 0.0f;
            const float* wr = Wl + n * (K + 1);
            for (int k = 0; k < K; ++k) {
                const float wv = wr[k];
#pragma unroll
                for (int r = 0; r < SR; ++r)
                    if (g + P * r < TW) acc[r] = fmaf(in[(g + P * r) * K + k], wv, acc[r]);
            }
            const float bn = sm[Y.bias + l * H + n];
#pragma unroll
            for (int r = 0; r < SR; ++r) {
                const int wl = g + P * r;
                if (wl < TW) {
                    const float t = tanhf(acc[r] + bn);
                    tl[wl * H + n] = t;
                    if (E.resnet) hout[wl * H + n] = res ? t + in[wl * K + n] : t;
                }
            }
        }
        __syncthreads();
        in = hout;
    }
    // member value A = w_out . h_L + b_out: lane-strided partials, then the butterfly
    for (int wl = warp; wl < TW; wl += NT / 32) {
        float part = 0.0f;
        for (int n = lane; n < H; n += 32) part = fmaf(sm[Y.wout + n], in[wl * H + n], part);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0 && w0 + wl < W) st.Aval[(size_t)m * W + w0 + wl] = part + E.bout[m];
    }
    // input gradient: g_L = w_out, Delta_l = g_l (1 - t_l^2), g_{l-1} = Delta_l W_l (+ g_l)
    float* G = sm + Y.G0;
    float* Gn = sm + Y.G1;
    for (int o = threadIdx.x; o < TW * H; o += NT) G[o] = sm[Y.wout + (o % H)];
    __syncthreads();
    for (int l = L - 1; l >= 0; --l) {
        const int Nout = l == 0 ? D : H, fin = Nout;
        const float* tl = sm + Y.t + l * TW * H;
        const float* Wl = sm + small_woff(D, H, l);
        const bool res = E.resnet && l > 0;
        float* Dl = Gn;   // Delta_l in the free buffer, then g_{l-1} over G
        for (int o = threadIdx.x; o < TW * H; o += NT) {
            const float t = tl[o];
            Dl[o] = G[o] * (1.0f - t * t);
        }
        __syncthreads();
        // g_{l-1}[j] = (g_l[j] if residual) + sum_k Delta_l[k] W_l[k][j], written over G after all reads
        // thread -> input j and walkers g, g + P, ... (P = NT / Nout groups, at most TW)
        {
            const int P = NT / Nout < TW ? NT / Nout : TW, j = threadIdx.x % Nout, g = threadIdx.x / Nout;
            float acc[SR];
            const bool act = g < P;
#pragma unroll
            for (int r = 0; r < SR; ++r) {
                const int wl = g + P * r;
                acc[r] = (act && wl < TW && res) ? G[wl * H + j] : 0.0f;
            }
            if (act)
                for (int k = 0; k < H; ++k) {
                    const float wv = Wl[k * (fin + 1) + j];
#pragma unroll
                    for (int r = 0; r < SR; ++r)
                        if (g + P * r < TW) acc[r] = fmaf(Dl[(g + P * r) * H + k], wv, acc[r]);
                }
            __syncthreads();   // every thread has read G for its initial values
            if (act)
#pragma unroll
                for (int r = 0; r < SR; ++r) {
                    const int wl = g + P * r;
                    if (wl < TW) G[wl * (l == 0 ? D : H) + j] = acc[r];
                }
            __syncthreads();
        }
    }
    // dA/ds_j = -sin s_j g0[2j] + cos s_j g0[2j+1] (torsion), g0[2j] (distance: input (s, 0))
    for (int idx = threadIdx.x; idx < C * TW; idx += NT) {
        const int wl = idx / C, j = idx - wl * C;
        const int wg = w0 + wl;
        if (wg < W) {
            const float cs = sm[Y.u + wl * D + 2 * j], sn = sm[Y.u + wl * D + 2 * j + 1];
            const float* g0 = G + wl * D;
            const bool dist = E.cvdist && __ldg(E.cvdist + j);
            st.gradA[((size_t)m * W + wg) * C + j] = dist ? g0[2 * j] : -sn * g0[2 * j] + cs * g0[2 * j + 1];
        }
    }
}

}  // namespace

// The small kernel's walkers per CTA for this call, 0 when it does not apply:
// the largest power of two up to 32 that still gives one wave of CTAs.
static int small_tile(const EnsDev& E, int W) {
    if (E.H > SM_MAX_WIDTH || E.D > NT || small_layout(E.D, E.L, E.H, E.resnet, 32).total > SM_MAX_FLOATS) return 0;
    int tw = 32;
    while (tw > 1 && (long long)((W + tw - 1) / tw) * E.M < 152) tw >>= 1;
    return tw;
}

// Rounded up over every tile shape, so that it grows with W: a system keeps the
// scratch of its largest walker count.  (Groups of seven take eight slots.)
size_t rid_mlp_fp32_scratch_floats(const EnsDev& E, int W, bool compact) {
    return (size_t)E.M * E.L * E.H * (compact ? f32_walkers(W) : (size_t)(W + 27) / 28 * 32 + 64);
}

// The kernel for a width, walkers per thread chosen.
template <int WCN, int CPT, bool BWD, bool SPLIT>
static void launch_shape(const MlpF32& E, int M, cudaStream_t s) {
    switch (choose_rpt(WCN, CPT, E.W, M, E.D, E.H, E.resnet, BWD, BWD && E.compact)) {
        case 2: return launch_f32<2, WCN, CPT, BWD, SPLIT>(E, M, s);
        case 4: return launch_f32<4, WCN, CPT, BWD, SPLIT>(E, M, s);
        case 7: return launch_f32<7, WCN, CPT, BWD, SPLIT>(E, M, s);
        default: return launch_f32<8, WCN, CPT, BWD, SPLIT>(E, M, s);
    }
}
// (Widths to 32 and 64 with eight columns a thread, three quarters or half of them for nothing: 20 steps of 100000
// walkers of 4 x 40-32x4-1 13.7 ms, 6.4 with two; 20000 walkers at width 64 4.16 -> 2.65 ms.  One GEMM a layer, as
// it was before, took 10.1 and 4.09 ms.)
template <bool SPLIT>
static void launch_values(const MlpF32& E, int M, cudaStream_t s) {
    if (E.H <= 32) launch_shape<1, 2, false, SPLIT>(E, M, s);
    else if (E.H <= 64) launch_shape<1, 4, false, SPLIT>(E, M, s);
    else if (E.H <= 128) launch_shape<1, 8, false, SPLIT>(E, M, s);
    else if (E.H <= 256) launch_shape<2, 8, false, SPLIT>(E, M, s);
    else launch_shape<4, 8, false, SPLIT>(E, M, s);
}

void rid_launch_mlp_fp32(const EnsDev& E, StateDev st, int W, int C, cudaStream_t s, bool values_only, bool compact) {
    if (const int tw = small_tile(E, W)) {
        const SmallLayout Y = small_layout(E.D, E.L, E.H, E.resnet, tw);
        const int wpt = (tw + NT / E.H - 1) / (NT / E.H);
        int sr = 1;
        while (sr < wpt) sr <<= 1;
        auto kern = sr == 1 ? k_mlp_fp32_small<1> : sr == 2 ? k_mlp_fp32_small<2> : sr == 4 ? k_mlp_fp32_small<4>
                  : sr == 8 ? k_mlp_fp32_small<8> : k_mlp_fp32_small<SR_MAX>;
        static RidOnce once;
        rid_opt_in(once, SM_MAX_FLOATS * 4, k_mlp_fp32_small<1>, k_mlp_fp32_small<2>, k_mlp_fp32_small<4>,
                   k_mlp_fp32_small<8>, k_mlp_fp32_small<SR_MAX>);
        kern<<<dim3((W + tw - 1) / tw, E.M), NT, (size_t)Y.total * sizeof(float), s>>>(E, st, W, C, tw);
        return;
    }
    MlpF32 A{};
    A.WT = E.WT;
    A.Wb = E.W;
    A.wt_st = A.wb_st = E.wstride;
    A.ldt = E.H;
    A.b = E.b;
    A.b_st = (long long)E.L * E.H;
    for (int l = 0; l < E.L; ++l) {
        A.toff[l] = A.woff[l] = E.loff[l];
        A.boff[l] = (long long)l * E.H;
    }
    A.wout = E.wout;
    A.wo_st = E.H;
    A.bout = E.bout;
    A.bo_st = 1;
    A.u = st.u;
    A.D = E.D;
    A.L = E.L;
    A.H = E.H;
    A.resnet = E.resnet;
    A.W = W;
    A.C = C;
    A.hs = st.hs;
    A.compact = compact;
    A.Aval = st.Aval;
    A.gradA = st.gradA;
    A.cvdist = E.cvdist;
    if (values_only) launch_values<false>(A, E.M, s);
    else if (E.H <= 256) launch_shape<2, 8, true, false>(A, E.M, s);
    else launch_shape<4, 8, true, false>(A, E.M, s);
}

void rid_launch_mlp_values(const MlpF32& E, int M, bool split, cudaStream_t s) {
    if (split) launch_values<true>(E, M, s);
    else launch_values<false>(E, M, s);
}
