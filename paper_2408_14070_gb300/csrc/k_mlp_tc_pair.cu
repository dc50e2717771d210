// k_mlp_tc_pair.cu -- the tcgen05 ensemble MLP on CTA pairs (cta_group::2).
//
// Same arithmetic and data layout as k_mlp_tc (BF16 / FP8 operands, FP32
// accumulation in TMEM, tanh saved in BF16, optional FP32 residual stream,
// member values from 16-column partials in column order), and the same warp
// roles: warp 0 TMA producer, warp 1 TMEM allocator and MMA issuer (the pair's
// even CTA only), warps 2..17 epilogue.  A cluster of two CTAs runs one member
// for 2 x ROWS walkers: each CTA keeps ROWS rows of the activations in its
// shared memory and streams half of every weight chunk's rows, and one
// tcgen05.mma of the even CTA multiplies both CTAs' rows by both halves.
// Every wait on an mbarrier is bounded in time (the TMEM allocation, which waits for
// CTAs that hold columns to end, and the cluster barriers are not).
//
// A GEMM is a serial chain: MMAs, accumulator to the epilogue, element work,
// operand back to the MMAs.  At 512 columns the 128 KB operand left room for
// two 32 KB weight stages a CTA, so the stream from L2 bounded the MMAs, and
// 16-column steps of 200 instructions with one load in flight the epilogue.
// In a pair a stage is half as large (five fit, and L2 is read half as often);
// the epilogue takes 16 columns per TMEM load, two FP32 operations an
// instruction, the saved tanh two steps ahead, keeps the residual stream in
// TMEM where two accumulators fit, and saves a plain BF16 layer's tanh from the
// operand tile after releasing it, while the MMAs run.  The release to the
// even CTA orders shared memory alone (pair_arrive).
// Measured per launch, one CTA per 128 walkers before -> pairs of 128 rows:
// 8 x 64-512x4-1 at 8192 walkers 436 -> 315 us (682 of 1873 TFLOP/s), 4 x
// 40-256x4-1 at 8192 walkers 79 -> 73 us, residual 127 -> 94 us; pairs of 64 rows,
// 1024 walkers of 4 x 40-256x4-1, 39 -> 31 us.  What is left is the chain.  Of 86 us
// for one wave at 512 columns (2048 walkers), 75 remain without the MMAs, 59 without
// the epilogue, 38 without both and the weights: hand-overs, saves and the call's
// ends.  Measured and not kept: the second 256 columns' MMAs under the first's
// epilogue, its results parked in TMEM (319 -> 310 us, and 5% slower to 256 columns).
#include "rid_pair_loads.cuh"
#include "rid_tc_ptx.cuh"

namespace {

struct Smem {
    uint64_t full[TC_MAX_STAGES];    // even CTA: both halves of a weight stage have landed
    uint64_t empty[TC_MAX_STAGES];   // both CTAs: the MMAs that read the stage have completed
    uint64_t acc_full;               // both CTAs: the GEMM's accumulator is complete
    uint64_t a_full;                 // even CTA: the next operand is complete (epilogue warps of both CTAs)
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;                  // of this CTA, at the end of either CTA
    int issued;                      // weight iterations whose part this CTA has issued
    int odd_issued;                  // even CTA: the odd CTA's
};

constexpr uint32_t PAIR_STAGE = 128u * 128u;   // half of a 256-row weight chunk
// A pair must not hold one SM's TMEM while its other half waits for columns that a CTA of another cluster
// holds, whose own half may wait for the first SM's.  So the columns of what can share an SM add up to 512 at
// most: one pair's CTA per SM, and with more than 256 columns nothing else that uses TMEM (no kernel that does
// fits beside PAIR_SMEM_MAX).
constexpr size_t PAIR_SMEM_MIN = 116 * 1024, PAIR_SMEM_MAX = 225 * 1024;

__device__ __forceinline__ void pair_mma(bool f8, uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
    if (f8)
        asm volatile(
            "{ .reg .pred p; setp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p; }" ::"r"(d),
            "l"(a), "l"(b), "r"(id), "r"(acc)
            : "memory");
    else
        asm volatile(
            "{ .reg .pred p; setp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d),
            "l"(a), "l"(b), "r"(id), "r"(acc)
            : "memory");
}
// Arrive on the barrier at this offset in both CTAs of the pair once every MMA issued so far has completed.
__device__ __forceinline__ void pair_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}
// Weight rows into this CTA's shared memory, counted on a barrier of the pair's even CTA.
__device__ __forceinline__ void pair_tma_load(uint32_t dst, const CUtensorMap* map, int row, uint32_t leader_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(leader_bar)
        : "memory");
}
// Hand this CTA's rows of an operand to the even CTA, whose MMAs read them: release at cluster scope of
// shared memory alone, before a relaxed arrive (the writers have handed it to the async proxy already).  An
// arrive that releases all memory costs half a microsecond a GEMM here, also from a thread that has written
// nothing: 30.5 -> 34.2 us a launch (128 walkers of 4 x 40-256x4-1), 30.6 with this fence.  (The default scope
// took 0.4 us less of a step's 49.8, 1024 walkers of 200 beads, and orders the arriving CTA only, which is why
// the even CTA's own rows take it: with the fence in both CTAs a step took 50.1 us.)
__device__ __forceinline__ void pair_arrive(uint32_t local_bar, uint32_t rank) {
    if (rank == 0) {                  // its own rows: the reader is in this CTA
        mbar_arrive(local_bar);
        return;
    }
    asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(mapa(local_bar, 0)) : "memory");
}
// The even CTA's wait for it: relaxed, then an acquire of shared memory alone.
__device__ __forceinline__ bool pair_try(uint32_t a, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void pair_acquire() {
    asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
}
// Sixteen 32-bit columns of this thread's TMEM lane, from or to registers.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"r"(
            r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Two FP32 operations an instruction.
__device__ __forceinline__ uint64_t pk2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// g (1 - t^2) for 16 columns, t in BF16
__device__ __forceinline__ void tanh_back(float (&g)[16], const uint4 (&t)[2]) {
    const uint32_t u[8] = {t[0].x, t[0].y, t[0].z, t[0].w, t[1].x, t[1].y, t[1].z, t[1].w};
    const uint64_t one = pk2(1.0f, 1.0f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float lo = __uint_as_float(u[i] << 16), hi = __uint_as_float(u[i] & 0xFFFF0000u);
        const uint64_t q = fma2(pk2(-lo, -hi), pk2(lo, hi), one);
        upk2(mul2(pk2(g[2 * i], g[2 * i + 1]), q), g[2 * i], g[2 * i + 1]);
    }
}
__device__ __forceinline__ void pack16(const float (&v)[16], uint4 (&o)[2]) {
    o[0] = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    o[1] = make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]), pack_bf16(v[12], v[13]), pack_bf16(v[14], v[15]));
}
__device__ __forceinline__ void unpack16(const uint4 (&t)[2], float (&v)[16]) {
    const uint32_t u[8] = {t[0].x, t[0].y, t[0].z, t[0].w, t[1].x, t[1].y, t[1].z, t[1].w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    }
}
// a += p for 16 consecutive floats of shared memory (a warp reads the same ones: broadcast)
__device__ __forceinline__ void add16(float (&a)[16], const float* p) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 b = reinterpret_cast<const float4*>(p)[i];
        upk2(add2(pk2(a[4 * i], a[4 * i + 1]), pk2(b.x, b.y)), a[4 * i], a[4 * i + 1]);
        upk2(add2(pk2(a[4 * i + 2], a[4 * i + 3]), pk2(b.z, b.w)), a[4 * i + 2], a[4 * i + 3]);
    }
}
__device__ __forceinline__ void ld16(const float* p, float (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 b = reinterpret_cast<const float4*>(p)[i];
        v[4 * i] = b.x;
        v[4 * i + 1] = b.y;
        v[4 * i + 2] = b.z;
        v[4 * i + 3] = b.w;
    }
}
// The two 16-byte pieces of columns gc .. gc + 15 (gc a multiple of 16) of a row of the BF16 A tile.
template <int ROWS>
__device__ __forceinline__ uint4* a_piece(unsigned char* A, int row, int gc, int k) {
    const int ch = ((gc >> 3) & 7) + k;
    return reinterpret_cast<uint4*>(A + (uint32_t)(gc >> 6) * (ROWS * 128u) + (uint32_t)row * 128u +
                                    (uint32_t)((ch ^ (row & 7)) << 4));
}
// 16 operand values in the format of the GEMM that reads them (F8OP: e4m3); w: the same, packed to BF16.
template <int ROWS>
__device__ __forceinline__ void a_store16(unsigned char* A, int row, int gc, bool f8op, const uint4 (&w)[2],
                                          const float (&v)[16]) {
    if (!f8op) {
        *a_piece<ROWS>(A, row, gc, 0) = w[0];
        *a_piece<ROWS>(A, row, gc, 1) = w[1];
    } else {
        uint32_t q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            q[i] = pack_e4m3x2(v[4 * i], v[4 * i + 1]) | (pack_e4m3x2(v[4 * i + 2], v[4 * i + 3]) << 16);
        const int ch = (gc >> 4) & 7;
        *reinterpret_cast<uint4*>(A + (uint32_t)(gc >> 7) * (ROWS * 128u) + (uint32_t)row * 128u +
                                  (uint32_t)((ch ^ (row & 7)) << 4)) = make_uint4(q[0], q[1], q[2], q[3]);
    }
}
// Eight operand values of row `row` at columns col .. col + 7 (col a multiple of 8) of an A tile of ROWS rows.
template <int ROWS>
__device__ __forceinline__ void pair_store8(unsigned char* A, int row, int col, int eb, uint4 bf, const float (&v)[8]) {
    if (eb == 2) {
        const int ch = (col >> 3) & 7;
        *reinterpret_cast<uint4*>(A + (uint32_t)(col >> 6) * (ROWS * 128u) + (uint32_t)row * 128u +
                                  (uint32_t)((ch ^ (row & 7)) << 4)) = bf;
    } else {
        const int ch = (col >> 4) & 7;
        *reinterpret_cast<uint2*>(A + (uint32_t)(col >> 7) * (ROWS * 128u) + (uint32_t)row * 128u +
                                  (uint32_t)((ch ^ (row & 7)) << 4) + (uint32_t)(col & 8)) = pack8_e4m3(v);
    }
}
// member_value with its loads ahead of the sums (one latency, not one for every few slices).
__device__ __forceinline__ float pair_member_value(const TcArgs& P, int m, int tile, int row) {
    const float* q = P.qsave + qs_off(m, tile, 0, row, P.ntiles);
    const int n = P.H / 16;
    float a = 0.0f, v[16];
    for (int s = 0; s < n; s += 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = s + i < n ? q[(s + i) * 128] : 0.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (s + i < n) a += v[i];
    }
    return a + __ldg(P.bout + m);
}

// Rows of the weight chunk of iteration `it`, and the even CTA's share of them.
template <bool F8>
__device__ __noinline__ void chunk_rows(const TcArgs& P, int it, int& rows, int& half) {
    rows = half = 0;
    for (int g = 0; g < P.ngemm; ++g) {
        const int N = P.gN[g], nch = P.gKp[g] * (F8 ? P.geb[g] : 2) / 128;
        for (int n0 = 0; n0 < N; n0 += 256, it -= nch)
            if (it < nch) {
                rows = N - n0 < 256 ? N - n0 : 256;
                half = min((rows + 31) / 32 * 16, rows);
                return;
            }
    }
}
// After a wait has run out (one thread of the even CTA, both CTAs past their
// roles): until the loads that either CTA has issued have landed, or the limit.
// A part that was not issued is counted as if it had landed, so that the
// stage's phase ends with the part that was.
template <bool F8>
__device__ __noinline__ void land_loads(const TcArgs& P, Smem& S) {
    const unsigned long long t0 = gtimer();
    for (int s = 0; s < P.stages; ++s) {
        const PairStageLoads q = pair_stage_loads(S.issued, S.odd_issued, P.stages, s);
        if (q.it < 0) continue;
        const uint32_t bar = smem_u32(&S.full[s]);
        if (q.even != q.odd) {
            int rows, half;
            chunk_rows<F8>(P, q.it, rows, half);
            if (q.even)
                asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar),
                             "r"((uint32_t)(rows - half) * 128u)
                             : "memory");
            else
                mbar_arrive_tx(bar, (uint32_t)(rows - half) * 128u);
        }
        while (!mbar_try(bar, (q.it / P.stages) & 1) && gtimer() - t0 < 2 * WAIT_NS) {}
    }
}

// 18 warps spread 5/5/4/4 over the four schedulers, each with 16K registers:
// at most 96 registers per thread
// F8: the forward GEMMs take FP8 e4m3 operands (the input-gradient GEMMs
// stay BF16).  RES: residual ensemble (h_l = h_{l-1} + tanh(z_l) for l >= 1).
// ROWS: walkers per CTA, 128 or 64.  TMEM of a 256-column block: with 128 rows
// a lane is a row and the block fills 256 columns; with 64, lanes 0..63 hold
// the rows' first half of the block's columns and lanes 64..127 the second
// half, so that the block fills 128 columns and every epilogue warp has work.
template <bool F8, bool RES, int ROWS>
__global__ void __maxnreg__(96)
    k_mlp_tc_pair(const __grid_constant__ TcArgs P, const __grid_constant__ CUtensorMap map_big,
                  const __grid_constant__ CUtensorMap map_small) {
    extern __shared__ __align__(1024) unsigned char dsm_raw[];
    // swizzled tiles need 1024-byte aligned atoms; the same offset in both CTAs
    unsigned char* dsm =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ Smem S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int m = blockIdx.y;
    // the 128-row tile of the scratch buffers that holds this CTA's rows, and their first row in it.  (With an
    // odd number of tiles the last pair's second CTA has none: it streams its half of the weights, its rows are
    // zeros that nothing reads, and its epilogue has no columns.)
    const int tile = ROWS == 128 ? blockIdx.x : blockIdx.x >> 1;
    const int row0 = ROWS == 128 ? 0 : (int)rank * 64;
    const int L = P.L, G = P.ngemm;   // 2L, or L for the member values alone
    unsigned char* Abuf = dsm;                                     // [Kpmax/64][ROWS][128 B]
    unsigned char* stages = dsm + (size_t)P.Kpmax * (2u * ROWS);
    const int NS = P.stages;
    volatile int* abort_flag = &S.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&S.full[s]), 1);
            mbar_init(smem_u32(&S.empty[s]), 1);
        }
        mbar_init(smem_u32(&S.acc_full), 1);
        mbar_init(smem_u32(&S.a_full), 2 * EPI_WARPS);
        mbar_init(smem_u32(&S.drain), 1);
        S.abort_flag = 0;
        S.issued = 0;
        S.odd_issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_sync_all();               // both CTAs run and their barriers are initialised
    // TMEM is allocated while the epilogue warps stage the input and the biases and warp 0 starts the weights.
    // (The even CTA's MMAs wait for arrivals that the odd CTA makes after its own allocation.)
    float* sbias = reinterpret_cast<float*>(stages + (size_t)NS * PAIR_STAGE);   // [L][H]
    float* swout = sbias + (size_t)L * P.H;                                      // [H]
    constexpr int NSUB = ROWS == 128 ? 4 : 8;          // epilogue warps that share a row's columns
    const int quarter = warp & 3;                      // TMEM lane quarter an epilogue warp may access
    const int sub = (warp - EPI_WARP0) >> 2;           // its part of the quarter's columns
    const int hf = ROWS == 128 ? 0 : quarter >> 1;                        // half of each block's columns
    const int arow = (ROWS == 128 ? quarter : quarter & 1) * 32 + lane;   // row of this CTA's A tile
    const int subx = ROWS == 128 ? sub : 2 * sub + hf;
    const int row = row0 + arow;                       // row of the scratch tile
    const int wg = tile * 128 + row;                   // global walker
    const bool valid = wg < P.W;
    if (warp >= EPI_WARP0) {
        // GEMM 0 input: u (FP32, [W][D], D even) -> its operand format (zeros past D)
        const int eb0 = F8 ? P.geb[0] : 2;
        for (int col = 8 * subx; col < P.gKp[0]; col += 8 * NSUB) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                float2 q = make_float2(0.0f, 0.0f);
                if (valid && col + i < P.D)
                    q = __ldg(reinterpret_cast<const float2*>(P.u + (size_t)wg * P.D + col + i));
                v[i] = q.x;
                v[i + 1] = q.y;
            }
            pair_store8<ROWS>(Abuf, arow, col, eb0, pack8(v), v);
        }
        // biases [L][H], then w_out [H] (H a multiple of 32)
        const int nb4 = L * P.H / 4;
        const float4* gb = reinterpret_cast<const float4*>(P.bias + (size_t)m * L * P.H);
        const float4* gw = reinterpret_cast<const float4*>(P.wout + (size_t)m * P.H);
        for (int i = threadIdx.x - 32 * EPI_WARP0; i < nb4 + P.H / 4; i += 32 * EPI_WARPS)
            reinterpret_cast<float4*>(sbias)[i] = i < nb4 ? __ldg(gb + i) : __ldg(gw + i - nb4);
        fence_async_smem();
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                     "r"((uint32_t)P.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    uint32_t tmem = 0;
    if (warp > 0) {
        fence_before();
        asm volatile("bar.sync 1, %0;" ::"r"(NTHREADS - 32) : "memory");
        fence_after();
        tmem = S.tmem_base;
    }

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            // (N is a multiple of 32: both CTAs load part of every stage, so neither runs ahead of the other)
            for (int g = 0; g < G && ok; ++g) {
                const int N = P.gN[g], nch = P.gKp[g] * (F8 ? P.geb[g] : 2) / 128;
                for (int n0 = 0; n0 < N && ok; n0 += 256) {
                    const int rows = N - n0 < 256 ? N - n0 : 256;
                    const int half = (rows + 31) / 32 * 16;                 // rows of the even CTA
                    const int mine = rank == 0 ? min(half, rows) : max(0, rows - half);
                    for (int c = 0; c < nch; ++c, ++it) {
                        const int s = it % NS;
                        if (!mbar_wait(smem_u32(&S.empty[s]), ((it / NS) & 1) ^ 1, abort_flag, P.err, 1)) {
                            ok = false;
                            break;
                        }
                        if (rank == 0) mbar_arrive_tx(smem_u32(&S.full[s]), (uint32_t)rows * 128u);
                        const uint32_t bar = mapa(smem_u32(&S.full[s]), 0);
                        const long long first =
                            (long long)m * P.member_rows + P.grow[g] + (long long)c * N + n0 + (rank == 0 ? 0 : half);
                        uint32_t dst = smem_u32(stages + (size_t)s * PAIR_STAGE);
                        int r = 0;
                        for (; r + 64 <= mine; r += 64, dst += 8192u)
                            pair_tma_load(dst, &map_big, (int)(first + r), bar);
                        for (; r < mine; r += 8, dst += 1024u) pair_tma_load(dst, &map_small, (int)(first + r), bar);
                    }
                }
            }
            S.issued = it;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (even CTA)
        if (lane == 0 && rank == 0) {
            int it = 0;
            bool ok = true;
            for (int g = 0; g < G && ok; ++g) {
                const int N = P.gN[g], nch = P.gKp[g] * (F8 ? P.geb[g] : 2) / 128;
                const bool f8 = F8 && P.geb[g] == 1;
                // completion g of a_full: both CTAs' input for g = 0, then their epilogues of GEMM
                // g - 1, which have also read the accumulator
                if (!mbar_wait_by<pair_try>(smem_u32(&S.a_full), g & 1, abort_flag, P.err, 4)) {
                    ok = false;
                    break;
                }
                pair_acquire();
                fence_after();
                for (int n0 = 0; n0 < N && ok; n0 += 256) {
                    const int rows = N - n0 < 256 ? N - n0 : 256;
                    const int cols = (rows + 31) / 32 * 32;    // columns past N take whatever the stage held, unread
                    const uint32_t id = f8 ? idesc_e4m3(2 * ROWS, cols) : idesc_bf16(2 * ROWS, cols);
                    const uint32_t dacc = tmem + (uint32_t)(ROWS == 128 ? n0 : n0 / 2);
                    for (int c = 0; c < nch; ++c, ++it) {
                        const int s = it % NS;
                        if (!mbar_wait(smem_u32(&S.full[s]), (it / NS) & 1, abort_flag, P.err, 4)) {
                            ok = false;
                            break;
                        }
                        fence_after();
                        const uint32_t a_atom = smem_u32(Abuf) + (uint32_t)c * (ROWS * 128u);
                        const uint32_t b_atom = smem_u32(stages + (size_t)s * PAIR_STAGE);
                        // K = 16 BF16 or 32 FP8 per MMA: 32 bytes into the 128-byte rows
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            pair_mma(f8, dacc, desc_sw128(a_atom + 32u * kk), desc_sw128(b_atom + 32u * kk), id,
                                     (c | kk) != 0);
                        pair_commit(smem_u32(&S.empty[s]));
                    }
                }
                if (ok) pair_commit(smem_u32(&S.acc_full));
            }
            pair_commit(smem_u32(&S.drain));
        }
        if (lane == 0) {
            // every MMA issued has completed, and its arrivals have reached this CTA, before it releases its TMEM
            const unsigned long long t0 = gtimer();
            while (!mbar_try(smem_u32(&S.drain), 0) && gtimer() - t0 < 2 * WAIT_NS) {}
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // Warp w reads TMEM lane quarter w mod 4 and owns a contiguous quarter
        // (sub = (w - 2) / 4) of the 16-column groups that the quarter's lanes hold.
        const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
        const int H = P.H;
        const uint32_t a_bar = smem_u32(&S.a_full);
        if (lane == 0) pair_arrive(a_bar, rank);       // the input is in place
        __nv_bfloat16* tsave_tile = P.tsave + ((size_t)m * P.ntiles + tile) * (size_t)L * 128 * H;
        // residual stream of a resnet ensemble: h_l (forward) and dA/dh_l (backward)
        // in FP32, one [H/8][128][8] block per tile and member, overwritten in place
        float* rsave_tile = RES ? P.rsave + ((size_t)m * P.ntiles + tile) * (size_t)128 * H + ts_off(0, row, 0, H) : nullptr;
        const uint32_t rcol = (uint32_t)P.acc_cols;    // ... or, where TMEM has room, in its columns rcol ..
        const bool rtm = RES && 2 * P.acc_cols <= P.tmem_cols;
        for (int g = 0; g < G; ++g) {
            const int N = P.gN[g];
            const bool fwd = g < L;
            // operand format of the next GEMM (2 BF16, 1 FP8) and its padded K
            const int ebn = (F8 && g + 1 < G) ? P.geb[g + 1] : 2;
            const int kpn = g + 1 < G ? P.gKp[g + 1] : N;
            const float ws = F8 ? P.wscale[(size_t)m * 2 * L + g] : 1.0f;   // [M][2L]
            const int l = fwd ? g : (2 * L - 1 - g);   // layer of this GEMM
            // what the epilogue does: hidden layer forward, last one, hidden layer backward, input gradient
            const bool last = fwd && l == L - 1;
            const bool tload = !fwd && l > 0;          // saved tanh of layer l - 1 needed
            // resnet: h_{l-1} is added to this layer's tanh (forward, l >= 1); dA/dh_l is added to the
            // product W_l^T Delta_l (backward, l >= 1), from the stream below l = L - 1, from w_out there
            const bool res_ld = RES && (fwd ? l >= 1 : l >= 1 && l < L - 1);
            const bool res_st = RES && (fwd ? l < L - 1 : l >= 2);
            // a plain BF16 operand of the next layer is the tanh itself: it is saved from there, after the
            // operand has been released
            const bool late = !RES && fwd && !last && ebn == 2;
            // the quarter's 16-column groups: first those of block 0, then of block 1
            const int rows0 = N < 256 ? N : 256, half0 = (rows0 + 31) / 32 * 16;
            const int rows1 = N - rows0, half1 = (rows1 + 31) / 32 * 16;
            int ng0, ng1;
            if (ROWS == 128) {
                ng0 = N / 16;
                ng1 = 0;
            } else {
                ng0 = (hf ? rows0 - half0 : min(half0, rows0)) / 16;
                ng1 = (hf ? rows1 - half1 : min(half1, rows1)) / 16;
                ng0 = max(ng0, 0);
                ng1 = max(ng1, 0);
            }
            const int ngr = tile < P.ntiles ? ng0 + ng1 : 0, gpw = (ngr + 3) / 4;
            const int i0 = min(sub * gpw, ngr), i1 = min(i0 + gpw, ngr);
            auto col_of = [&](int i) {
                if (ROWS == 128) return 16 * i;
                return i < ng0 ? hf * half0 + 16 * i : 256 + hf * half1 + 16 * (i - ng0);
            };
            const __nv_bfloat16* tsrc = tsave_tile + ts_off(tload ? l - 1 : 0, row, 0, H);
            __nv_bfloat16* tdst = tsave_tile + ts_off(l, row, 0, H);
            // saved tanh of the next two groups, loaded ahead of their use
            uint4 tb[2][2];
            auto tfetch = [&](int i, uint4 (&t)[2]) {
                const uint4* p = reinterpret_cast<const uint4*>(tsrc + (uint32_t)col_of(i) * 128u);
                t[0] = p[0];
                t[1] = p[128];
            };
            if (tload) {
                if (i0 < i1) tfetch(i0, tb[0]);
                if (!RES && i0 + 1 < i1) tfetch(i0 + 1, tb[1]);
            }
            if (!mbar_wait(smem_u32(&S.acc_full), g & 1, abort_flag, P.err, 8)) break;
            fence_after();
            auto group = [&](int i, uint4 (&tq)[2]) {
                const int gc = col_of(i);              // first of these 16 columns
                const uint32_t tcol = (uint32_t)(ROWS == 128 ? gc : (i < ng0 ? 16 * i : 128 + 16 * (i - ng0)));
                float acc[16], rp[16];
                tmem_ld16(trow + tcol, acc);
                float* rg = rsave_tile + (uint32_t)gc * 128u;
                if (res_ld) {
                    if (rtm) {
                        tmem_ld16(trow + rcol + tcol, rp);
                    } else {
                        const float4 *p0 = reinterpret_cast<const float4*>(rg), *p1 = p0 + 256;
                        const float4 q[4] = {p0[0], p0[1], p1[0], p1[1]};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            rp[4 * k] = q[k].x;
                            rp[4 * k + 1] = q[k].y;
                            rp[4 * k + 2] = q[k].z;
                            rp[4 * k + 3] = q[k].w;
                        }
                    }
                }
                auto res_store = [&](const float (&h)[16]) {
                    if (rtm) {
                        tmem_st16(trow + rcol + tcol, h);
                    } else {
                        float4 *p0 = reinterpret_cast<float4*>(rg), *p1 = p0 + 256;
                        p0[0] = make_float4(h[0], h[1], h[2], h[3]);
                        p0[1] = make_float4(h[4], h[5], h[6], h[7]);
                        p1[0] = make_float4(h[8], h[9], h[10], h[11]);
                        p1[1] = make_float4(h[12], h[13], h[14], h[15]);
                    }
                };
                tmem_wait_ld();
                if (fwd) {
                    // z = s_W (A W'^T) + b: the weight scale of an FP8 GEMM
                    if (F8) {
                        float b[16];
                        ld16(sbias + (uint32_t)(l * H + gc), b);
#pragma unroll
                        for (int q = 0; q < 16; ++q) acc[q] = fmaf(acc[q], ws, b[q]);
                    } else {
                        add16(acc, sbias + (uint32_t)(l * H + gc));
                    }
                    uint4 tw[2];
                    tw[0] = make_uint4(tanh_bf16x2(acc[0], acc[1]), tanh_bf16x2(acc[2], acc[3]),
                                       tanh_bf16x2(acc[4], acc[5]), tanh_bf16x2(acc[6], acc[7]));
                    tw[1] = make_uint4(tanh_bf16x2(acc[8], acc[9]), tanh_bf16x2(acc[10], acc[11]),
                                       tanh_bf16x2(acc[12], acc[13]), tanh_bf16x2(acc[14], acc[15]));
                    if (!last && !late) {
                        uint4* tp = reinterpret_cast<uint4*>(tdst + (uint32_t)gc * 128u);
                        tp[0] = tw[0];
                        tp[128] = tw[1];
                    }
                    if (!RES && !last && (!F8 || ebn == 2)) {
                        a_store16<ROWS>(Abuf, arow, gc, false, tw, acc);
                    } else {
                        // h_l = t_l (+ h_{l-1} of a residual network, in FP32)
                        float h[16];
                        unpack16(tw, h);
                        if (RES && res_ld) {
#pragma unroll
                            for (int q = 0; q < 16; ++q) h[q] = rp[q] + h[q];
                        }
                        if (RES && res_st) res_store(h);
                        if (last) {
                            // A = w_out . h_L; Delta_L = w_out (1 - t_L^2)
                            float wo[16], apart = 0.0f;
                            ld16(swout + gc, wo);
#pragma unroll
                            for (int q = 0; q < 16; ++q) apart = fmaf(wo[q], h[q], apart);
                            P.qsave[qs_off(m, tile, gc >> 4, row, P.ntiles)] = apart;
                            tanh_back(wo, tw);
                            uint4 w[2];
                            pack16(wo, w);
                            a_store16<ROWS>(Abuf, arow, gc, F8 && ebn == 1, w, wo);
                        } else {
                            uint4 w[2];
                            pack16(h, w);
                            a_store16<ROWS>(Abuf, arow, gc, F8 && ebn == 1, w, h);
                        }
                    }
                } else if (l > 0) {
                    // G_{l-1} -> Delta_{l-1} = G (1 - t_{l-1}^2); with a residual,
                    // G_{l-1} = W_l^T Delta_l + dA/dh_l first
                    if (RES) {
                        if (l == L - 1) {
                            ld16(swout + gc, rp);
                        }
#pragma unroll
                        for (int q = 0; q < 16; ++q) acc[q] = rp[q] + acc[q];
                        if (res_st) res_store(acc);
                    }
                    tanh_back(acc, tq);
                    if (i + (RES ? 1 : 2) < i1) tfetch(i + (RES ? 1 : 2), tq);
                    uint4 w[2];
                    pack16(acc, w);
                    a_store16<ROWS>(Abuf, arow, gc, false, w, acc);
                } else if (valid) {
                    // G_0 = dA/du: dA/ds_j = -sin s_j g[2j] + cos s_j g[2j+1] (torsion), g[2j] (distance)
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const int j = gc / 2 + p;
                        if (2 * j < P.D) {
                            const float2 u = __ldg(reinterpret_cast<const float2*>(P.u + (size_t)wg * P.D + 2 * j));
                            const bool dist = P.cvdist && __ldg(P.cvdist + j);   // input (s, 0)
                            P.gradA[((size_t)m * P.W + wg) * P.C + j] =
                                dist ? acc[2 * p] : -u.y * acc[2 * p] + u.x * acc[2 * p + 1];
                        }
                    }
                }
            };
            if (RES) {
                for (int i = i0; i < i1; ++i) group(i, tb[0]);
            } else {
                for (int i = i0; i < i1; i += 2) {
                    group(i, tb[0]);
                    if (i + 1 < i1) group(i + 1, tb[1]);
                }
            }
            if (RES && rtm) tmem_wait_st();
            if (g < G - 1) {
                // columns N .. kpn - 1 are K padding of the next GEMM: zero
                const float zero[8] = {};
                for (int gc = N + 8 * subx; gc < kpn; gc += 8 * NSUB)
                    pair_store8<ROWS>(Abuf, arow, gc, ebn, make_uint4(0, 0, 0, 0), zero);
                fence_async_smem();
                fence_before();
                __syncwarp();
                if (lane == 0) pair_arrive(a_bar, rank);
                if (late) {
                    // only this thread writes these operand columns again, after the GEMM that reads them
                    for (int i = i0; i < i1; ++i) {
                        const int gc = col_of(i);
                        uint4* tp = reinterpret_cast<uint4*>(tdst + (uint32_t)gc * 128u);
                        tp[0] = *a_piece<ROWS>(Abuf, arow, gc, 0);
                        tp[128] = *a_piece<ROWS>(Abuf, arow, gc, 1);
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    // member value A = w_out . h_L + b_out: the 16-column partials in column order
    if (warp >= EPI_WARP0 && warp < EPI_WARP0 + 4) {
        if ((ROWS == 128 || hf == 0) && valid && !S.abort_flag)
            P.Apart[(size_t)m * P.W + wg] = pair_member_value(P, m, tile, row);
    }
    if (threadIdx.x == 0 && S.abort_flag) st_cluster_u32(mapa(smem_u32(&S.abort_flag), rank ^ 1u), 1u);
    __syncwarp();
    cluster_sync_all();               // no CTA leaves while the pair's MMAs may touch it
    if (S.abort_flag) {               // the same in both CTAs
        if (threadIdx.x == 0 && rank == 1) st_cluster_u32(mapa(smem_u32(&S.odd_issued), 0), (uint32_t)S.issued);
        __syncwarp();
        cluster_sync_all();
        if (rank == 0 && threadIdx.x == 0) land_loads<F8>(P, S);
        __syncwarp();
        cluster_sync_all();           // ... nor while loads that no MMA has waited for are on their way
    }
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)P.tmem_cols)
                     : "memory");
    }
}

template <int ROWS>
cudaError_t launch_pair(TcArgs P, const CUtensorMap& big, const CUtensorMap& small, cudaStream_t s) {
    int nmax = 0;
    for (int g = 0; g < P.ngemm; ++g) nmax = P.gN[g] > nmax ? P.gN[g] : nmax;
    // shared memory: the A tile, the biases, and as many weight stages as fit
    const size_t fixed = 1024 + (size_t)P.Kpmax * (2 * ROWS) + sizeof(float) * (size_t)(P.L + 1) * P.H;
    if (fixed + 2 * PAIR_STAGE > PAIR_SMEM_MAX) return cudaErrorInvalidValue;
    P.stages = (int)((PAIR_SMEM_MAX - fixed) / PAIR_STAGE);
    if (P.stages > TC_MAX_STAGES) P.stages = TC_MAX_STAGES;
    size_t smem = fixed + (size_t)P.stages * PAIR_STAGE;
    // TMEM: the accumulator and, if it fits, a residual network's stream
    P.acc_cols = ROWS == 128 ? nmax : nmax <= 256 ? nmax / 2 : 128 + (nmax - 256) / 2;
    const int cols = P.resnet && P.acc_cols <= 256 ? 2 * P.acc_cols : P.acc_cols;
    P.tmem_cols = 32;
    while (P.tmem_cols < cols) P.tmem_cols *= 2;
    if (P.tmem_cols > 256) smem = PAIR_SMEM_MAX;
    else if (smem < PAIR_SMEM_MIN) smem = PAIR_SMEM_MIN;
    const int v = (P.geb[0] == 1 ? 1 : 0) + (P.resnet ? 2 : 0);
    auto kern = v == 0 ? k_mlp_tc_pair<false, false, ROWS> : v == 1 ? k_mlp_tc_pair<true, false, ROWS>
              : v == 2 ? k_mlp_tc_pair<false, true, ROWS> : k_mlp_tc_pair<true, true, ROWS>;
    static RidOnce once[4];
    if (const cudaError_t e = rid_opt_in(once[v], PAIR_SMEM_MAX, kern)) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ROWS == 128 ? (P.ntiles + 1) / 2 * 2 : 2 * P.ntiles, P.M, 1);
    cfg.blockDim = dim3(NTHREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P, big, small);
}

}  // namespace

cudaError_t rid_launch_mlp_tc_pair(const TcArgs& P, int rows, const CUtensorMap& big, const CUtensorMap& small,
                                   cudaStream_t s) {
    if (P.ngemm != P.L && P.ngemm != 2 * P.L) return cudaErrorInvalidValue;
    if (P.resnet && !P.rsave) return cudaErrorInvalidValue;
    return rows == 64 ? launch_pair<64>(P, big, small, s) : launch_pair<128>(P, big, small, s);
}
