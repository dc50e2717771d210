// k_mlp_tc.cu -- BF16 / FP8 ensemble MLP on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in TMEM, weights streamed by tensor TMA).
//
// Operands are BF16 (kind::f16) or, for the forward GEMMs of the FP8 mode,
// e4m3 (kind::f8f6f4); the byte layout is the same for both (128-byte rows,
// 64 BF16 or 128 FP8 columns per K-chunk, 32 bytes of K per MMA), so a GEMM's
// operand format only changes how its A operand is written and which MMA
// kind is issued.  FP8 weights are stored as W / s_W and the accumulator is
// scaled back by s_W in the epilogue.
//
// Work unit: one CTA = one tile of 128 walkers x one ensemble member.  It runs a
// single tile up to width 256, where two accumulators fit in TMEM; more tiles and
// wider members take CTA pairs (k_mlp_tc_pair).  The chain of 2L GEMMs
//   forward  l = 0..L-1 :  Z_l = H_{l-1} W_l^T      (128 x H,   K = D' or H)
//   backward l = L-1..0 :  G_{l-1} = Delta_l W_l     (128 x fin, K = H)
// runs with the activation tile (A operand, BF16) resident in shared memory
// and the weights (B operand) streamed in 64-wide K-chunks through a ring of
// TMA stages.  Both operands use the 128-byte swizzled K-major layout: rows of
// 128 bytes (64 BF16 along K), the 16-byte chunk c of row r stored at chunk
// c ^ (r mod 8), 8-row groups 1024 bytes apart.  The weights are swizzled on
// the host, so the TMA copies them as plain bytes.
//
// Epilogues (16 warps) read the FP32 accumulator from TMEM and write the next
// A operand chunk by chunk (64 columns); each chunk is released to the MMA
// issuer through its own mbarrier, and the accumulator is double buffered in
// TMEM, so the next GEMM's MMAs start on chunk 0 while later chunks of the
// current epilogue are still being written.
//   g_L = w_out, Delta_l = g_l * (1 - tanh^2 z_l), g_{l-1} = W_l^T Delta_l,
//   dA/ds_j = -sin s_j g_0[2j] + cos s_j g_0[2j+1].
// tanh(z_l) is kept as BF16 in a global scratch for the backward pass (laid
// out so that a warp's 32 rows move one contiguous 512-byte line), and a
// backward epilogue loads its part of it before waiting for the accumulator.
//
// Warp roles (576 threads): warp 0 = TMA producer, warp 1 = TMEM allocator +
// MMA issuer, warps 2..17 = epilogue: warp w reads TMEM lane quarter w mod 4
// (rows 32 (w mod 4) ..) and, inside every 64-column chunk, the 16 columns
// 16 ((w - 2) / 4) ...  Every wait is bounded in time; a wait that expires
// sets an error word, drains what was issued and returns.
#include "rid_tc_ptx.cuh"

namespace {

struct Smem {
    uint64_t full[TC_MAX_STAGES];
    uint64_t empty[TC_MAX_STAGES];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t a_chunk[TC_MAX_KCHUNKS];
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;
};

// 18 warps spread 5/5/4/4 over the four schedulers, each with 16K registers:
// at most 96 registers per thread
// F8: the forward GEMMs take FP8 e4m3 operands (the input-gradient GEMMs
// stay BF16); the BF16 instantiation has every operand format fixed at
// compile time.
// RES: residual ensemble (h_l = h_{l-1} + tanh(z_l) for l >= 1), its own
// instantiation so that the plain networks keep their register allocation.
template <bool F8, bool RES>
__global__ void __maxnreg__(96)
    k_mlp_tc(const __grid_constant__ TcArgs P, const __grid_constant__ CUtensorMap map_big,
             const __grid_constant__ CUtensorMap map_small) {
    extern __shared__ __align__(1024) unsigned char dsm_raw[];
    // swizzled tiles need 1024-byte aligned atoms
    unsigned char* dsm =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ Smem S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int tile = 0;            // a call of more than 128 walkers takes CTA pairs
    const int m = blockIdx.y;
    const int L = P.L, G = P.ngemm;   // 2L, or L for the member values alone
    unsigned char* Abuf = dsm;                                     // [Kpmax/64][128 rows][128 B]
    unsigned char* stages = dsm + (size_t)P.Kpmax * 256u;          // 128 rows x 2 B per column
    const uint32_t stage_bytes = P.stage_bytes;
    const int NS = P.stages;
    constexpr int NACC = 2;            // accumulators in TMEM
    volatile int* abort_flag = &S.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&S.full[s]), 1);
            mbar_init(smem_u32(&S.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&S.acc_full[b]), 1);
            mbar_init(smem_u32(&S.acc_empty[b]), EPI_WARPS);
        }
        for (int j = 0; j < TC_MAX_KCHUNKS; ++j) mbar_init(smem_u32(&S.a_chunk[j]), EPI_WARPS);
        mbar_init(smem_u32(&S.drain), 1);
        S.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                     "r"((uint32_t)P.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = S.tmem_base;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int it = 0;
            int last_it[TC_MAX_STAGES];
            for (int s = 0; s < NS; ++s) last_it[s] = -1;
            bool ok = true;
            for (int g = 0; g < G && ok; ++g) {
                const int N = P.gN[g], nch = P.gKp[g] * (F8 ? P.geb[g] : 2) / 128;
                for (int c = 0; c < nch && ok; ++c)
                    for (int n0 = 0; n0 < N; n0 += 256, ++it) {
                        const int rows = N - n0 < 256 ? N - n0 : 256;
                        const int s = it % NS;
                        if (!mbar_wait(smem_u32(&S.empty[s]), ((it / NS) & 1) ^ 1, abort_flag, P.err, 1)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_tx(smem_u32(&S.full[s]), (uint32_t)rows * 128u);
                        last_it[s] = it;
                        const long long row0 = (long long)m * P.member_rows + P.grow[g] + (long long)c * N + n0;
                        uint32_t dst = smem_u32(stages + (size_t)s * stage_bytes);
                        int r = 0;
                        for (; r + 64 <= rows; r += 64, dst += 8192u)
                            tma_load_2d(dst, &map_big, 0, (int)(row0 + r), smem_u32(&S.full[s]));
                        for (; r < rows; r += 8, dst += 1024u)
                            tma_load_2d(dst, &map_small, 0, (int)(row0 + r), smem_u32(&S.full[s]));
                    }
            }
            if (!ok) {
                // the loads already issued land before the CTA can exit
                for (int s = 0; s < NS; ++s)
                    if (last_it[s] >= 0) {
                        const unsigned long long t0 = gtimer();
                        while (!mbar_try(smem_u32(&S.full[s]), (last_it[s] / NS) & 1) && gtimer() - t0 < WAIT_NS) {}
                    }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            uint32_t cpar = 0;   // phase bit of every a_chunk[] barrier
            for (int g = 0; g < G && ok; ++g) {
                const int N = P.gN[g], nch = P.gKp[g] * (F8 ? P.geb[g] : 2) / 128;
                const bool f8 = F8 && P.geb[g] == 1;
                const int b = g % NACC;
                const uint32_t dacc = tmem + (uint32_t)(b * P.acc_cols);
                if (g >= NACC &&
                    !mbar_wait(smem_u32(&S.acc_empty[b]), ((g / NACC) - 1) & 1, abort_flag, P.err, 2)) {
                    ok = false;
                    break;
                }
                for (int c = 0; c < nch && ok; ++c) {
                    if (!mbar_wait(smem_u32(&S.a_chunk[c]), (cpar >> c) & 1u, abort_flag, P.err, 4)) {
                        ok = false;
                        break;
                    }
                    cpar ^= 1u << c;
                    fence_after();
                    const uint32_t a_atom = smem_u32(Abuf) + (uint32_t)c * (128u * 128u);
                    for (int n0 = 0; n0 < N; n0 += 256, ++it) {
                        const int rows = N - n0 < 256 ? N - n0 : 256;
                        const int s = it % NS;
                        if (!mbar_wait(smem_u32(&S.full[s]), (it / NS) & 1, abort_flag, P.err, 4)) {
                            ok = false;
                            break;
                        }
                        fence_after();
                        const uint32_t b_atom = smem_u32(stages + (size_t)s * stage_bytes);
                        // K = 16 BF16 or 32 FP8 per MMA: 32 bytes into the 128-byte rows
                        if (f8) {
                            const uint32_t id = idesc_e4m3(128, rows);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_e4m3(dacc + (uint32_t)n0, desc_sw128(a_atom + 32u * kk),
                                         desc_sw128(b_atom + 32u * kk), id, (c | kk) != 0);
                        } else {
                            const uint32_t id = idesc_bf16(128, rows);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_bf16(dacc + (uint32_t)n0, desc_sw128(a_atom + 32u * kk),
                                         desc_sw128(b_atom + 32u * kk), id, (c | kk) != 0);
                        }
                        mma_commit(smem_u32(&S.empty[s]));
                    }
                }
                if (ok) mma_commit(smem_u32(&S.acc_full[b]));
            }
            // every MMA issued has completed before TMEM can be released
            mma_commit(smem_u32(&S.drain));
            const unsigned long long t0 = gtimer();
            while (!mbar_try(smem_u32(&S.drain), 0) && gtimer() - t0 < WAIT_NS) {}
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int e = warp - EPI_WARP0;          // 0..15
        const int quarter = warp & 3;            // TMEM lane quarter this warp may access
        const int sub = e >> 2;                  // 16-column slice of every 64-column chunk
        const int row = quarter * 32 + lane;     // walker within the tile
        const int wg = tile * 128 + row;         // global walker
        const bool valid = wg < P.W;
        const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
        const int H = P.H;
        const int ET = 32 * EPI_WARPS;
        // GEMM 0 input first: u (FP32, [W][D]) -> its operand format, chunk by
        // chunk (zeros past D); a 128-byte chunk is 64 BF16 or 128 FP8 columns
        {
            const int eb0 = F8 ? P.geb[0] : 2, kc0 = 128 / eb0, nch0 = P.gKp[0] * eb0 / 128;
            for (int c = 0; c < nch0; ++c) {
                for (int k8 = 0; k8 < kc0 / 32; ++k8) {
                    const int col = c * kc0 + sub * (kc0 / 4) + k8 * 8;
                    float v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int k = col + i;
                        v[i] = (valid && k < P.D) ? __ldg(P.u + (size_t)wg * P.D + k) : 0.0f;
                    }
                    store_a8(Abuf, row, col, eb0, v);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&S.a_chunk[c]));
            }
        }
        float* sbias = reinterpret_cast<float*>(stages + (size_t)NS * stage_bytes);   // [L][H]
        float* swout = sbias + (size_t)L * H;                                          // [H]
        for (int idx = e * 32 + lane; idx < (L + 1) * H; idx += ET) {
            const int l = idx / H, c = idx - l * H;
            sbias[idx] = l < L ? __ldg(P.bias + ((size_t)m * L + l) * H + c) : __ldg(P.wout + (size_t)m * H + c);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(ET) : "memory");   // all epilogue warps, before any bounded wait
        __nv_bfloat16* tsave_tile = P.tsave + ((size_t)m * P.ntiles + tile) * (size_t)L * 128 * H;
        // residual stream of a resnet ensemble: h_l (forward) and dA/dh_l (backward)
        // in FP32, one [H/8][128][8] block per tile and member, overwritten in place
        float* rsave_tile = RES ? P.rsave + ((size_t)m * P.ntiles + tile) * (size_t)128 * H : nullptr;
        for (int g = 0; g < G; ++g) {
            const int N = P.gN[g];
            const bool fwd = g < L;
            // operand bytes of the next GEMM; with FP8 its 128-column K-chunks
            // span two of these 64-column chunks, and its K padding is zeroed too
            const int ebn = (F8 && g + 1 < G) ? P.geb[g + 1] : 2;
            const int nch = ebn == 1 ? 2 * ((N + 127) / 128) : (N + 63) / 64;
            const float ws = F8 ? P.wscale[(size_t)m * 2 * L + g] : 1.0f;   // [M][2L]
            const int l = fwd ? g : (2 * L - 1 - g);   // layer of this GEMM
            const int b = g % NACC;
            // resnet: h_{l-1} is added to this layer's tanh (forward, l >= 1);
            // dA/dh_l is added to the product W_l^T Delta_l (backward, l >= 1),
            // read from the stream below l = L-1 and from w_out at l = L-1
            const bool res_fwd = RES && fwd && l >= 1;
            const bool res_bwd = RES && !fwd && l >= 1;
            const bool res_ld = res_fwd || (res_bwd && l < L - 1);
            const bool res_st = RES && (fwd ? l < L - 1 : l >= 2);
            // saved tanh of layer l-1 for this warp's columns, loaded before the wait
            constexpr int PREF = RES ? 1 : 2;          // chunks prefetched; later ones load in place
            uint4 tall[PREF][2];
            if (!fwd && l > 0) {
#pragma unroll
                for (int c = 0; c < PREF; ++c)
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int col = c * 64 + sub * 16 + k * 8;
                        if (c < nch && col < N)
                            tall[c][k] = *reinterpret_cast<const uint4*>(tsave_tile + ts_off(l - 1, row, col, H));
                    }
            }
            if (!mbar_wait(smem_u32(&S.acc_full[b]), (g / NACC) & 1, abort_flag, P.err, 8)) break;
            fence_after();
            const uint32_t tacc = trow + (uint32_t)(b * P.acc_cols);
#pragma unroll
            for (int c = 0; c < TC_MAX_KCHUNKS; ++c) {
                if (c >= nch) break;
                const int col0 = c * 64 + sub * 16;    // first of this warp's 16 columns
                const int left = N - col0;
                const int ng = left <= 0 ? 0 : (left >= 16 ? 2 : 1);   // 8-column groups
                uint4 tcur[2];
                if (!fwd && l > 0) {
                    if (c < PREF) {
                        tcur[0] = tall[c < PREF ? c : 0][0];
                        tcur[1] = tall[c < PREF ? c : 0][1];
                    } else {
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            if (k < ng) tcur[k] = *reinterpret_cast<const uint4*>(tsave_tile + ts_off(l - 1, row, col0 + k * 8, H));
                    }
                }
                float4 rprev[2][2];
                if (res_ld) {
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (k < ng) {
                            const float4* rp = reinterpret_cast<const float4*>(rsave_tile + ts_off(0, row, col0 + k * 8, H));
                            rprev[k][0] = rp[0];
                            rprev[k][1] = rp[1];
                        }
                }
                float acc[2][8];
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (k < ng) tmem_ld8(tacc + (uint32_t)(col0 + k * 8), acc[k]);
                tmem_wait_ld();
                float apart = 0.0f;                    // w_out . h_L over this warp's 16 columns
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (k >= ng) break;
                    const int gc = col0 + k * 8;
                    if (fwd) {
                        const float* bias = sbias + (size_t)l * H + gc;
                        // z = s_W (A W'^T) + b: the weight scale of an FP8 GEMM (1 for BF16)
                        const uint4 tw =
                            F8 ? make_uint4(tanh_bf16x2(fmaf(acc[k][0], ws, bias[0]), fmaf(acc[k][1], ws, bias[1])),
                                            tanh_bf16x2(fmaf(acc[k][2], ws, bias[2]), fmaf(acc[k][3], ws, bias[3])),
                                            tanh_bf16x2(fmaf(acc[k][4], ws, bias[4]), fmaf(acc[k][5], ws, bias[5])),
                                            tanh_bf16x2(fmaf(acc[k][6], ws, bias[6]), fmaf(acc[k][7], ws, bias[7])))
                               : make_uint4(tanh_bf16x2(acc[k][0] + bias[0], acc[k][1] + bias[1]),
                                            tanh_bf16x2(acc[k][2] + bias[2], acc[k][3] + bias[3]),
                                            tanh_bf16x2(acc[k][4] + bias[4], acc[k][5] + bias[5]),
                                            tanh_bf16x2(acc[k][6] + bias[6], acc[k][7] + bias[7]));
                        *reinterpret_cast<uint4*>(tsave_tile + ts_off(l, row, gc, H)) = tw;
                        if (RES) {
                            // h_l = t_l (+ h_{l-1} for l >= 1), kept in FP32 for the next layer
                            float t[8], h[8];
                            unpack_bf16x8(tw, t);
                            const float rp[8] = {rprev[k][0].x, rprev[k][0].y, rprev[k][0].z, rprev[k][0].w,
                                                 rprev[k][1].x, rprev[k][1].y, rprev[k][1].z, rprev[k][1].w};
#pragma unroll
                            for (int i = 0; i < 8; ++i) h[i] = res_fwd ? rp[i] + t[i] : t[i];
                            if (res_st) {
                                float4* rs = reinterpret_cast<float4*>(rsave_tile + ts_off(0, row, gc, H));
                                rs[0] = make_float4(h[0], h[1], h[2], h[3]);
                                rs[1] = make_float4(h[4], h[5], h[6], h[7]);
                            }
                            if (l == L - 1) {
                                // A = w_out . h_L; Delta_L = w_out (1 - t_L^2)
                                float d[8];
                                const float* wo = swout + gc;
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    apart = fmaf(wo[i], h[i], apart);
                                    d[i] = wo[i] * (1.0f - t[i] * t[i]);
                                }
                                store_a8(Abuf, row, gc, ebn, d);
                            } else {
                                store_a8(Abuf, row, gc, ebn, h);
                            }
                        } else if (l == L - 1) {
                            float t[8], d[8];
                            unpack_bf16x8(tw, t);
                            const float* wo = swout + gc;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                apart = fmaf(wo[i], t[i], apart);
                                d[i] = wo[i] * (1.0f - t[i] * t[i]);
                            }
                            store_a8(Abuf, row, gc, ebn, d);
                        } else if (ebn == 2) {
                            *reinterpret_cast<uint4*>(Abuf + a_off(row, gc)) = tw;
                        } else {
                            float t[8];
                            unpack_bf16x8(tw, t);
                            store_a8(Abuf, row, gc, ebn, t);
                        }
                    } else if (l > 0) {
                        // G_{l-1} -> Delta_{l-1} = G (1 - t_{l-1}^2); with a residual,
                        // G_{l-1} = W_l^T Delta_l + dA/dh_l first
                        float t[8], d[8];
                        unpack_bf16x8(tcur[k], t);
                        if (res_bwd) {
                            float gl[8];
                            if (l == L - 1) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) gl[i] = swout[gc + i];
                            } else {
                                gl[0] = rprev[k][0].x; gl[1] = rprev[k][0].y; gl[2] = rprev[k][0].z; gl[3] = rprev[k][0].w;
                                gl[4] = rprev[k][1].x; gl[5] = rprev[k][1].y; gl[6] = rprev[k][1].z; gl[7] = rprev[k][1].w;
                            }
#pragma unroll
                            for (int i = 0; i < 8; ++i) gl[i] += acc[k][i];
                            if (res_st) {
                                float4* rs = reinterpret_cast<float4*>(rsave_tile + ts_off(0, row, gc, H));
                                rs[0] = make_float4(gl[0], gl[1], gl[2], gl[3]);
                                rs[1] = make_float4(gl[4], gl[5], gl[6], gl[7]);
                            }
#pragma unroll
                            for (int i = 0; i < 8; ++i) d[i] = gl[i] * (1.0f - t[i] * t[i]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 8; ++i) d[i] = acc[k][i] * (1.0f - t[i] * t[i]);
                        }
                        store_a8(Abuf, row, gc, ebn, d);
                    } else if (valid) {
                        // G_0 = dA/du: dA/ds_j = -sin s_j g[2j] + cos s_j g[2j+1] (torsion), g[2j] (distance)
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const int j = gc / 2 + p;
                            if (2 * j < P.D) {
                                const float cs = __ldg(P.u + (size_t)wg * P.D + 2 * j);
                                const float sn = __ldg(P.u + (size_t)wg * P.D + 2 * j + 1);
                                const bool dist = P.cvdist && __ldg(P.cvdist + j);   // input (s, 0)
                                P.gradA[((size_t)m * P.W + wg) * P.C + j] =
                                    dist ? acc[k][2 * p] : -sn * acc[k][2 * p] + cs * acc[k][2 * p + 1];
                            }
                        }
                    }
                }
                if (fwd && l == L - 1 && ng > 0) P.qsave[qs_off(m, tile, (col0 >> 4), row, P.ntiles)] = apart;
                if (g < G - 1) {
                    // columns past N are K padding of the next GEMM: zero
                    for (int k = ng; k < 2; ++k) zero_a8(Abuf, row, col0 + k * 8, ebn);
                    // a 128-byte K-chunk of the next GEMM's A operand is complete
                    // (this warp's part): every chunk for BF16, every second for FP8
                    if (ebn == 2 || (c & 1)) {
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&S.a_chunk[ebn == 2 ? c : (c >> 1)]));
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&S.acc_empty[b]));
        }
    }
    fence_before();
    __syncthreads();
    // member value A = w_out . h_L + b_out: the 16-column partials in column order
    if (warp >= EPI_WARP0 && warp < EPI_WARP0 + 4) {
        const int row = (warp & 3) * 32 + lane;
        const int wg = tile * 128 + row;
        if (wg < P.W && !S.abort_flag) P.Apart[(size_t)m * P.W + wg] = member_value(P, m, tile, row);
    }
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)P.tmem_cols)
                     : "memory");
    }
}

}  // namespace

size_t rid_mlp_tc_smem_bytes(const TcArgs& P) {
    return 1024 + (size_t)P.Kpmax * 256u + (size_t)P.stages * P.stage_bytes + sizeof(float) * (size_t)(P.L + 1) * P.H;
}

cudaError_t rid_launch_mlp_tc(const TcArgs& P, const CUtensorMap& big, const CUtensorMap& small, cudaStream_t s) {
    if (P.ngemm != P.L && P.ngemm != 2 * P.L) return cudaErrorInvalidValue;
    if (P.ntiles != 1 || P.nacc != 2) return cudaErrorInvalidValue;
    if (P.resnet && !P.rsave) return cudaErrorInvalidValue;
    const size_t smem = rid_mlp_tc_smem_bytes(P);
    const int v = (P.geb[0] == 1 ? 1 : 0) + (P.resnet ? 2 : 0);
    auto kern = v == 0 ? k_mlp_tc<false, false> : v == 1 ? k_mlp_tc<true, false>
              : v == 2 ? k_mlp_tc<false, true> : k_mlp_tc<true, true>;
    static RidOnce once[4];
    if (const cudaError_t e = rid_opt_in(once[v], RID_SMEM_MOST, kern)) return e;
    kern<<<dim3(1, P.M, 1), NTHREADS, smem, s>>>(P, big, small);
    return cudaGetLastError();
}
