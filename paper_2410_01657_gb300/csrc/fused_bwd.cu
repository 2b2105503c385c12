// Fused BF16 backward (adjoint) of the consistent NMP layer, Eq. 3, with
// per-layer recomputation of the MLP activations.
//
// Launch sequence of gnn_mp_backward (BF16):
//   k_proj_fwd    recompute P|Q = x W1a^T | x W1b^T (forward kernel)
//   k_node_bwd    recompute the node MLP from [a*, x], back-propagate dx_out:
//                 da* (FP32) and dx_in = dx_out + d[x part]; dW of the node MLP
//   halo          adjoint of Eq. 5c-5d = the same symmetric copy-sum on da*
//   k_edge_bwd    (edge_bwd.cu) recompute the edge MLP per receiver-aligned tile; the
//                 gradient of e' is de_out + da_i / d_ij (adjoint of Eq. 5b);
//                 back-propagate to de_in = g + W1c^T dz1, write dz1 (the
//                 gradient of the first pre-activation) per edge, sum it over
//                 each receiver's edges into dP (FP32, fixed edge order); dW
//   k_sender_sums, k_proj_bwd    dQ_j = sum of dz1 over the edges sent by j (sender CSR,
//                 fixed order); dx_in += dP W1a + dQ W1b; dW1a, dW1b
//   k_reduce_grads    per-CTA weight-gradient partials summed in a fixed order into dW
// No atomics anywhere: every sum has a fixed order, so results are bitwise
// reproducible.
//
// Weight gradients accumulate in TMEM across all tiles a CTA processes:
// D_k[out][in] += dz_k^T h_k is one tcgen05.mma per 16 rows with both operands
// MN-major views of the tiles the chain already holds in shared memory; a
// constant block with a column of ones appended to h_k yields the bias
// gradient sum_rows dz_k in column `in = H_in` of the same accumulator.
// Thread layout: 128 rows x H/16 column groups of 16 columns.

#include <algorithm>
#include <cstring>

#include "fused.h"
#include "fused_bwd_common.cuh"
#include "plain.h"
#include "profiler.h"

namespace gnn {
namespace fused {

cudaError_t take_device_error_bwd(unsigned int* out) { return take_device_error_word(out); }

// ------------------------------------------------------------------ shared memory plans

struct NodeBwdSmem {
    uint32_t w0, w, ain, ones2, g, hb, ones, gx, par, red, bar, tm, total;
};

template <int H>
__host__ __device__ inline NodeBwdSmem node_bwd_smem(int n_lin) {
    using C = CfgB<H>;
    NodeBwdSmem s;
    s.w0 = 0;
    s.w = align_up(2 * C::WT, 1024);
    s.ain = align_up(s.w + (n_lin - 1) * C::WT, 1024);
    s.ones2 = s.ain + 2 * C::TILE;                 // contiguous after ain: the next N-block of [ain ; ones]
    s.g = align_up(s.ones2 + 128 * C::S2, 1024);
    s.hb = s.g + C::TILE;
    s.ones = align_up(s.hb + (n_lin - 1) * C::TILE, 1024);
    s.gx = align_up(s.ones + 128 * C::S, 1024);         // the tile's dx_out rows (FP32), then its dx_in rows
    s.par = s.gx + 128 * H * 4;
    s.red = s.par + (n_lin + 2) * H * 4;
    s.bar = align_up(s.red + 4 * C::CG * 128 * 4, 8);   // mma, wgrad, ready, h[GNN_MAX_LIN], xa, gx
    s.tm = s.bar + 8 * (5 + GNN_MAX_LIN);
    uint32_t end = s.tm + 16;
    end = end > s.g + 32768 ? end : s.g + 32768;
    s.total = end + 1024;
    return s;
}

struct ProjBwdSmem {
    uint32_t w, a, x, bar, tm, total;
};

template <int H>
__host__ __device__ inline ProjBwdSmem proj_bwd_smem() {
    using C = CfgB<H>;
    ProjBwdSmem s;
    s.w = 0;
    s.a = align_up(2 * C::WT, 1024);
    s.x = s.a + 2 * C::TILE;
    s.bar = align_up(s.x + C::TILE, 8);
    s.tm = s.bar + 16;
    uint32_t end = s.tm + 16;
    end = end > s.a + 32768 ? end : s.a + 32768;
    s.total = end + 1024;
    return s;
}

// TMEM column plans
// Offset of the LayerNorm parameter gradients in a node-adjoint CTA's partials
// (after the weight-gradient blocks [H x (2H+16)] and (n_lin-1) x [H x (H+16)]).
template <int H>
__host__ __device__ inline int64_t node_ln_off(int n_lin) {
    return (int64_t)H * (2 * H + 16) + (int64_t)(n_lin - 1) * H * (H + 16);
}
template <int H>
__host__ __device__ inline uint32_t node_bwd_tcols(int n_lin) {
    return 2 * H + (2 * H + 16) + (n_lin - 1) * (H + 16);
}

// ------------------------------------------------------------------ k_node_bwd

struct NodeBwdArgs {
    const float* a_star;
    const float* x;
    const float* dx_out;   // (tmap_gx; read here to prefetch)
    float* part;           // per-CTA weight-gradient partials
    int64_t pstride;
    int64_t n_rows;
    MlpDev mlp;
    float eps;
    int64_t act_rows;   // SAVED: rows of one activation block of tmap_h (tiles * 128)
};

// SAVED: the forward stored the node MLP's hidden activations (block k, row
// k * act_rows + r, of tmap_h) and its BF16 input rows [a*, x] (tmap_xa); they
// arrive by TMA into the activation buffers and the input tile, each refilled
// with the next tile's rows once its last reader has passed (as in the edge adjoint),
// and only the last Linear is recomputed; a* and x are not read.
//
// A tile is a chain of 8 (5) dependent MMA and epilogue steps, 512 threads with
// 16 columns of a row each; what it moves (five FP32 rows of H per node) travels
// as whole rows: a* and x by coalesced pieces straight into the operand tile,
// dx_out by TMA into gx, where dx_in replaces it, and dx_in and da* (staged over
// the dead dz and h tiles) leave by TMA stores. With per-thread row accesses the
// loads and stores alone held the warps 15 cycles per issue (551k rows at H = 64: 0.52 ms, now
// 0.34; at H = 32 with 7 Linears 0.39 and 0.33).
template <int H, bool SAVED>
__global__ void __launch_bounds__(CfgB<H>::NT, 1) k_node_bwd(const __grid_constant__ CUtensorMap tmap_h,
                                                            const __grid_constant__ CUtensorMap tmap_xa,
                                                            const __grid_constant__ CUtensorMap tmap_gx,
                                                            const __grid_constant__ CUtensorMap tmap_dx,
                                                            const __grid_constant__ CUtensorMap tmap_da,
                                                            NodeBwdArgs A) {
    using C = CfgB<H>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    const int L = A.mlp.n_lin;
    const NodeBwdSmem P = node_bwd_smem<H>(L);
    uint8_t* sW0 = sm + P.w0;
    uint8_t* sW = sm + P.w;
    uint8_t* sAin = sm + P.ain;
    uint8_t* sG = sm + P.g;
    uint8_t* sHB = sm + P.hb;
    uint8_t* sOnes = sm + P.ones;
    float* sPar = reinterpret_cast<float*>(sm + P.par);
    float* sRed = reinterpret_cast<float*>(sm + P.red);
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + P.bar);   // MMA completion
    uint64_t* bar_w = bar + 1;                                  // weight-gradient MMAs of an adjoint step
    uint64_t* ready = bar + 2;                                  // one arrival per warp before an MMA
    uint64_t* h_full = bar + 3;                                 // SAVED: h_k of the tile has landed
    uint64_t* xa_full = bar + 3 + GNN_MAX_LIN;                  // SAVED: the tile's [a*, x] rows have landed
    uint64_t* gx_full = bar + 4 + GNN_MAX_LIN;                  // the tile's dx_out rows have landed
    uint8_t* sGX = sm + P.gx;
    // FP32 da* rows [128 x H]: over dz and h_0; SAVED, where the next h_0 is on its way, over the input tile
    uint8_t* sDA = SAVED ? sAin : sm + P.g;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    constexpr int S = C::S, S2 = C::S2, CW = C::CW;
    const uint32_t NCOLS = pow2_cols(node_bwd_tcols<H>(L));

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, g = warp >> 2, row = 32 * q + lane, c0 = g * CW;

    if (warp == 0) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar_w, 1);
        mbar_init(ready, C::NT / 32);
        mbar_init(gx_full, 1);
        if (SAVED) {
            for (int k = 0; k < L - 1; ++k) mbar_init(h_full + k, 1);
            mbar_init(xa_full, 1);
        }
        fence_mbar_init();
    }
    load_weight(sW0, A.mlp.W[0], 2 * H, 0, H, 2 * H, tid, C::NT);
    for (int k = 1; k < L; ++k) load_weight(sW + (k - 1) * C::WT, A.mlp.W[k], H, 0, H, H, tid, C::NT);
    fill_ones(sm + P.ones2, S2, tid, C::NT);
    fill_ones(sOnes, S, tid, C::NT);
    for (int i = tid; i < L * H; i += C::NT) sPar[i] = A.mlp.b[i / H][i % H];
    for (int i = tid; i < H; i += C::NT) {
        sPar[L * H + i] = A.mlp.gamma[i];
        sPar[(L + 1) * H + i] = A.mlp.beta[i];
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t tWork = tmem;
    auto tDW = [&](int k) -> uint32_t {
        return tmem + (uint32_t)(2 * H + (k == 0 ? 0 : (2 * H + 16) + (k - 1) * (H + 16)));
    };
    // LayerNorm parameter-gradient column sums, per warp (warp_colsum16): one register each
    constexpr int NCH = CW / 16;
    float acc_g[NCH], acc_b[NCH];
#pragma unroll
    for (int i = 0; i < NCH; ++i) acc_g[i] = acc_b[i] = 0.f;
    uint32_t ph = 0, ph_w = 0, ph_rdy = 0;
    bool ok = true, first = true;
    const int64_t n_tiles = (A.n_rows + 127) / 128;
    // MMA hand-off as in the edge adjoint: warps arrive on `ready` after their operand writes and
    // accumulator reads, thread 0 issues, every thread waits on the completion barrier itself
    auto handoff = [&](auto&& issue, uint64_t* done) {
        fence_proxy_async();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(ready);
        if (tid == 0) {
            ok = ok && mbar_wait(ready, ph_rdy);
            ph_rdy ^= 1;
            tc_fence_after();
            if (ok) {
                issue();
                mma_commit(done);
            }
        }
    };
    auto mma_wait = [&]() {
        ok = ok && mbar_wait(bar, ph);
        ph ^= 1;
        __syncwarp();
        tc_fence_after();
    };
    const uint32_t hmask = SAVED ? ((1u << (L - 1)) - 1u) : 0u;
    uint32_t ph_h = 0, h_pend = 0;   // per-thread parity of h_full[k]; thread 0's loads not yet waited for
    auto load_h = [&](int k, int64_t tt) {
        mbar_arrive_expect_tx(h_full + k, C::TILE);
        tma_load_2d(sHB + k * C::TILE, &tmap_h, 0, (int32_t)(k * A.act_rows + tt * 128), h_full + k);
        h_pend |= 1u << k;
    };
    auto wait_h = [&](int k) {
        ok = ok && mbar_wait(h_full + k, (ph_h >> k) & 1u);
        h_pend &= ~(1u << k);
    };
    uint32_t ph_xa = 0;
    bool xa_pend = false;   // thread 0
    auto load_xa = [&](int64_t tt) {
        mbar_arrive_expect_tx(xa_full, 2 * C::TILE);
#pragma unroll
        for (int kb = 0; kb < 2 * H / (S2 / 2); ++kb)
            tma_load_2d(sAin + kb * 128 * S2, &tmap_xa, kb * (S2 / 2), (int32_t)(tt * 128), xa_full);
        xa_pend = true;
    };
    if (SAVED && tid == 0 && (int64_t)blockIdx.x < n_tiles) {
        for (int k = 0; k < L - 1; ++k) load_h(k, blockIdx.x);
        load_xa(blockIdx.x);
    }
    uint32_t ph_gx = 0;
    bool gx_pend = false;   // thread 0
    auto load_gx = [&](int64_t tt) {
        mbar_arrive_expect_tx(gx_full, 128 * H * 4);
        tma_f32_tile<H>(sGX, &tmap_gx, tt * 128, gx_full);
        gx_pend = true;
    };
    if (tid == 0 && (int64_t)blockIdx.x < n_tiles) load_gx(blockIdx.x);

    for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        if (tid == 0 && t + gridDim.x < n_tiles) {   // the next tile's input rows into L2
            const int64_t rn = (t + gridDim.x) * 128;
            const uint32_t nb = (uint32_t)(std::min<int64_t>(128, A.n_rows - rn) * H * 4);
            prefetch_l2(A.a_star + rn * H, nb);
            prefetch_l2(A.x + rn * H, nb);
            prefetch_l2(A.dx_out + rn * H, nb);
        }
        if constexpr (!SAVED) {   // the operand tile [a*, x] by pieces of four columns: consecutive threads, whole rows
            constexpr int PPR = H / 4, IT = 128 * PPR / C::NT;
            const int nv = (int)std::min<int64_t>(128, A.n_rows - t * 128);
            float4 av[IT], xv[IT];
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                const int p = tid + i * C::NT;
                av[i] = xv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (p / PPR < nv) {
                    av[i] = __ldg(reinterpret_cast<const float4*>(A.a_star + t * 128 * H) + p);
                    xv[i] = __ldg(reinterpret_cast<const float4*>(A.x + t * 128 * H) + p);
                }
            }
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                const int p = tid + i * C::NT, rr = p / PPR, c = 4 * (p % PPR);
                *reinterpret_cast<uint2*>(sAin + tile_off(rr, c, 128, S2)) =
                    make_uint2(pack_bf16x2(av[i].x, av[i].y), pack_bf16x2(av[i].z, av[i].w));
                *reinterpret_cast<uint2*>(sAin + tile_off(rr, H + c, 128, S2)) =
                    make_uint2(pack_bf16x2(xv[i].x, xv[i].y), pack_bf16x2(xv[i].z, xv[i].w));
            }
        }
        // (thread 0 issues the tile's first MMA after the previous tile's da* store has read the dz and h
        // tiles: nobody writes those before that MMA has completed)
        if (tid == 0) bulk_wait_read_all();
        // ---- recompute the chain (SAVED: only the last Linear, from the saved h_{L-2})
        float v[CW];
        if constexpr (SAVED) {
            if (tid == 0) {
                wait_h(L - 2);
                ok = ok && mbar_wait(xa_full, ph_xa);   // the input tile of the step-0 weight gradient
                ph_xa ^= 1;
                xa_pend = false;
                tc_fence_after();
                if (ok) {
                    issue_mma(tWork, sHB + (L - 2) * C::TILE, sW + (L - 2) * C::WT, H, H);
                    mma_commit(bar);
                }
            }
            mma_wait();
            ld_acc<CW>(tWork, q, c0, v);
            add_bias2<CW>(v, sPar + (L - 1) * H + c0);
        } else {
            handoff([&] { issue_mma(tWork, sAin, sW0, H, 2 * H); }, bar);
        }
        for (int k = 0; k < (SAVED ? 0 : L); ++k) {
            mma_wait();
            ld_acc<CW>(tWork, q, c0, v);
            add_bias2<CW>(v, sPar + k * H + c0);
            if (k < L - 1) {
                elu_inplace2<CW>(v);
                st_row_tile<CW>(sHB + k * C::TILE, row, c0, S, v);
                handoff([&] { issue_mma(tWork, sHB + k * C::TILE, sW + k * C::WT, H, H); }, bar);
            }
        }
        tc_fence_before();
        float gv[CW];   // dx_out (zero past n_rows)
        ok = ok && mbar_wait(gx_full, ph_gx);
        ph_gx ^= 1;
        __syncwarp();
        auto load_gv = [&] {
#pragma unroll
            for (int i = 0; i < CW / 4; ++i) {
                const float4 z = ld_f32x4_tile<H>(sGX, row, c0 + 4 * i);
                gv[4 * i] = z.x; gv[4 * i + 1] = z.y; gv[4 * i + 2] = z.z; gv[4 * i + 3] = z.w;
            }
        };
        load_gv();
        // ---- LayerNorm adjoint (statistics and adjoint sums in one exchange)
        float dz[CW];
#pragma unroll
        for (int i = 0; i < CW; ++i) dz[i] = gv[i] * sPar[L * H + c0 + i];
        float mean, rstd, s1, s2;
        row_stats_adj<H, C::CG, CW>(v, dz, sRed, row, g, A.eps, mean, rstd, s1, s2);
#pragma unroll
        for (int i = 0; i < CW; ++i) {
            v[i] = (v[i] - mean) * rstd;   // xhat
            dz[i] = rstd * (dz[i] - s1 - v[i] * s2);
        }
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            float t16[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) t16[i] = gv[16 * j + i] * v[16 * j + i];
            acc_g[j] += warp_colsum16(t16, lane);
            acc_b[j] += warp_colsum16(gv + 16 * j, lane);
        }
        // ---- chain adjoint, layer L-1 .. 0
        for (int k = L - 1; k >= 0; --k) {
            if (k < L - 1) {   // the previous step's wgrad reads sG
                ok = ok && mbar_wait(bar_w, ph_w);
                ph_w ^= 1;
            }
            if (SAVED && k > 0) wait_h(k - 1);   // this step's wgrad operand and ELU derivative input
            st_row_tile<CW>(sG, row, c0, S, dz);
            handoff([&] {
                if (k == 0) {
                    issue_dgrad(tWork, sG, S, sW0, S2, H, (uint32_t)H * S2, 2 * H, H);
                    mma_commit(bar);
                    issue_wgrad(tDW(0), sG, S, 128u * S, sAin, S2, 128u * S2, 2 * H + 16, !first);
                } else {
                    issue_dgrad(tWork, sG, S, sW + (k - 1) * C::WT, S, H, (uint32_t)H * S, H, H);
                    mma_commit(bar);
                    uint8_t* hk = sHB + (k - 1) * C::TILE;
                    issue_wgrad(tDW(k), sG, S, 128u * S, hk, S, (uint32_t)(smem_u32(sOnes) - smem_u32(hk)), H + 16,
                                !first);
                }
            }, bar_w);
            // SAVED: h_k's last reader (step k + 1) is done: the next tile's h_k goes there
            if (SAVED && tid == 0 && ok && k <= L - 2 && t + gridDim.x < n_tiles) load_h(k, t + gridDim.x);
            mma_wait();
            if (k > 0) {
                float dh[CW], hv[CW];
                ld_acc<CW>(tWork, q, c0, dh);
                ld_row_tile<CW>(sHB + (k - 1) * C::TILE, row, c0, S, hv);
                elu_bwd2<CW>(dz, dh, hv);
            } else {
                float da[CW], dxp[CW];
                ld_acc<CW>(tWork, q, c0, da);
                ld_acc<CW>(tWork, q, H + c0, dxp);
                ok = ok && mbar_wait(bar_w, ph_w);   // dz and h are dead
#pragma unroll
                for (int i = 0; i < CW / 4; ++i) {
                    st_f32x4_tile<H>(sDA, row, c0 + 4 * i, make_float4(da[4 * i], da[4 * i + 1], da[4 * i + 2], da[4 * i + 3]));
                    st_f32x4_tile<H>(sGX, row, c0 + 4 * i,
                                     make_float4(gv[4 * i] + dxp[4 * i], gv[4 * i + 1] + dxp[4 * i + 1],
                                                 gv[4 * i + 2] + dxp[4 * i + 2], gv[4 * i + 3] + dxp[4 * i + 3]));
                }
                fence_proxy_async();
            }
            tc_fence_before();
        }
        first = false;
        ph_w ^= 1;
        ph_h ^= hmask;
        if (tid == 0) gx_pend = false;
        __syncwarp();
        if (__syncthreads_or(!ok)) break;   // the block leaves together after a timeout
        tc_fence_after();
        if (tid == 0) {   // da* and dx_in leave; the next tile's rows come once they have been read
            constexpr int BW = H < 32 ? H : 32;
#pragma unroll
            for (int b = 0; b < H / BW; ++b) {
                tma_store_2d(&tmap_dx, b * BW, (int32_t)(t * 128), sGX + b * 128 * BW * 4);
                tma_store_2d(&tmap_da, b * BW, (int32_t)(t * 128), sDA + b * 128 * BW * 4);
            }
            bulk_commit();
            if (t + gridDim.x < n_tiles) {
                bulk_wait_read_all();
                load_gx(t + gridDim.x);
                if (SAVED) load_xa(t + gridDim.x);
            }
        }
    }
    if (tid == 0) {
        if (gx_pend) mbar_wait(gx_full, ph_gx);
        bulk_wait_all();
    }
    if (SAVED && tid == 0) {   // loads issued before a timeout ended the tile loop
        for (int k = 0; k < L - 1; ++k)
            if ((h_pend >> k) & 1u) mbar_wait(h_full + k, (ph_h >> k) & 1u);
        if (xa_pend) mbar_wait(xa_full, ph_xa);
    }
    // ---- flush the CTA's partial gradients
    tc_fence_before();
    ok = __syncthreads_and(ok) != 0;
    tc_fence_after();
    float* part = A.part + (int64_t)blockIdx.x * A.pstride;
    if (ok) {
        int64_t off = 0;
        for (int k = 0; k < L; ++k) {
            const int N = k == 0 ? 2 * H + 16 : H + 16;
            if (!first) flush_acc<C::CG>(tDW(k), N, H, q, lane, g, part + off);
            else
                for (int i = tid; i < H * N; i += C::NT) part[off + i] = 0.f;
            off += (int64_t)H * N;
        }
    }
    colsum_store<H, NCH>(acc_g, sRed, q, lane, c0, tid, C::NT, part + node_ln_off<H>(L));
    colsum_store<H, NCH>(acc_b, sRed, q, lane, c0, tid, C::NT, part + node_ln_off<H>(L) + H);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ------------------------------------------------------------------ k_proj_bwd

struct ProjBwdArgs {
    const float* x;
    const float* dP;
    const __nv_bfloat16* dQ;   // sender-side sums of dz1 (k_sender_sums), as the operand rounds them
    const float* W1;
    float* dx_in;       // += dP W1a + dQ W1b
    float* part;
    int64_t pstride;
    int64_t n_rows;
};

// dQ_j = sum of dz1 over the edges sent by j, in edge order, FP32, rounded to
// BF16 once (the operand that k_proj_bwd multiplies). One thread per 8 columns
// of a row: the gathers of whole 16-byte pieces are the kernel, so it wants
// every warp the SM holds; inside the projection adjoint (4 to 8 warps per SM
// at H <= 64, 16 at H = 128) they were a chain of exposed latencies.
template <int H>
__global__ void __launch_bounds__(256) k_sender_sums(const int32_t* __restrict__ t_ptr,
                                                     const int32_t* __restrict__ t_eid,
                                                     const __nv_bfloat16* __restrict__ dz1, int64_t n_rows,
                                                     __nv_bfloat16* __restrict__ dQ) {
    constexpr int PPR = H / 8, UB = 6;   // a lattice node sends to six others
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t r = i / PPR;
    const int c = (int)(i % PPR) * 8;
    if (r >= n_rows) return;
    float dq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int32_t k1 = __ldg(t_ptr + r + 1);
    for (int32_t kb = __ldg(t_ptr + r); kb < k1; kb += UB) {
        uint4 z[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u)
            z[u] = kb + u < k1 ? __ldg(reinterpret_cast<const uint4*>(dz1 + (int64_t)__ldg(t_eid + kb + u) * H + c))
                               : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            if (kb + u < k1) {
                const uint32_t w[4] = {z[u].x, z[u].y, z[u].z, z[u].w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float f0, f1;
                    unpack_bf16x2(w[k], f0, f1);
                    dq[2 * k] += f0;
                    dq[2 * k + 1] += f1;
                }
            }
        }
    }
    st_bf16x8(dQ + r * H + c, dq);
}

// Thread layout: 128 rows x H/32 column groups of 32 columns.
template <int H>
struct CfgP {
    static constexpr int S = span_of(H);
    static constexpr int S2 = span_of(2 * H);
    static constexpr int CG = H >= 32 ? H / 32 : 1;
    static constexpr int CW = H / CG;
    static constexpr int NT = 128 * CG;
};

// One CTA per SM (the launch says why); the register bound leaves room for two up to H = 64.
// The weight gradient [dW1a; dW1b] = [dP dQ]^T x is one M = 2H MMA up to
// H = 64 and two M = 128 halves at H = 128.
template <int H>
__global__ void __launch_bounds__(CfgP<H>::NT, H >= 128 ? 1 : 2) k_proj_bwd(ProjBwdArgs A) {
    using C = CfgP<H>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    const ProjBwdSmem P = proj_bwd_smem<H>();
    uint8_t* sW = sm + P.w;
    uint8_t* sA = sm + P.a;
    uint8_t* sX = sm + P.x;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + P.bar);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    constexpr int S = C::S, S2 = C::S2, CW = C::CW;
    constexpr bool MSPLIT = 2 * H > 128;
    constexpr uint32_t NCOLS = pow2_cols(MSPLIT ? 3 * H : 2 * H);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, g = warp >> 2, row = 32 * q + lane, c0 = g * CW;

    if (warp == 0) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    // [W1a; W1b] as a [2H x H] row tile (rows = stacked outputs, contiguous = inputs)
    load_weight(sW, A.W1, 3 * H, 0, H, H, tid, C::NT, 2 * H, 0);
    load_weight(sW, A.W1, 3 * H, H, H, H, tid, C::NT, 2 * H, H);
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t tWork = tmem, tDW = tmem + H;
    uint32_t ph = 0;
    bool ok = true, first = true;
    const int64_t n_tiles = (A.n_rows + 127) / 128;

    for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        if (tid == 0 && t + gridDim.x < n_tiles) {   // the next tile's input rows into L2
            const int64_t rn = (t + gridDim.x) * 128;
            const int64_t nr = std::min<int64_t>(128, A.n_rows - rn);
            prefetch_l2(A.dP + rn * H, (uint32_t)(nr * H * 4));
            prefetch_l2(A.x + rn * H, (uint32_t)(nr * H * 4));
            prefetch_l2(A.dQ + rn * H, (uint32_t)(nr * H * 2));
            prefetch_l2(A.dx_in + rn * H, (uint32_t)(nr * H * 4));   // its update
        }
        // the operand tiles [dP dQ] and x, filled by pieces of four columns: consecutive threads
        // read consecutive pieces, so every global access is a run of whole rows
        constexpr int PPR = H / 4, IT = 128 * PPR / C::NT, UB = 4;   // pieces per row; steps; steps in flight
        const int64_t rt = t * 128;
        const int nv = (int)std::min<int64_t>(128, A.n_rows - rt);
#pragma unroll 1
        for (int i0 = 0; i0 < IT; i0 += UB) {
            float4 dp[UB], xv[UB];
            uint2 dq[UB];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int p = tid + (i0 + u) * C::NT, rr = p / PPR, c = 4 * (p % PPR);
                dp[u] = xv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                dq[u] = make_uint2(0u, 0u);
                if (rr < nv) {
                    const int64_t o = (rt + rr) * H + c;
                    dp[u] = __ldg(reinterpret_cast<const float4*>(A.dP + o));
                    xv[u] = __ldg(reinterpret_cast<const float4*>(A.x + o));
                    dq[u] = __ldg(reinterpret_cast<const uint2*>(A.dQ + o));
                }
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int p = tid + (i0 + u) * C::NT, rr = p / PPR, c = 4 * (p % PPR);
                *reinterpret_cast<uint2*>(sA + tile_off(rr, c, 128, S2)) =
                    make_uint2(pack_bf16x2(dp[u].x, dp[u].y), pack_bf16x2(dp[u].z, dp[u].w));
                *reinterpret_cast<uint2*>(sA + tile_off(rr, H + c, 128, S2)) = dq[u];
                *reinterpret_cast<uint2*>(sX + tile_off(rr, c, 128, S)) =
                    make_uint2(pack_bf16x2(xv[u].x, xv[u].y), pack_bf16x2(xv[u].z, xv[u].w));
            }
        }
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            issue_dgrad(tWork, sA, S2, sW, S, 2 * H, (uint32_t)(2 * H) * S, H, 2 * H);
            if constexpr (MSPLIT) {   // dW1a from the dP columns, dW1b from the dQ columns
                issue_wgrad(tDW, sA, S2, 128u * S2, sX, S, 128u * S, H, !first);
                issue_wgrad(tDW + H, sA + (H / (S2 / 2)) * 128 * S2, S2, 128u * S2, sX, S, 128u * S, H, !first);
            } else {
                issue_wgrad(tDW, sA, S2, 128u * S2, sX, S, 128u * S, H, !first);
            }
            mma_commit(bar);
        }
        ok = block_wait(bar, ph, tid);
        ph ^= 1;
        tc_fence_after();
        if (!ok) break;
        float d[CW];
        ld_acc<CW>(tWork, q, c0, d);
        tc_fence_before();
        // dx_in += d by the same pieces: the MMAs have read the operand tile, which now stages the
        // FP32 rows [128 x H] (16-byte pieces swizzled by row)
        float4* sD = reinterpret_cast<float4*>(sA);
        constexpr int SWM = PPR >= 8 ? 7 : PPR - 1;
#pragma unroll
        for (int i = 0; i < CW / 4; ++i)
            sD[row * PPR + (((c0 / 4) + i) ^ (row & SWM))] =
                make_float4(d[4 * i], d[4 * i + 1], d[4 * i + 2], d[4 * i + 3]);
        __syncthreads();
#pragma unroll 1
        for (int i0 = 0; i0 < IT; i0 += UB) {
            float4 o[UB];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int p = tid + (i0 + u) * C::NT, rr = p / PPR;
                if (rr < nv) o[u] = *(reinterpret_cast<const float4*>(A.dx_in + rt * H) + p);
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int p = tid + (i0 + u) * C::NT, rr = p / PPR, c = p % PPR;
                if (rr < nv) {
                    const float4 v = sD[rr * PPR + (c ^ (rr & SWM))];
                    *(reinterpret_cast<float4*>(A.dx_in + rt * H) + p) =
                        make_float4(o[u].x + v.x, o[u].y + v.y, o[u].z + v.z, o[u].w + v.w);
                }
            }
        }
        first = false;
        __syncthreads();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    float* part = A.part + (int64_t)blockIdx.x * A.pstride;
    if (ok) {
        if (first) {
            for (int i = tid; i < 2 * H * H; i += C::NT) part[i] = 0.f;
        } else if constexpr (MSPLIT) {
            flush_acc<C::CG>(tDW, H, H, q, lane, g, part);
            flush_acc<C::CG>(tDW + H, H, H, q, lane, g, part + H * H);
        } else {
            flush_acc<C::CG>(tDW, H, 2 * H, q, lane, g, part);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ------------------------------------------------------------------ partial reduction

// dst[r*dst_ld + c] += sum over CTAs b of part[b*pstride + src_off + r*src_ld + c]. A block
// takes 32 elements; its eight warps take every eighth CTA, in order, eight loads
// in flight each, and their sums are added in warp order: the sum over 152 CTAs
// is three round trips to L2 where one thread per element made ten (8 us a
// launch at 0.1 to 12 MB of partials; 3 now).
struct RedArgs {
    RedSeg seg[MAX_SEGS];
    int n_seg;
    int blk[MAX_SEGS + 1];   // first block of each segment
};

__global__ void __launch_bounds__(256) k_reduce_grads(const __grid_constant__ RedArgs A) {
    __shared__ float red[8][32];
    int s = 0;
    while ((int)blockIdx.x >= A.blk[s + 1]) ++s;
    const RedSeg& sg = A.seg[s];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j = ((int)blockIdx.x - A.blk[s]) * 32 + lane;
    const int r = j / sg.cols, c = j % sg.cols;
    const bool in = r < sg.rows;
    float acc = 0.f;
    if (in) {
        const float* p = sg.part + sg.src_off + (int64_t)r * sg.src_ld + c;
        constexpr int U = 8;
        for (int b0 = w; b0 < sg.n_cta; b0 += 8 * U) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = b0 + 8 * u < sg.n_cta ? __ldg(p + (int64_t)(b0 + 8 * u) * sg.pstride) : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) acc += v[u];
        }
    }
    red[w][lane] = acc;
    __syncthreads();
    if (w == 0 && in) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += red[k][lane];
        sg.dst[(int64_t)r * sg.dst_ld + c] += t;
    }
}

// =================================================================== host side

int reduce_grads(RedSeg* segs, int n, cudaStream_t s) {
    RedArgs A{};
    GNN_REQUIRE(n <= MAX_SEGS, GNN_EUNSUPPORTED, "reduce_grads: too many segments");
    auto flush = [&]() -> int {
        const int blocks = A.blk[A.n_seg];
        if (blocks == 0) return GNN_OK;
        {
            ProfScope _ps(s, "k_reduce_grads");
            k_reduce_grads<<<blocks, 256, 0, s>>>(A);
        }
        A.n_seg = 0;
        GNN_LAUNCH_CHECK("k_reduce_grads");
        return GNN_OK;
    };
    auto dest = [](const RedSeg& g) { return Dest{g.dst, g.dst_ld, g.rows, g.cols}; };
    int rc;
    for (int i = 0; i < n; ++i) {
        if (segs[i].n_cta <= 0) continue;
        bool apart = true;
        for (int k = 0; k < A.n_seg; ++k) apart = apart && !may_overlap(dest(A.seg[k]), dest(segs[i]));
        if (!apart && (rc = flush())) return rc;
        A.seg[A.n_seg] = segs[i];
        A.blk[A.n_seg + 1] = A.blk[A.n_seg] + (segs[i].rows * segs[i].cols + 31) / 32;
        ++A.n_seg;
    }
    return flush();
}

int reduce_grads(RedSeg* segs, int n, const float* part, int64_t pstride, int n_cta, cudaStream_t s) {
    for (int i = 0; i < n; ++i) {
        segs[i].part = part;
        segs[i].pstride = pstride;
        segs[i].n_cta = n_cta;
    }
    return reduce_grads(segs, n, s);
}

namespace {

using namespace host;

struct BwdWs {
    __nv_bfloat16* pq;
    float* a;
    float* da;
    float* dP;
    __nv_bfloat16* dz1;
    float *part_node, *part_edge, *part_proj;
    size_t bytes;
};

int64_t edge_pstride(int H, int L) { return (int64_t)L * H * (H + 16) + 2 * H; }
int64_t node_pstride(int H, int L) { return (int64_t)H * (2 * H + 16) + (int64_t)(L - 1) * H * (H + 16) + 2 * H; }
int64_t proj_pstride(int H) { return (int64_t)2 * H * H; }

BwdWs carve_bwd(void* ws, const gnn_graph_dev& G, int H, int Le, int Ln, bool need_a) {
    BwdWs w{};
    size_t off = 0;
    auto take = [&](size_t n) {
        off = (off + 255) & ~(size_t)255;
        void* p = ws ? (char*)ws + off : nullptr;
        off += n;
        return p;
    };
    const int64_t NR = G.n_rows, E = G.n_edges;
    const int64_t ncta = num_sms();
    w.pq = (__nv_bfloat16*)take((size_t)NR * 2 * H * 2);
    w.a = need_a ? (float*)take((size_t)NR * H * 4) : nullptr;
    w.da = (float*)take((size_t)NR * H * 4);
    w.dP = (float*)take((size_t)NR * H * 4);
    w.dz1 = (__nv_bfloat16*)take((size_t)E * H * 2);
    // per-CTA weight-gradient partials, apart, so that one launch sums them all: at most one CTA per SM and
    // row tile (the edge kernel's tiles may change after the workspace has been sized)
    const int64_t nrow = std::min(ncta, (NR + 127) / 128);
    w.part_node = (float*)take((size_t)nrow * node_pstride(H, Ln) * 4);
    w.part_edge = (float*)take((size_t)ncta * edge_pstride(H, Le) * 4);
    w.part_proj = (float*)take((size_t)nrow * proj_pstride(H) * 4);
    w.bytes = off + 256;
    return w;
}

template <int H>
int proj_backward_h(const gnn_graph_dev& G, const gnn_mp_params& W, const float* x_in, const float* dP,
                    const __nv_bfloat16* dz1, __nv_bfloat16* dQ, float* dx_in, const gnn_mp_params& dW, float* part,
                    RedSeg* seg, int* n_seg, cudaStream_t s) {
    *n_seg = 0;
    const int64_t NR = G.n_rows;
    if (NR == 0) return GNN_OK;
    ProjBwdArgs A;
    A.x = x_in;
    A.dP = dP;
    A.dQ = dQ;
    A.W1 = W.edge.W[0];
    A.dx_in = dx_in;
    A.part = part;
    A.pstride = proj_pstride(H);
    A.n_rows = NR;
    {
        ProfScope _ps(s, "k_sender_sums");
        k_sender_sums<H><<<(unsigned)((NR * (H / 8) + 255) / 256), 256, 0, s>>>(G.t_ptr, G.t_eid, dz1, NR, dQ);
    }
    GNN_LAUNCH_CHECK("k_sender_sums");
    const ProjBwdSmem P = proj_bwd_smem<H>();
    int grid;
    int rc = persistent_grid(k_proj_bwd<H>, CfgP<H>::NT, P.total, pow2_cols(2 * H > 128 ? 3 * H : 2 * H),
                             (NR + 127) / 128, &grid);
    if (rc) return rc;
    // One CTA per SM although two fit: the tensor core truncates its running sums, so the number of
    // tiles one accumulator takes is part of dW1a's and dW1b's value (2 CTAs: 2e-5 apart at 6M rows).
    grid = std::min(grid, num_sms());
    {
        ProfScope _ps(s, "k_proj_bwd");
        k_proj_bwd<H><<<grid, CfgP<H>::NT, P.total, s>>>(A);
    }
    GNN_LAUNCH_CHECK("k_proj_bwd");
    seg[0] = RedSeg{dW.edge.W[0], 3 * H, H, H, 0, H, part, A.pstride, grid};                     // dW1a -> W1[:, 0:H]
    seg[1] = RedSeg{dW.edge.W[0] + H, 3 * H, H, H, (int64_t)H * H, H, part, A.pstride, grid};    // dW1b -> W1[:, H:2H]
    *n_seg = 2;
    return GNN_OK;
}

template <int H>
int backward_h(const gnn_graph_dev& G, const gnn_mp_config& cfg, const gnn_mp_params& W, const float* x_in,
               const __nv_bfloat16* e_in, const float* a_star, const float* dx_out, const __nv_bfloat16* de_out,
               float* dx_in, __nv_bfloat16* de_in, const gnn_mp_params& dW, void* ws, size_t ws_bytes,
               cudaStream_t s, const __nv_bfloat16* act) {
    using C = CfgB<H>;
    const int Le = W.edge.n_lin, Ln = W.node.n_lin;
    auto deep = [](int n) { return edge_backward_supported(H, n) && node_bwd_tcols<H>(n) <= 512; };
    int most = GNN_MAX_LIN;
    while (most > 0 && !deep(most)) --most;
    GNN_REQUIRE(Le <= most && Ln <= most, GNN_EUNSUPPORTED,
                "gnn_mp_backward: BF16 backward at H=%d supports at most %d Linear layers per MLP", H, most);
    BwdWs w = carve_bwd(ws, G, H, Le, Ln, a_star == nullptr);
    GNN_REQUIRE(ws_bytes >= w.bytes, GNN_ENOMEM, "gnn_mp_backward: workspace too small");
    const int64_t NR = G.n_rows, E = G.n_edges;
    if (NR == 0) return GNN_OK;
    int rc;
    // 0. recompute P|Q (and a* when it was not saved); saved activations need no P|Q
    if (!act || !a_star) {
        if ((rc = proj_forward(G, H, W, x_in, w.pq, s))) return rc;
    }
    if (!a_star) {
        if ((rc = aggregate_forward(G, cfg, W, e_in, w.pq, nullptr, w.a, s))) return rc;
    }
    const float* astar = a_star ? a_star : w.a;
    const int nsm = num_sms();
    RedSeg seg[MAX_SEGS];
    int n = 0;
    // 1. node MLP adjoint
    {
        NodeBwdArgs A;
        A.a_star = astar;
        A.x = x_in;
        A.dx_out = dx_out;
        A.part = w.part_node;
        A.pstride = node_pstride(H, Ln);
        A.n_rows = NR;
        A.mlp = mlp_dev(W.node);
        A.eps = cfg.ln_eps;
        A.act_rows = (NR + 127) / 128 * 128;
        const NodeBwdSmem P = node_bwd_smem<H>(Ln);
        CUtensorMap tm_hn, tm_xa, tm_gx, tm_dx, tm_da;
        std::memset(&tm_hn, 0, sizeof(tm_hn));
        std::memset(&tm_xa, 0, sizeof(tm_xa));
        if ((rc = make_f32_tmap(&tm_gx, dx_out, NR, H))) return rc;
        if ((rc = make_f32_tmap(&tm_dx, dx_in, NR, H))) return rc;
        if ((rc = make_f32_tmap(&tm_da, w.da, NR, H))) return rc;
        if (act) {
            const __nv_bfloat16* an = act + mp_act_elems_edge(G, W, H);
            if ((rc = make_row_tmap(&tm_hn, an, (int64_t)(Ln - 1) * A.act_rows, H))) return rc;
            if ((rc = make_row_tmap(&tm_xa, an + (int64_t)(Ln - 1) * A.act_rows * H, A.act_rows, 2 * H))) return rc;
        }
        int grid = 0;
        auto run = [&](auto kern) -> int {
            int r = persistent_grid(kern, C::NT, P.total, pow2_cols(node_bwd_tcols<H>(Ln)), (NR + 127) / 128, &grid);
            if (r) return r;
            grid = std::min(grid, nsm);
            {
                ProfScope _ps(s, "k_node_bwd");
                kern<<<grid, C::NT, P.total, s>>>(tm_hn, tm_xa, tm_gx, tm_dx, tm_da, A);
            }
            GNN_LAUNCH_CHECK("k_node_bwd");
            return GNN_OK;
        };
        if ((rc = act ? run(k_node_bwd<H, true>) : run(k_node_bwd<H, false>))) return rc;
        int64_t off = 0;
        auto add = [&](float* dst, int ld, int rows, int cols, int64_t src, int64_t src_ld) {
            seg[n++] = RedSeg{dst, ld, rows, cols, src, src_ld, A.part, A.pstride, grid};
        };
        for (int k = 0; k < Ln; ++k) {
            const int in = k == 0 ? 2 * H : H;
            const int N = in + 16;
            add(dW.node.W[k], in, H, in, off, N);
            add(dW.node.b[k], 1, H, 1, off + in, N);
            off += (int64_t)H * N;
        }
        add(dW.node.gamma, H, 1, H, off, 0);
        add(dW.node.beta, H, 1, H, off + H, 0);
    }
    // 2. adjoint of the halo swap + sync
    if (cfg.halo_mode == GNN_HALO_SYNC) {
        if ((rc = plain::halo(G, w.da, H, s))) return rc;
    }
    // 3. edge MLP adjoint
    if (E > 0) {
        EdgeBackward o{};
        o.pq = w.pq;
        o.da = w.da;
        o.e_in = e_in;
        o.de_out = de_out;
        o.act = act;
        o.de_in = de_in;
        o.dz1 = w.dz1;
        o.dP = w.dP;
        o.part = w.part_edge;
        o.pstride = edge_pstride(H, Le);
        o.eps = cfg.ln_eps;
        int grid = 0;
        if ((rc = edge_backward(G, H, W, o, &grid, s))) return rc;
        int64_t off = 0;
        auto add = [&](float* dst, int ld, int rows, int cols, int64_t src, int64_t src_ld) {
            seg[n++] = RedSeg{dst, ld, rows, cols, src, src_ld, o.part, o.pstride, grid};
        };
        for (int k = 0; k < Le; ++k) {
            const int N = H + 16;
            if (k == 0) add(dW.edge.W[0] + 2 * H, 3 * H, H, H, off, N);   // W1c columns of W1
            else add(dW.edge.W[k], H, H, H, off, N);
            add(dW.edge.b[k], 1, H, 1, off + H, N);
            off += (int64_t)H * N;
        }
        add(dW.edge.gamma, H, 1, H, off, 0);
        add(dW.edge.beta, H, 1, H, off + H, 0);
    } else {
        GNN_CUDA_CHECK(cudaMemsetAsync(w.dP, 0, sizeof(float) * NR * H, s), "memset");
    }
    // 4. projection adjoint: sender-side sums, dx_in += [dP dQ] [W1a; W1b], dW1a, dW1b
    // (P|Q is done with)
    int np = 0;
    if ((rc = proj_backward_h<H>(G, W, x_in, w.dP, w.dz1, w.pq, dx_in, dW, w.part_proj, seg + n, &np, s))) return rc;
    return reduce_grads(seg, n + np, s);
}

}  // namespace

size_t mp_backward_ws(const gnn_graph_dev& G, const gnn_mp_config& cfg, const gnn_mp_params& W) {
    if (cfg.hidden == 128) return backward_h128_ws(G, W);
    return carve_bwd(nullptr, G, cfg.hidden, W.edge.n_lin, W.node.n_lin, true).bytes;
}

int proj_backward128(const gnn_graph_dev& G, const gnn_mp_params& W, const float* x_in, const float* dP,
                     const __nv_bfloat16* dz1, __nv_bfloat16* dQ, float* dx_in, const gnn_mp_params& dW, float* part,
                     cudaStream_t s) {
    RedSeg seg[2];
    int n = 0;
    int rc = proj_backward_h<128>(G, W, x_in, dP, dz1, dQ, dx_in, dW, part, seg, &n, s);
    return rc ? rc : reduce_grads(seg, n, s);
}

int mp_backward(const gnn_graph_dev& G, const gnn_mp_config& cfg, const gnn_mp_params& W, const float* x_in,
                const __nv_bfloat16* e_in, const float* a_star, const float* dx_out, const __nv_bfloat16* de_out,
                float* dx_in, __nv_bfloat16* de_in, const gnn_mp_params& dW, void* ws, size_t ws_bytes,
                cudaStream_t s, const __nv_bfloat16* act) {
    if (!mp_act_bytes(G, cfg, W)) act = nullptr;
    switch (cfg.hidden) {
        case 16: return backward_h<16>(G, cfg, W, x_in, e_in, a_star, dx_out, de_out, dx_in, de_in, dW, ws, ws_bytes, s, act);
        case 32: return backward_h<32>(G, cfg, W, x_in, e_in, a_star, dx_out, de_out, dx_in, de_in, dW, ws, ws_bytes, s, act);
        case 64: return backward_h<64>(G, cfg, W, x_in, e_in, a_star, dx_out, de_out, dx_in, de_in, dW, ws, ws_bytes, s, act);
        case 128: return backward_h128(G, cfg, W, x_in, e_in, a_star, dx_out, de_out, dx_in, de_in, dW, ws, ws_bytes, s);
        default:
            return set_error(GNN_EUNSUPPORTED, "gnn_mp_backward: the BF16 backward covers H in {16, 32, 64, 128}");
    }
}

}  // namespace fused
}  // namespace gnn
