// Edge adjoint of the fused BF16 backward at H <= 64 (Eq. 3 through Eq. 5a-5b):
// per receiver-aligned tile, recompute the edge MLP (or load its saved
// activations), form the gradient of e' = de_out + da_i / d_ij, back-propagate
// to de_in = g + W1c^T dz_0, write dz_0 per edge and its receiver sums dP, and
// accumulate every weight gradient.
//
// What bounds it: a tile is a chain of 8 (recomputing, 4 Linears) or 5
// dependent MMA -> TMEM load -> FP32 epilogue -> shared-memory operand steps.
// With one tile per SM the warps issue 43 % of the time and wait for MMA round
// trips the rest. So NG groups of warps take alternate tiles of a CTA, each
// with its own tiles, accumulator and barriers, and one group's epilogues run
// in the other's round trips. Two tiles at H = 64 fit because a tile has no
// buffer of its own for its gradients: dz_{L-1} replaces the de_out rows once
// they are read, and dz_k replaces h_k, which its own epilogue has just read
// and whose weight gradient (step k + 1) has completed.
//
// The weight-gradient accumulators D_k[out][in | ones] fill TMEM and are shared
// by the groups. Their MMAs are issued in tile order: per layer a turn goes round
// the groups (one barrier each), so the FP32 sums have a fixed order and
// results stay bitwise reproducible. Groups run in antiphase, so a turn has
// nearly always come long before it is needed.
//
// Measured on 3.23M edges (25,793 tiles): H = 64 recomputing 1.87 -> 1.60 ms, from
// saved activations (3.38M edges) 1.47 -> 1.05 ms, H = 32 with 7 Linears 1.84 ->
// 1.23 ms, each against one tile per SM with next-tile prefetch into shared memory.

#include <algorithm>
#include <cstring>

#include "fused.h"
#include "fused_bwd_common.cuh"
#include "profiler.h"

namespace gnn {
namespace fused {

cudaError_t take_device_error_edge_bwd(unsigned int* out) { return take_device_error_word(out); }

namespace {

using namespace host;

// NG tile groups of 128 rows x CG column groups of CW columns.
template <int H, int NG_, int CW_>
struct EbCfg {
    static constexpr int NG = NG_, CW = CW_, CG = H / CW, GT = 128 * CG, NT = NG * GT;
    static constexpr int S = span_of(H), TILE = 128 * H * 2, WT = H * H * 2;
    static constexpr int NS = CW / 16;                       // 16-column pieces per thread
    static constexpr int RED = CG == 1 ? 0 : (CG + NS - 1);  // 16-byte row-statistics chunks per row
};

struct EbSmem {
    uint32_t grp, gstride, e, de, hb, ones, w, rec, par, red, bar, tm, total;
};

// A group's tiles: e, de_out (then dz_{L-1}, then de_in), h_0 .. h_{L-2} (then
// dz_0 .. dz_{L-2}); behind h_0 also the FP32 staging of dz_0 for dP. The
// M = 128 views of a dz tile (H < 128 columns) read 32 KB from its start: past
// the last group that is the ones block, the weights and the rest.
template <class C, int H>
__host__ __device__ inline EbSmem eb_smem(int n_lin) {
    EbSmem s;
    s.grp = 0;
    s.e = 0;
    s.de = C::TILE;
    s.hb = 2 * C::TILE;
    const uint32_t a = (uint32_t)(n_lin - 1) * C::TILE, b = C::TILE + 128 * H * 4;
    s.gstride = align_up(s.hb + (a > b ? a : b), 1024);
    s.ones = C::NG * s.gstride;
    s.w = s.ones + 128 * C::S;
    s.rec = align_up(s.w + n_lin * C::WT, 128);
    s.par = s.rec + C::NG * GNN_TILE_META_BYTES;
    s.red = align_up(s.par + (n_lin + 2) * H * 4, 16);
    const uint32_t red = (uint32_t)C::NG * C::RED * 128 * 16, end_red = 2 * C::NG * 4 * H * 4;
    s.bar = s.red + (red > end_red ? red : end_red);   // (the final column sums also go through red)
    s.tm = s.bar + 8 * C::NG * (4 + 2 * GNN_MAX_LIN);
    const uint32_t end = s.tm + 16, view = s.ones - C::TILE + 32768;
    s.total = (end > view ? end : view) + 1024;
    return s;
}

template <class C, int H>
__host__ __device__ inline uint32_t eb_cols(int n_lin) { return C::NG * H + n_lin * (H + 16); }

struct EbArgs {
    const uint8_t* tile_meta;   // per-tile records (GNN_TILE_META_BYTES each)
    int64_t n_tiles;
    const __nv_bfloat16* pq;    // P rows [n_rows x H]
    const __nv_bfloat16* q;     // Q rows [n_rows x H]
    const float* da;            // gradient of the aggregate after the halo adjoint
    const __nv_bfloat16* e_in;
    const __nv_bfloat16* de_out;   // or NULL
    const __nv_bfloat16* act;      // SAVED
    __nv_bfloat16* de_in;
    __nv_bfloat16* dz1;         // per-edge gradient of the first pre-activation
    float* dP;                  // per-row sum of dz_0 over the row's received edges
    float* part;
    int64_t pstride;
    MlpDev mlp;
    float eps;
    int64_t act_rows;           // SAVED: rows of one activation block of tmap_h (tiles * 128)
};

// SAVED: the forward stored the hidden activations h_0 .. h_{L-2} of every edge
// (row k * act_rows + t * 128 + i of tmap_h for edge row i of tile t); they
// arrive by TMA and only the last Linear is recomputed.
template <int H, int NG, int CW, bool SAVED>
__global__ void __launch_bounds__(EbCfg<H, NG, CW>::NT, 1) k_edge_bwd(const __grid_constant__ CUtensorMap tmap_e,
                                                                     const __grid_constant__ CUtensorMap tmap_de,
                                                                     const __grid_constant__ CUtensorMap tmap_h,
                                                                     const __grid_constant__ EbArgs A) {
    using C = EbCfg<H, NG, CW>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = aligned_smem(smem_raw);
    const int L = A.mlp.n_lin;
    const EbSmem P = eb_smem<C, H>(L);
    constexpr int S = C::S, CG = C::CG, GT = C::GT, NT = C::NT, TILE = C::TILE, WT = C::WT, NS = C::NS, RED = C::RED;
    const int tid = threadIdx.x, lane = tid & 31, gi = tid / GT, gt = tid - gi * GT;
    const int gw = gt >> 5, q = gw & 3, g = gw >> 2, row = 32 * q + lane, c0 = g * CW;
    const bool leader = gt == 0;

    uint8_t* sE = sm + P.grp + gi * P.gstride + P.e;
    uint8_t* sDE = sm + P.grp + gi * P.gstride + P.de;
    uint8_t* sHB = sm + P.grp + gi * P.gstride + P.hb;
    uint8_t* sOnes = sm + P.ones;
    uint8_t* sW = sm + P.w;
    uint8_t* rec = sm + P.rec + gi * GNN_TILE_META_BYTES;
    float* sStage = reinterpret_cast<float*>(sHB + TILE);   // FP32 dz_0 rows
    float* sPar = reinterpret_cast<float*>(sm + P.par);
    float4* sRed = reinterpret_cast<float4*>(sm + P.red) + gi * RED * 128;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + P.bar);
    constexpr int NB = 4 + 2 * GNN_MAX_LIN;                        // barriers of a group
    uint64_t* full = bars + gi * NB;                               // record, e and de_out rows
    uint64_t* bar = full + 1;                                      // chain and input-gradient MMAs
    uint64_t* bar_w = full + 2;                                    // weight-gradient MMAs
    uint64_t* ready = full + 3;                                    // one arrival per warp before an MMA
    uint64_t* h_full = full + 4;                                   // SAVED: h_k has landed
    uint64_t* turn = full + 4 + GNN_MAX_LIN;                       // [L]: this group may issue its next dW_k
    uint64_t* turn_next = bars + (gi + 1) % NG * NB + 4 + GNN_MAX_LIN;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + P.tm);
    const uint32_t NCOLS = pow2_cols(eb_cols<C, H>(L));

    if (tid < 32) {
        tmem_alloc(tslot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < NG; ++i) {
            uint64_t* b = bars + i * NB;
            mbar_init(b, 1);
            mbar_init(b + 1, 1);
            mbar_init(b + 2, 1);
            mbar_init(b + 3, GT / 32);
            for (int k = 0; k < L - 1; ++k) mbar_init(b + 4 + k, 1);
            for (int k = 0; k < L; ++k) mbar_init(b + 4 + GNN_MAX_LIN + k, 1);
        }
        fence_mbar_init();
    }
    load_weight(sW, A.mlp.W[0], 3 * H, 2 * H, H, H, tid, NT);
    for (int k = 1; k < L; ++k) load_weight(sW + k * WT, A.mlp.W[k], H, 0, H, H, tid, NT);
    fill_ones(sOnes, S, tid, NT);
    for (int i = tid; i < L * H; i += NT) sPar[i] = A.mlp.b[i / H][i % H];
    for (int i = tid; i < H; i += NT) {
        sPar[L * H + i] = A.mlp.gamma[i];
        sPar[(L + 1) * H + i] = A.mlp.beta[i];
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t tWork = tmem + (uint32_t)(gi * H);
    auto tDW = [&](int k) -> uint32_t { return tmem + (uint32_t)(NG * H + k * (H + 16)); };
    const uint32_t ones_addr = smem_u32(sOnes);
    // LayerNorm gradient sums sum_rows g * xhat and sum_rows g, per warp (warp_colsum16)
    float acc_g[NS], acc_b[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) acc_g[i] = acc_b[i] = 0.f;
    uint32_t ph = 0, ph_rdy = 0, ph_w = 0, ph_full = 0;
    bool ok = true;
    int64_t j = gi;   // this tile's place in the CTA's sequence

    // MMA hand-off without group barriers: every warp arrives on `ready` once its operand writes and its
    // reads of the accumulator are done; the leader waits for all warps and issues; every thread waits for
    // the completion by itself. After a timeout a thread stops waiting and issuing, and the group leaves
    // the tile loop together at the tile's end.
    auto handoff = [&](auto&& issue) {
        fence_proxy_async();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(ready);
        if (leader) {
            ok = ok && mbar_wait(ready, ph_rdy);
            ph_rdy ^= 1;
            tc_fence_after();
            if (ok) issue();
        }
    };
    auto mma_wait = [&]() {
        ok = ok && mbar_wait(bar, ph);
        ph ^= 1;
        __syncwarp();
        tc_fence_after();
    };
    // leader: dW_k += dz^T [h | ones] in its turn
    auto issue_dw = [&](int k, const uint8_t* dz, const uint8_t* hk) {
        if (j > 0) {   // turns so far: one per round, none before the first tile
            ok = ok && mbar_wait(turn + k, (uint32_t)(j / NG - (gi == 0 ? 1 : 0)) & 1u);
            tc_fence_after();
        }
        if (!ok) return;
        issue_wgrad(tDW(k), dz, S, 128u * S, hk, S, ones_addr - smem_u32(hk), H + 16, j > 0);
        mma_commit(bar_w);
        tc_fence_before();
        mbar_arrive(turn_next + k);
    };
    auto header = [&](int64_t t) { return ld_nc_v4s32(A.tile_meta + t * GNN_TILE_META_BYTES); };   // {r0, r1, e0, ne}
    // leader: the record, e, de_out (and saved h_k) rows of tile t
    bool pending = false;
    auto load_tile = [&](int64_t t, int32_t e0) {
        mbar_arrive_expect_tx(full, TILE * (A.de_out ? 2 : 1) + GNN_TILE_META_BYTES);
        bulk_load(rec, A.tile_meta + t * GNN_TILE_META_BYTES, GNN_TILE_META_BYTES, full);
        tma_load_2d(sE, &tmap_e, 0, e0, full);
        if (A.de_out) tma_load_2d(sDE, &tmap_de, 0, e0, full);
        if (SAVED)
            for (int k = L - 2; k >= 0; --k) {
                mbar_arrive_expect_tx(h_full + k, TILE);
                tma_load_2d(sHB + k * TILE, &tmap_h, 0, (int32_t)(k * A.act_rows + t * 128), h_full + k);
            }
        pending = true;
    };
    // leader: what the next tile reads, into L2 (its loads start when this tile's buffers are free)
    auto prefetch_tile = [&](int64_t t, int4 h) {
        const int32_t nr = min(max(h.y - h.x, 0), 128), ne = min(max(h.w, 0), 128);
        if (nr == 0 || ne == 0) return;
        prefetch_l2(A.tile_meta + t * GNN_TILE_META_BYTES, GNN_TILE_META_BYTES);
        prefetch_l2(A.e_in + (int64_t)h.z * H, (uint32_t)ne * H * 2);
        if (A.de_out) prefetch_l2(A.de_out + (int64_t)h.z * H, (uint32_t)ne * H * 2);
        prefetch_l2(A.da + (int64_t)h.x * H, (uint32_t)nr * H * 4);
        if (SAVED) {
            for (int k = 0; k < L - 1; ++k) prefetch_l2(A.act + ((int64_t)k * A.act_rows + t * 128) * H, TILE);
        } else {
            prefetch_l2(A.pq + (int64_t)h.x * H, (uint32_t)nr * H * 2);
        }
    };
    const int64_t stride = (int64_t)gridDim.x * NG;
    int64_t t = (int64_t)blockIdx.x + gi * (int64_t)gridDim.x;
    int4 hdr_next = make_int4(0, 0, 0, 0);
    if (leader && t < A.n_tiles) {
        load_tile(t, header(t).z);
        if (t + stride < A.n_tiles) hdr_next = header(t + stride);
    }

    for (; t < A.n_tiles; t += stride, j += NG) {
        ok = ok && mbar_wait(full, ph_full);
        __syncwarp();
        const int32_t* hdr = reinterpret_cast<const int32_t*>(rec);
        const int32_t* sRp = reinterpret_cast<const int32_t*>(rec + 16);
        const int16_t* sSeg = reinterpret_cast<const int16_t*>(rec + 544);
        const int32_t* sSnd = reinterpret_cast<const int32_t*>(rec + 800);
        const float* sW1d = reinterpret_cast<const float*>(rec + 1312);
        const int32_t r0 = hdr[0], r1 = hdr[1], e0 = hdr[2], ne = ok ? hdr[3] : 0;
        const bool valid = row < ne;
        const bool more = t + stride < A.n_tiles;
        if (leader && ok) {
            if (SAVED) ok = mbar_wait(h_full + L - 2, ph_full);
            tc_fence_after();
            if (ok) {
                if (SAVED) issue_mma(tWork, sHB + (L - 2) * TILE, sW + (L - 1) * WT, H, H);
                else issue_mma(tWork, sE, sW, H, H);
                mma_commit(bar);
            }
            if (more) prefetch_tile(t + stride, hdr_next);
        }
        const int64_t rcv = valid ? (int64_t)r0 + sSeg[row] : 0;
        // ---- recompute the chain (SAVED: only the last Linear, from the saved h_{L-2})
        if constexpr (!SAVED) {
            // the receiver's P and the sender's Q columns, requested while the first Linear runs
            uint4 up[CW / 8], uq[CW / 8];
            if (valid) {
                const uint4* pp = reinterpret_cast<const uint4*>(A.pq + rcv * H + c0);
                const uint4* pqp = reinterpret_cast<const uint4*>(A.q + (int64_t)sSnd[row] * H + c0);
#pragma unroll
                for (int i = 0; i < CW / 8; ++i) {
                    up[i] = __ldg(pp + i);
                    uq[i] = __ldg(pqp + i);
                }
            }
            mma_wait();
#pragma unroll
            for (int h = 0; h < CW; h += 16) {
                float v[16];
                tmem_ld16(tWork + ((uint32_t)(32 * q) << 16) + (uint32_t)(c0 + h), v);
                tmem_ld_wait();
                if (valid) {
#pragma unroll
                    for (int kc = 0; kc < 2; ++kc) {
                        const uint4 a = up[h / 8 + kc], b = uq[h / 8 + kc];
                        const uint32_t pw[4] = {a.x, a.y, a.z, a.w}, qw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float p0, p1, q0, q1;
                            unpack_bf16x2(pw[i], p0, p1);
                            unpack_bf16x2(qw[i], q0, q1);
                            const float2 t2 = __fadd2_rn(__fadd2_rn(make_float2(p0, p1), make_float2(q0, q1)),
                                                         *reinterpret_cast<const float2*>(sPar + c0 + h + 8 * kc + 2 * i));
                            float2* vv = reinterpret_cast<float2*>(v + 8 * kc + 2 * i);
                            *vv = __fadd2_rn(*vv, t2);
                        }
                    }
                } else {
                    add_bias2<16>(v, sPar + c0 + h);
                }
                elu_inplace2<16>(v);
                st_row_tile<16>(sHB, row, c0 + h, S, v);
            }
            handoff([&] {
                issue_mma(tWork, sHB, sW + WT, H, H);
                mma_commit(bar);
            });
            for (int k = 1; k < L - 1; ++k) {
                mma_wait();
#pragma unroll
                for (int h = 0; h < CW; h += 16) {
                    float v[16];
                    tmem_ld16(tWork + ((uint32_t)(32 * q) << 16) + (uint32_t)(c0 + h), v);
                    tmem_ld_wait();
                    add_bias2<16>(v, sPar + k * H + c0 + h);
                    elu_inplace2<16>(v);
                    st_row_tile<16>(sHB + k * TILE, row, c0 + h, S, v);
                }
                handoff([&] {
                    issue_mma(tWork, sHB + k * TILE, sW + (k + 1) * WT, H, H);
                    mma_commit(bar);
                });
            }
        }
        // ---- gradient of e' (adjoint of Eq. 5b plus the upstream edge gradient), while the last Linear runs
        float gv[CW];
        if (valid) {
            const float* src = A.da + rcv * H + c0;
            float dar[CW];
#pragma unroll
            for (int i = 0; i < CW / 4; ++i) {
                const float4 u = __ldg(reinterpret_cast<const float4*>(src) + i);
                dar[4 * i] = u.x; dar[4 * i + 1] = u.y; dar[4 * i + 2] = u.z; dar[4 * i + 3] = u.w;
            }
            const float w = sW1d[row];
            if (A.de_out) {
                float deo[CW];
                ld_row_tile<CW>(sDE, row, c0, S, deo);
#pragma unroll
                for (int i = 0; i < CW; ++i) gv[i] = __fmaf_rn(w, dar[i], deo[i]);
            } else {
#pragma unroll
                for (int i = 0; i < CW; ++i) gv[i] = w * dar[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < CW; ++i) gv[i] = 0.f;
        }
        // ---- LayerNorm adjoint: statistics and adjoint sums per 16 columns, combined in column order
        // (roundings written out: a different contraction flips BF16 roundings downstream)
        mma_wait();
        {
            float4 st[NS];   // {sum v, sum v^2, sum d, sum d v}, d = g gamma
            float v[CW];
            ld_acc<CW>(tWork, q, c0, v);
            add_bias2<CW>(v, sPar + (L - 1) * H + c0);
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                float sv = 0.f, sq = 0.f, sd = 0.f, sdv = 0.f;
#pragma unroll
                for (int i = 16 * p; i < 16 * p + 16; ++i) {
                    const float d = __fmul_rn(gv[i], sPar[L * H + c0 + i]);
                    sv = __fadd_rn(sv, v[i]);
                    sq = __fmaf_rn(v[i], v[i], sq);
                    sd = __fadd_rn(sd, d);
                    sdv = __fmaf_rn(d, v[i], sdv);
                }
                st[p] = make_float4(sv, sq, sd, sdv);
            }
            auto acc4 = [](float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); };
            float4 tot = st[0];
            if constexpr (CG == 1) {
#pragma unroll
                for (int p = 1; p < NS; ++p) tot = acc4(tot, st[p]);
            } else if constexpr (NS == 1) {   // CG threads per row, one piece each
                sRed[g * 128 + row] = st[0];
                named_sync(1 + gi, GT);
                tot = sRed[row];
#pragma unroll
                for (int p = 1; p < CG; ++p) tot = acc4(tot, sRed[p * 128 + row]);
            } else {                          // two threads, two pieces each: (p0 + p1) | p2 | p3
                static_assert(CG == 2 && NS == 2, "two threads of two pieces");
                if (g == 0) {
                    sRed[row] = acc4(st[0], st[1]);
                } else {
                    sRed[128 + row] = st[0];
                    sRed[256 + row] = st[1];
                }
                named_sync(1 + gi, GT);
                tot = acc4(acc4(sRed[row], sRed[128 + row]), sRed[256 + row]);
            }
            const float mean = tot.x * (1.f / H);
            const float rstd = rsqrtf(fmaxf(__fmaf_rn(tot.y, 1.f / H, -__fmul_rn(mean, mean)), 0.f) + A.eps);
            const float s1 = tot.z * (1.f / H);
            const float s2 = __fmul_rn(__fmul_rn(rstd, __fmaf_rn(-mean, tot.z, tot.w)), 1.f / H);
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                float t16[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    float& x = v[16 * p + i];
                    x = (x - mean) * rstd;   // xhat
                    t16[i] = gv[16 * p + i] * x;
                }
                acc_g[p] += warp_colsum16(t16, lane);
                acc_b[p] += warp_colsum16(gv + 16 * p, lane);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float d = __fmul_rn(gv[16 * p + i], sPar[L * H + c0 + 16 * p + i]);
                    t16[i] = __fmul_rn(rstd, __fmaf_rn(-v[16 * p + i], s2, __fsub_rn(d, s1)));
                }
                st_row_tile<16>(sDE, row, c0 + 16 * p, S, t16);   // dz_{L-1} over the thread's own de_out columns
            }
        }
        // ---- chain adjoint: step k has dz_k in its tile
        for (int k = L - 1; k >= 1; --k) {
            uint8_t* dzk = k == L - 1 ? sDE : sHB + k * TILE;
            uint8_t* hk = sHB + (k - 1) * TILE;
            if (SAVED) ok = ok && mbar_wait(h_full + k - 1, ph_full);   // the weight gradient's operand, and ELU'
            handoff([&] {
                issue_dgrad(tWork, dzk, S, sW + k * WT, S, H, (uint32_t)H * S, H, H);
                mma_commit(bar);
                issue_dw(k, dzk, hk);
            });
            mma_wait();
            // dz_{k-1} = dh ELU'(h_{k-1}), written over h_{k-1} once dW_k has read it
            uint32_t dzb[CW / 2];
            float4* stage4 = reinterpret_cast<float4*>(sStage);
            constexpr int NC = H / 4;
            bool waited = false;
#pragma unroll
            for (int h = 0; h < CW; h += 16) {
                float dh[16], hv[16], dz[16];
                tmem_ld16(tWork + ((uint32_t)(32 * q) << 16) + (uint32_t)(c0 + h), dh);
                ld_row_tile<16>(hk, row, c0 + h, S, hv);
                tmem_ld_wait();
                elu_bwd2<16>(dz, dh, hv);
#pragma unroll
                for (int i = 0; i < 8; ++i) dzb[h / 2 + i] = pack_bf16x2(dz[2 * i], dz[2 * i + 1]);
                if (k == 1) {   // FP32 rows for dP: over h_1 .. (their gradients' MMAs are done: dW_1 is the last)
                    if (!waited) {
                        ok = ok && mbar_wait(bar_w, ph_w);
                        __syncwarp();
                        waited = true;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        stage4[row * NC + stage_chunk<NC>((c0 + h) / 4 + i, row)] =
                            make_float4(dz[4 * i], dz[4 * i + 1], dz[4 * i + 2], dz[4 * i + 3]);
                }
            }
            if (!waited) ok = ok && mbar_wait(bar_w, ph_w);
            ph_w ^= 1;
#pragma unroll
            for (int i = 0; i < CW / 8; ++i)
                *reinterpret_cast<uint4*>(hk + tile_off(row, c0 + 8 * i, 128, S)) =
                    make_uint4(dzb[4 * i], dzb[4 * i + 1], dzb[4 * i + 2], dzb[4 * i + 3]);
        }
        // ---- first Linear: W1c^T dz_0 and dW1c; dz_0 per edge and its receiver sums
        handoff([&] {
            issue_dgrad(tWork, sHB, S, sW, S, H, (uint32_t)H * S, H, H);
            mma_commit(bar);
            issue_dw(0, sHB, sE);
        });
        named_sync(1 + gi, GT);   // every dz_0 row is staged
        {
            constexpr int CPR = H / 8;   // 16-byte chunks per row
            for (int i = gt; i < ne * CPR; i += GT) {
                const int r = i / CPR, jj = i - r * CPR;
                *reinterpret_cast<uint4*>(A.dz1 + ((int64_t)e0 + r) * H + 8 * jj) =
                    *reinterpret_cast<const uint4*>(sHB + tile_off(r, 8 * jj, 128, S));
            }
            constexpr int NC = H / 4;
            const float4* stage4 = reinterpret_cast<const float4*>(sStage);
            const int nr = ok ? r1 - r0 : 0;
            for (int it = gt; it < nr * NC; it += GT) {
                const int rr = it / NC, c = it % NC;
                const int32_t b0 = sRp[rr], b1 = sRp[rr + 1];
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int32_t e = b0; e < b1; ++e) {
                    const float4 u4 = stage4[e * NC + stage_chunk<NC>(c, e)];
                    acc.x += u4.x;
                    acc.y += u4.y;
                    acc.z += u4.z;
                    acc.w += u4.w;
                }
                *reinterpret_cast<float4*>(A.dP + (int64_t)(r0 + rr) * H + 4 * c) = acc;
            }
        }
        mma_wait();
#pragma unroll
        for (int h = 0; h < CW; h += 16) {
            float o[16];
            tmem_ld16(tWork + ((uint32_t)(32 * q) << 16) + (uint32_t)(c0 + h), o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = gv[h + i] + o[i];   // residual + W1c^T dz_0
            st_row_tile<16>(sDE, row, c0 + h, S, o);                // (dz_{L-1}'s MMAs are done)
        }
        tc_fence_before();
        named_sync(1 + gi, GT);   // every row of de_in is in the tile
        {
            constexpr int CPR = H / 8;
            for (int i = gt; i < ne * CPR; i += GT) {
                const int r = i / CPR, jj = i - r * CPR;
                *reinterpret_cast<uint4*>(A.de_in + ((int64_t)e0 + r) * H + 8 * jj) =
                    *reinterpret_cast<const uint4*>(sDE + tile_off(r, 8 * jj, 128, S));
            }
        }
        ok = ok && mbar_wait(bar_w, ph_w);   // dW_0 has read e and dz_0
        ph_w ^= 1;
        ph_full ^= 1;
        fence_proxy_async();
        const bool all = named_and(ok, 1 + gi, GT);   // the tile's buffers are free; the group leaves together
        tc_fence_after();
        if (leader) pending = false;
        if (!all) break;
        if (leader && more) {
            load_tile(t + stride, hdr_next.z);
            if (t + 2 * stride < A.n_tiles) hdr_next = header(t + 2 * stride);
        }
    }
    if (leader && pending) {   // loads issued before a timeout ended the tile loop
        mbar_wait(full, ph_full);
        if (SAVED)
            for (int k = 0; k < L - 1; ++k) mbar_wait(h_full + k, ph_full);
    }
    __syncwarp();
    tc_fence_before();
    ok = __syncthreads_and(ok) != 0;
    tc_fence_after();
    // ---- flush the CTA's partial gradients: per layer [H x (H + 16)], then gamma, beta
    float* part = A.part + (int64_t)blockIdx.x * A.pstride;
    const int wq = (tid >> 5) & 3, wg = tid >> 7;
    if (ok)
        for (int k = 0; k < L; ++k)
            flush_acc<NT / 128>(tDW(k), H + 16, H, wq, lane, wg, part + (int64_t)k * H * (H + 16));
    {   // column sums of the groups' warps, in group and quarter order
        float* red = reinterpret_cast<float*>(sm + P.red);
        if ((lane & 1) == 0) {
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                red[(gi * 4 + q) * H + c0 + 16 * p + (lane >> 1)] = acc_g[p];
                red[(NG * 4 + gi * 4 + q) * H + c0 + 16 * p + (lane >> 1)] = acc_b[p];
            }
        }
        __syncthreads();
        for (int i = tid; i < 2 * H; i += NT) {
            const int c = i % H, b = i / H;
            float s = 0.f;
            for (int k = 0; k < NG * 4; ++k) s += red[(b * NG * 4 + k) * H + c];
            part[(int64_t)L * H * (H + 16) + i] = s;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid < 32) tmem_dealloc(tmem, NCOLS);
}

template <int H, int NG, int CW>
int launch(const gnn_graph_dev& G, const EbArgs& A, const CUtensorMap& tm_e, const CUtensorMap& tm_de,
           const CUtensorMap& tm_h, int* grid, cudaStream_t s) {
    using C = EbCfg<H, NG, CW>;
    const uint32_t smem = eb_smem<C, H>(A.mlp.n_lin).total, cols = pow2_cols(eb_cols<C, H>(A.mlp.n_lin));
    auto run = [&](auto kern) -> int {
        int rc = persistent_grid(kern, C::NT, smem, cols, G.n_edge_tiles, grid, 1);
        if (rc) return rc;
        {
            ProfScope _ps(s, "k_edge_bwd");
            kern<<<*grid, C::NT, smem, s>>>(tm_e, tm_de, tm_h, A);
        }
        GNN_LAUNCH_CHECK("k_edge_bwd");
        return GNN_OK;
    };
    return A.act ? run(k_edge_bwd<H, NG, CW, true>) : run(k_edge_bwd<H, NG, CW, false>);
}

template <int H, int NG, int CW>
bool fits(int n_lin) {
    using C = EbCfg<H, NG, CW>;
    return eb_cols<C, H>(n_lin) <= 512 && eb_smem<C, H>(n_lin).total <= 227 * 1024;
}

}  // namespace

bool edge_backward_supported(int H, int n_lin) {
    if (H == 64) return fits<64, 2, 32>(n_lin);
    if (H == 32) return fits<32, 2, 16>(n_lin);
    return H == 16 && fits<16, 4, 16>(n_lin);
}

int edge_backward(const gnn_graph_dev& G, int H, const gnn_mp_params& W, const EdgeBackward& o, int* grid,
                  cudaStream_t s) {
    const int64_t NR = G.n_rows, E = G.n_edges;
    const int L = W.edge.n_lin;
    GNN_REQUIRE(G.tile_meta && ((uintptr_t)G.tile_meta & 15) == 0, GNN_EINVAL,
                "gnn_mp_backward: tile_meta must be a 16-byte aligned device array");
    GNN_REQUIRE(edge_backward_supported(H, L), GNN_EUNSUPPORTED, "fused edge adjoint does not fit on an SM");
    CUtensorMap tm_e, tm_de, tm_h;
    int rc;
    if ((rc = make_row_tmap(&tm_e, o.e_in, E, H))) return rc;
    if ((rc = make_row_tmap(&tm_de, o.de_out ? o.de_out : o.e_in, E, H))) return rc;
    tm_h = tm_e;
    if (o.act && (rc = make_row_tmap(&tm_h, o.act, (int64_t)(L - 1) * G.n_edge_tiles * 128, H))) return rc;
    EbArgs A{};
    A.tile_meta = (const uint8_t*)G.tile_meta;
    A.n_tiles = G.n_edge_tiles;
    A.pq = o.pq;
    A.q = o.pq + NR * H;
    A.da = o.da;
    A.e_in = o.e_in;
    A.de_out = o.de_out;
    A.act = o.act;
    A.de_in = o.de_in;
    A.dz1 = o.dz1;
    A.dP = o.dP;
    A.part = o.part;
    A.pstride = o.pstride;
    A.mlp = mlp_dev(W.edge);
    A.eps = o.eps;
    A.act_rows = G.n_edge_tiles * 128;
    // H = 32: four groups of one thread per row while their tiles fit (up to 5 Linears), else two of two
    // threads per row
    if (H == 64) return launch<64, 2, 32>(G, A, tm_e, tm_de, tm_h, grid, s);
    if (H == 32)
        return fits<32, 4, 32>(L) ? launch<32, 4, 32>(G, A, tm_e, tm_de, tm_h, grid, s)
                                  : launch<32, 2, 16>(G, A, tm_e, tm_de, tm_h, grid, s);
    return launch<16, 4, 16>(G, A, tm_e, tm_de, tm_h, grid, s);
}

}  // namespace fused
}  // namespace gnn
