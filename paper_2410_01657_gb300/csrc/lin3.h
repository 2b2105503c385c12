// FP32 Linear layers on the tensor cores (lin3.cu): every FP32 operand is an
// exact sum of three BF16 values, products and sums are FP32.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gnn {
namespace lin3 {

constexpr int kMaxWidth = 128;   // widest N and K of one launch (per source)
constexpr int kMaxCtas = 160;    // most CTAs of a launch
constexpr int kMaxReduce = 24;   // most sums of one reduce launch

// What happens to a row tile's products acc = sum_s A_s W_s^T on their way out.
enum Mode {
    kElu = 0,     // out = ELU(acc + bias + (P[recv] + Q[snd] or add))
    kLayerNorm,   // out = res + gamma * xhat(acc + bias) + beta            (add = res, may be NULL)
    kLnAdjoint,   // out = dL/d(acc + bias) of the LayerNorm for the upstream g = g0, or g0 + w * da[recv]
    kEluAdjoint,  // out = acc * ELU'(z), add = h = ELU(z)
    kAdd          // out = acc + bias + (add, or with da: g0 + w * da[recv])
};

struct Args {
    int64_t rows;
    const float* A[2];         // sources [rows x K[s]], row stride lda[s]
    int64_t lda[2];
    int K[2];                  // K[1] = 0: one source
    const float* W[2];         // source s: W[s][n * sn + k * sk] (+ noff for n >= nsplit, n counted from nsplit)
    int64_t sn, sk;
    int nsplit;
    int64_t noff;
    int N;
    const float* bias;         // [N] or NULL
    float* out;                // row stride ldo
    int64_t ldo;
    const float* add;          // row stride ldadd
    int64_t ldadd;
    const float* P;            // row stride ldpq
    const float* Q;
    int64_t ldpq;
    const int32_t* recv;       // receiver / sender row of every row of the tile (edges)
    const int32_t* snd;
    const float* g0;           // [rows x N] or NULL (zero)
    const float* da;           // [receivers x N] or NULL
    const float* w;            // [rows]
    const float* gamma;
    const float* beta;
    float eps;
    float* part;               // kLnAdjoint: per-CTA column sums of g * xhat, then of g ([2N])
    // set by run()
    int n_tiles, NP, KB, nkb[2], stages;
};

// One Linear over all rows; *ctas receives the number of CTAs (partials).
int run(Mode mode, Args a, cudaStream_t s, int* ctas = nullptr);
// True when the weights of `sources` sources of width K and N outputs fit one launch.
bool fits(int N, int K, int sources);

// Per-CTA partials of dW[n][k] = sum_r G[r][n] X[r][k] ([N x K]) and, when db,
// of sum_r G[r][n] ([N] behind it) into part; *ctas receives their number.
int wgrad(int64_t rows, const float* G, int64_t ldg, int N, const float* X, int64_t ldx, int K, bool db, float* part,
          cudaStream_t s, int* ctas);
// Most CTAs of a launch over `rows` rows (a row tile has 64 or 128): sizes the per-CTA partial sums.
inline int64_t max_ctas(int64_t rows) { return rows + 63 < (int64_t)kMaxCtas * 64 ? (rows + 63) / 64 : kMaxCtas; }
inline int64_t wgrad_floats(int64_t rows, int N, int K) { return max_ctas(rows) * (N * K + N); }

// out [rows x K] = (G W) ELU'(H) and the partials of wgrad(G, H) in one pass
// (G [rows x N], H = ELU outputs [rows x K], W [N x K], all dense).
bool chain_fits(int N, int K);
int chain(int64_t rows, const float* G, int N, const float* H, int K, const float* W, float* out, bool db, float* part,
          cudaStream_t s, int* ctas);

// dst[n * ldd + k] += sum over z of part[z * stride + n * K + k], z ascending per lane. One launch, and another
// wherever a destination may overlap an earlier one.
struct Sum {
    const float* part;
    int64_t stride;
    int nz, N, K;
    float* dst;
    int64_t ldd;
};
int reduce(const Sum* sums, int n, cudaStream_t s);

cudaError_t take_device_error(unsigned int* out);

}  // namespace lin3
}  // namespace gnn
