// pp_mlp.cu -- the surrogate network of the screened DE: a multilayer
// perceptron d_in -> H -> H -> H -> 1 with GELU activations that predicts the
// (normalised) log10 of the pair number from normalised pulse parameters.
// The three hidden layers run on the tensor cores (pp_gemm.cu: BF16 operands,
// FP32 accumulation); biases, activations, the output unit, the loss and Adam
// run on the CUDA cores in FP32.  Not part of the paper.
//
// Parameters (one flat FP32 vector, this order):
//   W1 [H][d_in], b1 [H], W2 [H][H], b2 [H], W3 [H][H], b3 [H], w4 [H], b4 [1].
// Forward, for a batch X [B][d_in] (B padded to a multiple of 128 with zero rows):
//   Z1 = X W1^T + b1, A1 = gelu(Z1), Z2 = A1 W2^T + b2, A2 = gelu(Z2),
//   Z3 = A2 W3^T + b3, A3 = gelu(Z3), y = A3 w4 + b4,
// gelu(z) = z Phi(z) = z (1 + erf(z / sqrt 2)) / 2.  Loss: mean over the valid
// rows of (y - t)^2.  Backward: dy = 2 (y - t) / B_valid; dW = dZ^T A, db = sum
// of dZ over rows, dA = dZ W, dZ = dA gelu'(Z), gelu'(z) = Phi(z) + z phi(z).
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "pp_internal.cuh"

namespace {

constexpr int kRows = 128;  // batch rows are padded to this

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad(float z)
{
    const float Phi = 0.5f * (1.0f + erff(z * 0.70710678118654752f));
    const float phi = 0.39894228040143268f * expf(-0.5f * z * z);
    return Phi + z * phi;
}

// Packed BF16 offset of element (r, c) in a matrix with cols_pad columns (see pp_gemm.cu).
__device__ __forceinline__ size_t packed_off(int r, int c, int cols_pad)
{
    return ((size_t)(r / 128) * (cols_pad / 64) + c / 64) * 8192 + ((r % 128) / 8) * 512 + ((c % 64) / 8) * 64 +
           (r % 8) * 8 + (c % 8);
}

// The passes between the products work on 32 x 32 tiles: a CTA reads a tile once, a row per warp,
// and from shared memory writes it both packed and packed transposed (a product wants its operands
// along the index that is summed, and the weight gradients sum over rows), and sums its columns.
// Packed, eight elements of a row are 16 bytes and eight such rows 128 bytes, so every store is a
// full line.  At 256 rows these passes and the products are launches of 3 to 8 us that hardly fill
// the chip: what counts is their number, and that no thread walks down all rows.  Loss and gradient
// of 256 rows, 32 -> 256 -> 256 -> 256 -> 1: 209 us in 34 launches, of which 79 us of column sums by
// one thread per column -> 119 us in 19 launches.  (256 threads of 4 elements: the same.)
constexpr int kSide = 32;
constexpr int kTileThreads = kSide * kSide;
using Tile = float[kSide][kSide + 1];

// Rows r0 .., columns c0 .. of a matrix: P packed with cols_pad columns, PT its transpose packed
// with rows_pad columns; either may be NULL.  Warps 0 .. 3 write the one, 4 .. 7 the other.
__device__ __forceinline__ void store_packed(const Tile &s, int r0, int c0, int rows_pad, int cols_pad, uint16_t *P,
                                             uint16_t *PT)
{
    constexpr int kRuns = kSide * kSide / 8;
    const bool trans = threadIdx.x >= kRuns;
    uint16_t *out = trans ? PT : P;
    if (!out || threadIdx.x >= 2 * kRuns)
        return;
    const int i = threadIdx.x % kRuns, line = i / 4, run = i % 4 * 8;
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float a = trans ? s[run + 2 * j][line] : s[line][run + 2 * j];
        const float b = trans ? s[run + 2 * j + 1][line] : s[line][run + 2 * j + 1];
        w[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
               (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16;
    }
    const size_t at = trans ? packed_off(c0 + line, r0 + run, rows_pad) : packed_off(r0 + line, c0 + run, cols_pad);
    *(uint4 *)(out + at) = make_uint4(w[0], w[1], w[2], w[3]);
}

// X (B x C) -> packed, and packed transposed.
__global__ void __launch_bounds__(kTileThreads)
    pack_input_kernel(const float *__restrict__ X, int B, int C, uint16_t *__restrict__ P, uint16_t *__restrict__ PT)
{
    __shared__ Tile s;
    const int r0 = blockIdx.y * kSide, c0 = blockIdx.x * kSide, r = threadIdx.x / kSide, c = threadIdx.x % kSide;
    s[r][c] = X[(size_t)(r0 + r) * C + c0 + c];
    __syncthreads();
    store_packed(s, r0, c0, B, C, P, PT);
}

// Z (B x H) += bias; Ap = packed gelu(Z).  Rows >= nvalid are zeroed.  For a gradient (AT not
// NULL) Z is kept and gelu(Z) is packed transposed too.
__global__ void __launch_bounds__(kTileThreads)
    bias_gelu_pack_kernel(float *__restrict__ Z, const float *__restrict__ bias, int B, int H, int nvalid,
                          uint16_t *__restrict__ Ap, uint16_t *__restrict__ AT)
{
    __shared__ Tile s;
    const int r0 = blockIdx.y * kSide, c0 = blockIdx.x * kSide, r = threadIdx.x / kSide, c = threadIdx.x % kSide;
    const size_t at = (size_t)(r0 + r) * H + c0 + c;
    const float z = r0 + r < nvalid ? Z[at] + bias[c0 + c] : 0.0f;
    s[r][c] = gelu(z);
    if (AT)
        Z[at] = z;
    __syncthreads();
    store_packed(s, r0, c0, B, H, Ap, AT);
}

// Last layer: Z (B x H) += bias (zero in rows >= nvalid, kept for a gradient), y[r] = gelu(Z[r]) . w4 + b4;
// one warp per row.
__global__ void output_kernel(float *__restrict__ Z, const float *__restrict__ bias, const float *__restrict__ w4,
                              const float *__restrict__ b4, int B, int H, int nvalid, bool keep,
                              float *__restrict__ y)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= B)
        return;
    float acc = 0.0f;
    for (int c = lane; c < H; c += 32) {
        const float z = warp < nvalid ? Z[(size_t)warp * H + c] + bias[c] : 0.0f;
        if (keep)
            Z[(size_t)warp * H + c] = z;
        acc = fmaf(gelu(z), w4[c], acc);
    }
    for (int off = 16; off > 0; off >>= 1)
        acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0)
        y[warp] = acc + b4[0];
}

// loss = mean (y - t)^2 over the valid rows, dy = 2 (y - t) / nvalid (0 on padded rows) and
// db4 = sum dy (fixed-order single-block sums).
__global__ void loss_kernel(const float *__restrict__ y, const float *__restrict__ t, int B, int nvalid,
                            float *__restrict__ dy, float *__restrict__ loss, float *__restrict__ db4)
{
    __shared__ float red[2][256];
    float acc = 0.0f, sum = 0.0f;
    for (int r = threadIdx.x; r < B; r += blockDim.x) {
        const float e = r < nvalid ? y[r] - t[r] : 0.0f;
        const float d = 2.0f * e / (float)nvalid;
        dy[r] = d;
        acc += e * e;
        sum += d;
    }
    red[0][threadIdx.x] = acc;
    red[1][threadIdx.x] = sum;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (loss)
            *loss = red[0][0] / (float)nvalid;
        *db4 = red[1][0];
    }
}

// dZ = dA gelu'(Z), packed and packed transposed, and its column sums per tile row of 32 into
// part[blockIdx.y][c].  dA is the product of the layer above or, in the last layer (OUT), dy w4^T;
// there part4 takes the sums of dy gelu(Z).
template <bool OUT>
__global__ void __launch_bounds__(kTileThreads)
    delta_kernel(const float *__restrict__ dA, const float *__restrict__ w4, const float *__restrict__ Z, int B, int H,
                 uint16_t *__restrict__ P, uint16_t *__restrict__ PT, float *__restrict__ part,
                 float *__restrict__ part4)
{
    __shared__ Tile s, s4;
    const int r0 = blockIdx.y * kSide, c0 = blockIdx.x * kSide, r = threadIdx.x / kSide, c = threadIdx.x % kSide;
    const size_t at = (size_t)(r0 + r) * H + c0 + c;
    const float z = Z[at];
    if constexpr (OUT) {
        const float dy = dA[r0 + r];
        s[r][c] = dy * w4[c0 + c] * gelu_grad(z);
        s4[r][c] = dy * gelu(z);
    } else {
        s[r][c] = dA[at] * gelu_grad(z);
    }
    __syncthreads();
    store_packed(s, r0, c0, B, H, P, PT);
    // columns: by warps that store nothing
    if (r == kSide - 1 || (OUT && r == kSide - 2)) {
        const Tile &x = r == kSide - 1 ? s : s4;
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < kSide; ++k)
            acc += x[k][c];
        (r == kSide - 1 ? part : part4)[(size_t)blockIdx.y * H + c0 + c] = acc;
    }
}

// The rest of the gradient: blocks [0, 4 H / 32) sum the tile rows' column sums of the four vectors
// (32 columns each, 32 threads a column, fixed order); the others copy W1's block from the
// product, whose rows are padded to ldd.
struct GradientEnd {
    const float *part;      // [4][tiles][H]
    float *sums[4];
    const float *D;         // rows x ldd, NULL: in place already
    float *W1;
    int tiles, H, din, ldd;
};

__global__ void __launch_bounds__(kTileThreads) gradient_end_kernel(GradientEnd q)
{
    const int groups = q.H / kSide;
    if ((int)blockIdx.x >= 4 * groups) {
        const long long i = (long long)(blockIdx.x - 4 * groups) * kTileThreads + threadIdx.x;
        if (i < (long long)q.H * q.din)
            q.W1[i] = q.D[(size_t)(i / q.din) * q.ldd + i % q.din];
        return;
    }
    constexpr int kWays = kTileThreads / kSide;
    __shared__ Tile red;
    const int v = blockIdx.x / groups, c = blockIdx.x % groups * kSide + threadIdx.x % kSide, w = threadIdx.x / kSide;
    const float *part = q.part + (size_t)v * q.tiles * q.H + c;
    float acc = 0.0f;
    for (int i = w; i < q.tiles; i += kWays)
        acc += part[(size_t)i * q.H];
    red[w][threadIdx.x % kSide] = acc;
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 1; k < kWays; ++k)
            acc += red[k][threadIdx.x];
        q.sums[v][c] = acc;
    }
}

// Adam (Kingma, Ba 2015) with bias correction; step is the 1-based step number.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, long long n, float lr, float b1, float b2, float eps,
                            float c1, float c2)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// FP64 parameter vectors -> normalised FP32 network inputs: (x - lo) / (hi - lo) - 1/2
__global__ void features_kernel(const double *__restrict__ P, int B, int D, const double *__restrict__ lo,
                                const double *__restrict__ hi, int ldx, float *__restrict__ X)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)B * D)
        return;
    const int r = (int)(i / D), c = (int)(i % D);
    X[(size_t)r * ldx + c] = (float)((P[i] - lo[c]) / (hi[c] - lo[c]) - 0.5);
}

// trial[i] = props[r*][i] with r* = argmax_r y[r NP + i] (first maximum);
// kept[i] = r* NP + i
__global__ void pick_best_kernel(const double *__restrict__ props, const float *__restrict__ y, int R, int NP,
                                 int D, double *__restrict__ trial, int32_t *__restrict__ kept)
{
    const int i = blockIdx.x;
    int best = 0;
    float bv = y[i];
    for (int r = 1; r < R; ++r) {
        const float v = y[(size_t)r * NP + i];
        if (v > bv) {
            bv = v;
            best = r;
        }
    }
    for (int j = threadIdx.x; j < D; j += blockDim.x)
        trial[(size_t)i * D + j] = props[((size_t)best * NP + i) * D + j];
    if (threadIdx.x == 0)
        kept[i] = best * NP + i;
}

__device__ __forceinline__ float rank_key(float v) { return isnan(v) ? -INFINITY : v; }

// Global top-NP of the n = R NP predictions: element k has rank
// #{j : y_j > y_k or (y_j = y_k and j < k)} (NaN ranks as -inf); the element of
// rank r < NP goes to row r of trial and kept[r] = k.
constexpr int kRankThreads = 256;
__global__ void __launch_bounds__(kRankThreads) rank_top_kernel(const double *__restrict__ props,
                                                                const float *__restrict__ y, int n, int NP,
                                                                int D, double *__restrict__ trial,
                                                                int32_t *__restrict__ kept)
{
    __shared__ float tile[kRankThreads];
    const int k = blockIdx.x * kRankThreads + threadIdx.x;
    const float yk = k < n ? rank_key(y[k]) : 0.0f;
    int rank = 0;
    for (int j0 = 0; j0 < n; j0 += kRankThreads) {
        const int j = j0 + threadIdx.x;
        tile[threadIdx.x] = j < n ? rank_key(y[j]) : -INFINITY;
        __syncthreads();
        const int m = min(kRankThreads, n - j0);
        for (int q = 0; q < m; ++q) {
            const float v = tile[q];
            rank += (v > yk) || (v == yk && j0 + q < k);
        }
        __syncthreads();
    }
    if (k < n && rank < NP) {
        kept[rank] = k;
        for (int c = 0; c < D; ++c)
            trial[(size_t)rank * D + c] = props[(size_t)k * D + c];
    }
}

// Selection after global screening: individual i takes the best exactly scored
// trial among those whose parent (kept[r] mod NP) is i (first maximum, NaN never
// chosen) when its pair number is >= fit[i].  One block per individual.
__global__ void group_select_kernel(double *__restrict__ pop, double *__restrict__ fit,
                                    const double *__restrict__ trial, const double *__restrict__ tfit,
                                    const int32_t *__restrict__ kept, int NP, int D)
{
    __shared__ int s_best;
    const int i = blockIdx.x;
    if (threadIdx.x == 0) {
        int best = -1;
        double bv = 0.0;
        for (int r = 0; r < NP; ++r) {
            const double v = tfit[r];
            if (kept[r] % NP != i || isnan(v))
                continue;
            if (best < 0 || v > bv) {
                best = r;
                bv = v;
            }
        }
        s_best = (best >= 0 && bv >= fit[i]) ? best : -1;
    }
    __syncthreads();
    const int r = s_best;
    if (r < 0)
        return;
    for (int j = threadIdx.x; j < D; j += blockDim.x)
        pop[(size_t)i * D + j] = trial[(size_t)r * D + j];
    if (threadIdx.x == 0)
        fit[i] = tfit[r];
}

// SplitMix64 output k of the generator seeded with s (Steele, Lea, Flood 2014).
__host__ __device__ __forceinline__ uint64_t mlp_sm64_at(uint64_t s, uint64_t k)
{
    uint64_t z = s + (k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Row order of one training epoch: a bijection of [0, n) from a 4-round Feistel
// network on b-bit integers (b the least even number with 2^b >= n; halves of
// hb = b/2 bits; round i maps (L, R) to (R, L xor (out(k_i, R) mod 2^hb)), out =
// SplitMix64), applied again while the value is >= n (cycle walking: the walk
// stays on the cycle through x, which returns below n within 2^b steps).
struct RowShuffle {
    uint64_t k[4];
    int hb;
    long long n;
};

__device__ __forceinline__ long long shuffled_row(const RowShuffle &r, long long x)
{
    const uint64_t mask = (1ull << r.hb) - 1ull;
    const long long dom = 1ll << (2 * r.hb);
    for (long long it = 0; it < dom; ++it) {
        uint64_t L = (uint64_t)x >> r.hb, R = (uint64_t)x & mask;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint64_t F = mlp_sm64_at(r.k[i], R) & mask;
            const uint64_t nL = R;
            R = L ^ F;
            L = nL;
        }
        x = (long long)((L << r.hb) | R);
        if (x < r.n)
            break;
    }
    return x;
}

// Mini-batch rows r0 .. r0 + rows - 1 of an epoch into the staging buffers.
__global__ void gather_rows_kernel(const float *__restrict__ X, const float *__restrict__ t, int din,
                                   RowShuffle sh, long long r0, int rows, float *__restrict__ Xs,
                                   float *__restrict__ ts)
{
    const int i = blockIdx.x;
    if (i >= rows)
        return;
    const long long src = shuffled_row(sh, r0 + i);
    for (int j = threadIdx.x; j < din; j += blockDim.x)
        Xs[(size_t)i * din + j] = X[(size_t)src * din + j];
    if (threadIdx.x == 0)
        ts[i] = t[src];
}

// He initialisation: parameter i of a weight block with fan-in f is
// sqrt(2/f) times a standard normal from the Box-Muller transform of outputs
// 2i and 2i+1; biases are zero.  Blocks: [W1 | b1 | W2 | b2 | W3 | b3 | w4 | b4].
__global__ void he_init_kernel(float *__restrict__ p, long long n, long long oW1, long long ob1,
                               long long oW2, long long ob2, long long oW3, long long ob3, long long ow4,
                               long long ob4, int din, int H, uint64_t seed)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    int fan = 0;
    if (i >= oW1 && i < ob1)
        fan = din;
    else if ((i >= oW2 && i < ob2) || (i >= oW3 && i < ob3) || (i >= ow4 && i < ob4))
        fan = H;
    if (!fan) {
        p[i] = 0.0f;
        return;
    }
    const double u1 = ((double)(mlp_sm64_at(seed, 2 * (uint64_t)i) >> 11) + 1.0) * 0x1.0p-53;  // (0, 1]
    const double u2 = (double)(mlp_sm64_at(seed, 2 * (uint64_t)i + 1) >> 11) * 0x1.0p-53;
    const double z = sqrt(-2.0 * log(u1)) * cos(2.0 * M_PI * u2);
    p[i] = (float)(z * sqrt(2.0 / fan));
}

// t = (log10(max(N, floor)) - shift) / scale
__global__ void log_targets_kernel(const double *__restrict__ N, int n, double floor_, double shift,
                                   double scale, float *__restrict__ t)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const double v = N[i];
        t[i] = (float)((log10(v > floor_ ? v : floor_) - shift) / scale);
    }
}

inline unsigned nb(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

struct pp_mlp {
    int dev = 0, din = 0, H = 0, dinp = 0, bmax = 0;
    long long nparam = 0;
    long long off_W1, off_b1, off_W2, off_b2, off_W3, off_b3, off_w4, off_b4;
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
    long long step = 0;
    // packed weights
    void *W1p = nullptr, *W2p = nullptr, *W3p = nullptr, *W2Tp = nullptr, *W3Tp = nullptr;
    // activations (bmax rows)
    float *X = nullptr, *Z1 = nullptr, *Z2 = nullptr, *Z3 = nullptr, *y = nullptr, *dy = nullptr, *dA = nullptr,
          *D = nullptr, *part = nullptr;
    void *Xp = nullptr, *A1p = nullptr, *A2p = nullptr, *dZp = nullptr;
    void *XTp = nullptr, *A1Tp = nullptr, *A2Tp = nullptr, *dZTp = nullptr;  // transposed, for the gradients
    // shuffled mini-batches of pp_mlp_fit (bmax rows)
    float *Xs = nullptr, *ts = nullptr;
};

namespace {

size_t packed_bytes(int r, int c) { return (size_t)((r + 127) / 128 * 128) * ((c + 63) / 64 * 64) * 2; }

void mlp_free(pp_mlp *h)
{
    if (!h)
        return;
    void *ptrs[] = {h->p, h->m, h->v, h->g, h->W1p, h->W2p, h->W3p, h->W2Tp, h->W3Tp, h->X, h->Z1, h->Z2,
                    h->Z3, h->y, h->dy, h->dA, h->D, h->part, h->Xp, h->A1p, h->A2p, h->dZp, h->XTp, h->A1Tp,
                    h->A2Tp, h->dZTp, h->Xs, h->ts};
    for (void *q : ptrs)
        if (q)
            cudaFree(q);
    delete h;
}

int repack_weights(pp_mlp *h, cudaStream_t st)
{
    const int H = h->H;
    int rc = pp::launch_pack_bf16(h->p + h->off_W1, H, h->din, h->din, 0, h->W1p, H, h->dinp, st);
    if (!rc)
        rc = pp::launch_pack_bf16(h->p + h->off_W2, H, H, H, 0, h->W2p, H, H, st);
    if (!rc)
        rc = pp::launch_pack_bf16(h->p + h->off_W3, H, H, H, 0, h->W3p, H, H, st);
    if (!rc)  // W^T for dA = dZ W: B operand [in][out]
        rc = pp::launch_pack_bf16(h->p + h->off_W2, H, H, H, 1, h->W2Tp, H, H, st);
    if (!rc)
        rc = pp::launch_pack_bf16(h->p + h->off_W3, H, H, H, 1, h->W3Tp, H, H, st);
    return rc;
}

// CTAs of the tiled passes over a (rows x cols) matrix
dim3 tiles(int rows, int cols) { return dim3(cols / kSide, rows / kSide); }

// Forward on X (rows x din, already in h->X, rows padded to Bp); y into h->y.  grad: what the
// backward pass reads is kept (the sums of each layer, the activations transposed).
int forward(pp_mlp *h, int Bp, int nvalid, bool grad, cudaStream_t st)
{
    const int H = h->H;
    pack_input_kernel<<<tiles(Bp, h->dinp), kTileThreads, 0, st>>>(h->X, Bp, h->dinp, (uint16_t *)h->Xp,
                                                                  grad ? (uint16_t *)h->XTp : nullptr);
    int rc = pp::launch_gemm_bf16(h->Xp, h->W1p, h->Z1, Bp, H, h->dinp, H, st);
    if (rc)
        return rc;
    bias_gelu_pack_kernel<<<tiles(Bp, H), kTileThreads, 0, st>>>(h->Z1, h->p + h->off_b1, Bp, H, nvalid,
                                                                (uint16_t *)h->A1p,
                                                                grad ? (uint16_t *)h->A1Tp : nullptr);
    rc = pp::launch_gemm_bf16(h->A1p, h->W2p, h->Z2, Bp, H, H, H, st);
    if (rc)
        return rc;
    bias_gelu_pack_kernel<<<tiles(Bp, H), kTileThreads, 0, st>>>(h->Z2, h->p + h->off_b2, Bp, H, nvalid,
                                                                (uint16_t *)h->A2p,
                                                                grad ? (uint16_t *)h->A2Tp : nullptr);
    rc = pp::launch_gemm_bf16(h->A2p, h->W3p, h->Z3, Bp, H, H, H, st);
    if (rc)
        return rc;
    output_kernel<<<nb((long long)Bp * 32), 256, 0, st>>>(h->Z3, h->p + h->off_b3, h->p + h->off_w4, h->p + h->off_b4,
                                                           Bp, H, nvalid, grad, h->y);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "surrogate forward");
}

// Backward after forward with grad; gradient into h->g.  The weight gradients of the hidden layers
// are products straight into their blocks of it.
int backward(pp_mlp *h, const float *t, int Bp, int nvalid, float *loss, cudaStream_t st)
{
    const int H = h->H, ntile = Bp / kSide;
    float *g = h->g, *part = h->part;
    uint16_t *dZp = (uint16_t *)h->dZp, *dZTp = (uint16_t *)h->dZTp;
    const size_t np = (size_t)ntile * H;
    loss_kernel<<<1, 256, 0, st>>>(h->y, t, Bp, nvalid, h->dy, loss, g + h->off_b4);
    // layer 3: dZ3, dW3 = dZ3^T A2, dA2 = dZ3 W3
    delta_kernel<true><<<tiles(Bp, H), kTileThreads, 0, st>>>(h->dy, h->p + h->off_w4, h->Z3, Bp, H, dZp, dZTp, part,
                                                             part + 3 * np);
    int rc = pp::launch_gemm_pair_bf16(dZTp, h->A2Tp, g + h->off_W3, H, H, Bp, dZp, h->W3Tp, h->dA, Bp, H, H, st);
    if (rc)
        return rc;
    // layer 2
    delta_kernel<false><<<tiles(Bp, H), kTileThreads, 0, st>>>(h->dA, nullptr, h->Z2, Bp, H, dZp, dZTp, part + np,
                                                              nullptr);
    rc = pp::launch_gemm_pair_bf16(dZTp, h->A1Tp, g + h->off_W2, H, H, Bp, dZp, h->W2Tp, h->dA, Bp, H, H, st);
    if (rc)
        return rc;
    // layer 1: dW1 = dZ1^T X, its columns padded unless d_in is a multiple of 64
    delta_kernel<false><<<tiles(Bp, H), kTileThreads, 0, st>>>(h->dA, nullptr, h->Z1, Bp, H, nullptr, dZTp,
                                                              part + 2 * np, nullptr);
    const bool padded = h->din != h->dinp;
    rc = pp::launch_gemm_bf16(dZTp, h->XTp, padded ? h->D : g + h->off_W1, H, h->dinp, Bp, h->dinp, st);
    if (rc)
        return rc;
    GradientEnd q = {part, {g + h->off_b3, g + h->off_b2, g + h->off_b1, g + h->off_w4}, h->D, g + h->off_W1, ntile, H,
                     h->din, h->dinp};
    const unsigned copies = padded ? nb((long long)H * h->din, kTileThreads) : 0;
    gradient_end_kernel<<<4 * (H / kSide) + copies, kTileThreads, 0, st>>>(q);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "surrogate backward");
}

int stage_inputs(pp_mlp *h, const float *X, int B, cudaStream_t st)
{
    const int Bp = (B + kRows - 1) / kRows * kRows;
    cudaError_t e = cudaMemsetAsync(h->X, 0, sizeof(float) * (size_t)Bp * h->dinp, st);
    if (e == cudaSuccess)
        e = cudaMemcpy2DAsync(h->X, sizeof(float) * h->dinp, X, sizeof(float) * h->din, sizeof(float) * h->din,
                              B, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "surrogate input staging");
}

}  // namespace

using namespace pp;

extern "C" {

int pp_mlp_create(int32_t d_in, int32_t hidden, int32_t max_batch, pp_mlp **out)
{
    clear_error();
    if (!out)
        return fail(PP_ERR_INVALID_ARG, "out must not be NULL");
    *out = nullptr;
    // hidden is a whole number of 128-row GEMM tiles: it is the M of the weight-gradient
    // products and the K (and packed width) of the hidden layers
    if (d_in < 1 || d_in > 256 || (hidden != 128 && hidden != 256) || max_batch < 1 || max_batch > (1 << 20))
        return fail(PP_ERR_INVALID_ARG, "need 1 <= d_in <= 256, hidden = 128 or 256, 1 <= max_batch <= 2^20");
    pp_mlp *h = new pp_mlp();
    cudaGetDevice(&h->dev);
    h->din = d_in;
    h->H = hidden;
    h->dinp = (d_in + 63) / 64 * 64;
    if (h->dinp > 256) {
        delete h;
        return fail(PP_ERR_INVALID_ARG, "d_in too large");
    }
    h->bmax = (max_batch + kRows - 1) / kRows * kRows;
    const long long H = hidden;
    h->off_W1 = 0;
    h->off_b1 = H * d_in;
    h->off_W2 = h->off_b1 + H;
    h->off_b2 = h->off_W2 + H * H;
    h->off_W3 = h->off_b2 + H;
    h->off_b3 = h->off_W3 + H * H;
    h->off_w4 = h->off_b3 + H;
    h->off_b4 = h->off_w4 + H;
    h->nparam = h->off_b4 + 1;
    const size_t BH = (size_t)h->bmax * hidden;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **pp_, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaMalloc(pp_, bytes);
        if (e == cudaSuccess)
            e = cudaMemset(*pp_, 0, bytes);
    };
    alloc((void **)&h->p, sizeof(float) * h->nparam);
    alloc((void **)&h->m, sizeof(float) * h->nparam);
    alloc((void **)&h->v, sizeof(float) * h->nparam);
    alloc((void **)&h->g, sizeof(float) * h->nparam);
    alloc(&h->W1p, packed_bytes(hidden, h->dinp));
    alloc(&h->W2p, packed_bytes(hidden, hidden));
    alloc(&h->W3p, packed_bytes(hidden, hidden));
    alloc(&h->W2Tp, packed_bytes(hidden, hidden));
    alloc(&h->W3Tp, packed_bytes(hidden, hidden));
    alloc((void **)&h->X, sizeof(float) * (size_t)h->bmax * h->dinp);
    float **acts[] = {&h->Z1, &h->Z2, &h->Z3, &h->dA};
    for (float **a : acts)
        alloc((void **)a, sizeof(float) * BH);
    alloc((void **)&h->D, sizeof(float) * (size_t)hidden * h->dinp);
    alloc((void **)&h->part, sizeof(float) * 4 * BH / kSide);
    alloc((void **)&h->y, sizeof(float) * h->bmax);
    alloc((void **)&h->dy, sizeof(float) * h->bmax);
    alloc(&h->Xp, packed_bytes(h->bmax, h->dinp));
    alloc(&h->XTp, packed_bytes(h->dinp, h->bmax));
    void **hidden_packed[] = {&h->A1p, &h->A2p, &h->dZp}, **hidden_trans[] = {&h->A1Tp, &h->A2Tp, &h->dZTp};
    for (int i = 0; i < 3; ++i) {
        alloc(hidden_packed[i], packed_bytes(h->bmax, hidden));
        alloc(hidden_trans[i], packed_bytes(hidden, h->bmax));
    }
    alloc((void **)&h->Xs, sizeof(float) * (size_t)h->bmax * h->din);
    alloc((void **)&h->ts, sizeof(float) * h->bmax);
    if (e != cudaSuccess) {
        mlp_free(h);
        return cuda_fail(e, "surrogate allocation");
    }
    *out = h;
    return PP_OK;
}

void pp_mlp_destroy(pp_mlp *h) { mlp_free(h); }

int64_t pp_mlp_num_params(const pp_mlp *h) { return h ? h->nparam : 0; }

int pp_mlp_set_params(pp_mlp *h, const float *params, void *stream)
{
    clear_error();
    if (!h || !params)
        return fail(PP_ERR_INVALID_ARG, "handle and params must not be NULL");
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(h->p, params, sizeof(float) * h->nparam, cudaMemcpyDefault, st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(h->m, 0, sizeof(float) * h->nparam, st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(h->v, 0, sizeof(float) * h->nparam, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "surrogate parameters");
    h->step = 0;
    return repack_weights(h, st);
}

int pp_mlp_init(pp_mlp *h, uint64_t seed, void *stream)
{
    clear_error();
    if (!h)
        return fail(PP_ERR_INVALID_ARG, "network handle is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    he_init_kernel<<<nb(h->nparam), 256, 0, st>>>(h->p, h->nparam, h->off_W1, h->off_b1, h->off_W2, h->off_b2,
                                                   h->off_W3, h->off_b3, h->off_w4, h->off_b4, h->din, h->H,
                                                   seed);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemsetAsync(h->m, 0, sizeof(float) * h->nparam, st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(h->v, 0, sizeof(float) * h->nparam, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "surrogate initialisation");
    h->step = 0;
    return repack_weights(h, st);
}

int pp_mlp_get_params(const pp_mlp *h, float *params, void *stream)
{
    clear_error();
    if (!h || !params)
        return fail(PP_ERR_INVALID_ARG, "handle and params must not be NULL");
    cudaError_t e = cudaMemcpyAsync(params, h->p, sizeof(float) * h->nparam, cudaMemcpyDefault,
                                    (cudaStream_t)stream);
    return e == cudaSuccess ? PP_OK : cuda_fail(e, "surrogate parameters");
}

int pp_mlp_forward(pp_mlp *h, const float *X, int32_t B, float *y, void *stream)
{
    clear_error();
    if (!h || !X || !y || B < 1 || B > h->bmax)
        return fail(PP_ERR_INVALID_ARG, "need a handle, X, y and 1 <= B <= max_batch");
    cudaStream_t st = (cudaStream_t)stream;
    const int Bp = (B + kRows - 1) / kRows * kRows;
    int rc = stage_inputs(h, X, B, st);
    if (!rc)
        rc = forward(h, Bp, B, false, st);
    if (rc)
        return rc;
    cudaError_t e = cudaMemcpyAsync(y, h->y, sizeof(float) * B, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? PP_OK : cuda_fail(e, "surrogate output");
}

int pp_mlp_loss_grad(pp_mlp *h, const float *X, const float *t, int32_t B, float *loss, float *grad,
                     void *stream)
{
    clear_error();
    if (!h || !X || !t || B < 1 || B > h->bmax)
        return fail(PP_ERR_INVALID_ARG, "need a handle, X, t and 1 <= B <= max_batch");
    cudaStream_t st = (cudaStream_t)stream;
    const int Bp = (B + kRows - 1) / kRows * kRows;
    int rc = stage_inputs(h, X, B, st);
    if (!rc)
        rc = forward(h, Bp, B, true, st);
    if (!rc) {
        // targets on padded rows are never read (dy = 0 there)
        rc = backward(h, t, Bp, B, loss, st);
    }
    if (rc)
        return rc;
    if (grad) {
        cudaError_t e = cudaMemcpyAsync(grad, h->g, sizeof(float) * h->nparam, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "surrogate gradient");
    }
    return PP_OK;
}

int pp_mlp_train_step(pp_mlp *h, const float *X, const float *t, int32_t B, float lr, float *loss,
                      void *stream)
{
    int rc = pp_mlp_loss_grad(h, X, t, B, loss, nullptr, stream);
    if (rc)
        return rc;
    cudaStream_t st = (cudaStream_t)stream;
    h->step += 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.0f - powf(b1, (float)h->step), c2 = 1.0f - powf(b2, (float)h->step);
    adam_kernel<<<nb(h->nparam), 256, 0, st>>>(h->p, h->g, h->m, h->v, h->nparam, lr, b1, b2, eps, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "Adam");
    return repack_weights(h, st);
}

int pp_mlp_fit(pp_mlp *h, const float *X, const float *t, int32_t n, int32_t batch, int32_t epochs,
               float lr0, float lr1, uint64_t seed, float *epoch_loss, void *stream)
{
    clear_error();
    if (!h || !X || !t || n < 1 || batch < 1 || batch > h->bmax || epochs < 1)
        return fail(PP_ERR_INVALID_ARG, "need a network, X and t, n >= 1, 1 <= batch <= max_batch, epochs >= 1");
    if (!(lr0 >= 0.0f) || !(lr1 >= 0.0f))
        return fail(PP_ERR_INVALID_ARG, "learning rates must be non-negative");
    cudaStream_t st = (cudaStream_t)stream;
    RowShuffle sh;
    sh.n = n;
    sh.hb = 0;
    while ((1ll << (2 * sh.hb)) < (long long)n)
        ++sh.hb;
    const long long per = (n + (long long)batch - 1) / batch, total = per * epochs;
    long long k = 0;
    for (int e = 0; e < epochs; ++e) {
        for (int i = 0; i < 4; ++i)
            sh.k[i] = mlp_sm64_at(seed, 4 * (uint64_t)e + (uint64_t)i);
        for (long long b = 0; b < per; ++b, ++k) {
            const int r0 = (int)(b * batch), rows = (int)std::min<long long>(batch, n - r0);
            // cosine schedule from lr0 (first step) to lr1 (last step)
            const double c = total > 1 ? 0.5 * (1.0 + cos(M_PI * (double)k / (double)(total - 1))) : 1.0;
            const float lr = (float)(lr1 + (lr0 - lr1) * c);
            float *loss = (epoch_loss && b == per - 1) ? epoch_loss + e : nullptr;
            const float *Xb = X + (size_t)r0 * h->din, *tb = t + r0;
            if (seed != 0) {
                gather_rows_kernel<<<rows, 64, 0, st>>>(X, t, h->din, sh, r0, rows, h->Xs, h->ts);
                cudaError_t eg = cudaGetLastError();
                if (eg != cudaSuccess)
                    return cuda_fail(eg, "mini-batch gather");
                Xb = h->Xs;
                tb = h->ts;
            }
            const int rc = pp_mlp_train_step(h, Xb, tb, rows, lr, loss, stream);
            if (rc)
                return rc;
        }
    }
    return PP_OK;
}

int pp_mlp_log_targets(const double *N, int32_t n, double floor_value, double shift, double scale, float *t,
                       void *stream)
{
    clear_error();
    if (!N || !t || n < 0 || !(floor_value > 0.0) || !(scale != 0.0) || !isfinite(shift) || !isfinite(scale))
        return fail(PP_ERR_INVALID_ARG, "need N and t, n >= 0, floor > 0, finite shift and non-zero scale");
    if (n == 0)
        return PP_OK;
    log_targets_kernel<<<nb(n), 256, 0, (cudaStream_t)stream>>>(N, n, floor_value, shift, scale, t);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : cuda_fail(e, "log targets");
}

int pp_de_screened_step(double *pop, double *fit, int32_t NP, const pp_field_spec *spec,
                        const pp_grid *grid, int32_t precision, int32_t scheme, const double *lo,
                        const double *hi, const uint8_t *periodic, double F, double CR, uint64_t seed,
                        uint64_t generation, int32_t R, int32_t mode, pp_mlp *mlp, double *trial_out,
                        double *trial_fit_out, float *pred_out, int32_t *kept_out, void *stream)
{
    clear_error();
    int rc = check_spec(spec);
    if (!rc)
        rc = check_grid(grid);
    if (rc)
        return rc;
    if (!pop || !fit || !lo || !hi || !mlp)
        return fail(PP_ERR_INVALID_ARG, "pop, fit, lo, hi and mlp must not be NULL");
    if (precision != PP_FP64 && precision != PP_FP32 && precision != PP_FP32_FAST)
        return fail(PP_ERR_INVALID_ARG, "precision must be PP_FP64, PP_FP32 or PP_FP32_FAST");
    if (scheme != PP_RK4 && scheme != PP_MAGNUS4 && scheme != PP_SPLIT2)
        return fail(PP_ERR_INVALID_ARG, "scheme must be PP_RK4, PP_MAGNUS4 or PP_SPLIT2");
    const int D = 4 * spec->K;
    if (NP < 4 || NP > 65535 || R < 1 || R > 64 || (long long)R * NP > mlp->bmax || D != mlp->din)
        return fail(PP_ERR_INVALID_ARG, "need NP >= 4, 1 <= R <= 64, R NP <= the network's max_batch "
                                        "and 4K equal to its input size");
    if (!(CR >= 0.0 && CR <= 1.0) || !isfinite(F))
        return fail(PP_ERR_INVALID_ARG, "CR must be in [0, 1] and F finite");
    if (mode != PP_SCREEN_PER_INDIVIDUAL && mode != PP_SCREEN_GLOBAL)
        return fail(PP_ERR_INVALID_ARG, "mode must be PP_SCREEN_PER_INDIVIDUAL or PP_SCREEN_GLOBAL");
    cudaStream_t st = (cudaStream_t)stream;
    void *props = nullptr, *X = nullptr, *y = nullptr, *trial = nullptr, *tfit = nullptr, *A = nullptr;
    void *kept = nullptr;
    const int ld = 2 * spec->n_steps + 1;
    rc = scratch(SCR_SCREEN_PROPS, sizeof(double) * (size_t)R * NP * D, &props);
    if (!rc)
        rc = scratch(SCR_SCREEN_X, sizeof(float) * (size_t)R * NP * D, &X);
    if (!rc)
        rc = scratch(SCR_SCREEN_Y, sizeof(float) * (size_t)R * NP, &y);
    if (!rc && !trial_out)
        rc = scratch(SCR_TRIAL, sizeof(double) * (size_t)NP * D, &trial);
    if (!rc && !trial_fit_out)
        rc = scratch(SCR_TFIT, sizeof(double) * (size_t)NP, &tfit);
    if (!rc)
        rc = scratch(SCR_A, sizeof(double) * 2 * (size_t)ld * NP, &A);
    if (!rc && !kept_out)
        rc = scratch(SCR_SCREEN_KEPT, sizeof(int32_t) * (size_t)NP, &kept);
    if (rc)
        return rc;
    int32_t *kp = kept_out ? kept_out : (int32_t *)kept;
    double *tr = trial_out ? trial_out : (double *)trial;
    double *tf = trial_fit_out ? trial_fit_out : (double *)tfit;
    // R proposals per individual, each from its own counter-RNG stream (generation R g + r), in one launch
    rc = launch_de_propose(pop, NP, D, lo, hi, periodic, F, CR, seed, generation * (uint64_t)R, (double *)props, st, R);
    if (rc)
        return rc;
    features_kernel<<<nb((long long)R * NP * D), 256, 0, st>>>((const double *)props, R * NP, D, lo, hi, D,
                                                                (float *)X);
    rc = pp_mlp_forward(mlp, (const float *)X, R * NP, (float *)y, stream);
    if (rc)
        return rc;
    if (pred_out) {
        cudaError_t e = cudaMemcpyAsync(pred_out, y, sizeof(float) * (size_t)R * NP, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess)
            return cuda_fail(e, "screening predictions");
    }
    if (mode == PP_SCREEN_PER_INDIVIDUAL)
        pick_best_kernel<<<NP, 64, 0, st>>>((const double *)props, (const float *)y, R, NP, D, tr, kp);
    else
        rank_top_kernel<<<nb((long long)R * NP, kRankThreads), kRankThreads, 0, st>>>(
            (const double *)props, (const float *)y, R * NP, NP, D, tr, kp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "screening pick");
    if ((rc = launch_synth_field(tr, NP, spec, (double *)A, ld, nullptr, nullptr, st)))
        return rc;
    if ((rc = launch_pair_number((double *)A, NP, ld, nullptr, spec->T / spec->n_steps, grid, precision,
                                 scheme, tf, nullptr, st)))
        return rc;
    if (mode == PP_SCREEN_PER_INDIVIDUAL)
        return launch_de_select(pop, fit, tr, tf, NP, D, st);
    group_select_kernel<<<NP, 64, 0, st>>>(pop, fit, tr, tf, kp, NP, D);
    e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : cuda_fail(e, "screening selection");
}

int pp_mlp_features(const double *params, int32_t B, int32_t D, const double *lo, const double *hi,
                    float *X, void *stream)
{
    clear_error();
    if (!params || !lo || !hi || !X || B < 1 || D < 1)
        return fail(PP_ERR_INVALID_ARG, "bad arguments");
    features_kernel<<<nb((long long)B * D), 256, 0, (cudaStream_t)stream>>>(params, B, D, lo, hi, D, X);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : cuda_fail(e, "features");
}

}  // extern "C"
