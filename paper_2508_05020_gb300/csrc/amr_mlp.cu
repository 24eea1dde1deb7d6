// Learned refinement indicator, standalone calls of include/amr.h: feature
// embedding of 1D samples, BF16 tensor-core inference, FP32 gradient and Adam
// training. The paper leaves the refinement criterion to the runtime program
// (Sec. 4.2); this network is one such program. Training is deterministic:
// every reduction is a fixed-order loop, no atomics.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "amr.h"
#include "amr_internal.h"
#include "amr_mlp_core.cuh"
#include "amr_mlp_tc.cuh"

namespace amr {
int mlp_k(int dim) { return mlp_kin(dim); }
long mlp_n_weights(int dim) {
    const long K = mlp_kin(dim);
    return MLP_H * K + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1;
}
}  // namespace amr

using namespace amr;
namespace cg = cooperative_groups;

namespace {

// ---------------------------------------------------------------------------
// features: 1D 5-point samples (rho, u, p) embedded along axis a with sign s
// (point at offset o takes sample index 2 + s o_a, velocity component a = s u),
// normalised by the centre: rho/rho0 - 1, u/c0, p/p0 - 1, c0 = sqrt(gamma p0/rho0).
// Row 2 d i + 2 a + (s > 0); per point (z, y, x lexicographic) features (rho, u.., p).
// ---------------------------------------------------------------------------
__global__ void k_features(int D, double gamma, const double* __restrict__ smp, long n, float* __restrict__ X) {
    const int K = mlp_kin(D), F = D + 2;
    const long rows = n * 2 * D;
    for (long it = blockIdx.x * (long)blockDim.x + threadIdx.x; it < rows * K; it += (long)gridDim.x * blockDim.x) {
        const long row = it / K;
        const int k = (int)(it - row * K);
        const long i = row / (2 * D);
        const int r = (int)(row - i * 2 * D);
        const int a = r >> 1;
        const int s = (r & 1) ? 1 : -1;
        const int j = k / F, f = k - j * F;
        const int o[3] = {j % 5 - 2, D >= 2 ? (j / 5) % 5 - 2 : 0, D == 3 ? j / 25 - 2 : 0};
        const int idx = 2 + s * o[a];
        const double* S = smp + i * 15;
        const double r0 = S[2 * 3 + 0], p0 = S[2 * 3 + 2];
        const double c0 = sqrt(gamma * p0 / r0);
        double v;
        if (f == 0) v = S[idx * 3 + 0] / r0 - 1.0;
        else if (f == F - 1) v = S[idx * 3 + 2] / p0 - 1.0;
        else v = (f - 1 == a ? S[idx * 3 + 1] * s : 0.0) / c0;
        X[it] = (float)v;
    }
}

// standalone inference on feature rows (n x K floats, ABI feature order) on
// the tcgen05 core: 128-row tiles, features copied (BF16) into the canonical
// field-major chunk layout. Rows a timed-out CTA did not reach stay NaN.
template <int D> struct InferLayout {
    static constexpr size_t ABUF = (sizeof(MlpTcSmem<D>) + 127) / 128 * 128;
    static constexpr size_t HBUF = ABUF + 2 * sizeof(__nv_bfloat16) * TC_M * TC_KC;
    static constexpr size_t SLOTS = HBUF + sizeof(__nv_bfloat16) * TC_M * MLP_H;
    static constexpr size_t TOTAL = SLOTS + 4 * sizeof(uint64_t) + 128;
};

template <int D>
__global__ void __launch_bounds__(512, 1) k_infer(const float* __restrict__ X, long n, const float* __restrict__ w,
                                                  float* __restrict__ z, int* err) {
    using Lay = InferLayout<D>;
    constexpr int K = mlp_kin(D), KP = mlp_kpad(D), F = D + 2, NP = mlp_npts(D), PTS = mlp_pts(D);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    MlpTcSmem<D>& s = *reinterpret_cast<MlpTcSmem<D>*>(base);
    __nv_bfloat16* abuf = reinterpret_cast<__nv_bfloat16*>(base + Lay::ABUF);
    __nv_bfloat16* hbuf = reinterpret_cast<__nv_bfloat16*>(base + Lay::HBUF);
    uint64_t* slots = reinterpret_cast<uint64_t*>(base + Lay::SLOTS);
    mlp_tc_stage_weights<D>(s, w);
    TcState st;
    tc_setup(st, slots);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int frow = (warp & 3) * 32 + lane, fslice = warp >> 2;
    const long tiles = (n + TC_M - 1) / TC_M;
    for (long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long r = tile * TC_M + frow;
        const float* x = X + (r < n ? r : n - 1) * K;
        auto fill = [&](int cc, __nv_bfloat16* dst) {
            const int k0 = cc * TC_KC + fslice * 16;
            uint32_t wv[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float v2[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int kp = k0 + 2 * e + h;
                    const int f = kp / PTS, j = kp - f * PTS;
                    v2[h] = (kp < KP && j < NP) ? x[j * F + f] : 0.f;
                }
                wv[e] = pack_bf16(v2[0], v2[1]);
            }
            *reinterpret_cast<uint4*>(dst + canon_off(frow, fslice * 16, TC_KC)) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
            *reinterpret_cast<uint4*>(dst + canon_off(frow, fslice * 16 + 8, TC_KC)) = make_uint4(wv[4], wv[5], wv[6], wv[7]);
        };
        const float zz = mlp_tile_tc<D>(st, s, abuf, hbuf, fill);
        if (!__syncthreads_and(st.ok ? 1 : 0)) {
            if (threadIdx.x == 0) atomicOr(err, 1);
            break;
        }
        if (warp < 4) {
            const long ro = tile * TC_M + warp * 32 + lane;
            if (ro < n) z[ro] = zz;
        }
    }
    tc_teardown(st);
}

// ---------------------------------------------------------------------------
// FP32 training kernels (rows of a minibatch selected by idx): loss and
// gradient of n rows in three launches.
//   k_rows     everything that is local to a row: both hidden layers, the
//              logit, dz, the gradients of the hidden layers, and this block's
//              part of the gradients of b1, W2, b2, w3, b3 and of the loss
//   k_w1grad   dW1 = dH1^T X, split over the rows
//   k_gradsum  the parts added in a fixed order (and the Adam update in training)
// Every sum has a fixed order, so equal calls give equal bits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float softplus(float x) { return fmaxf(x, 0.f) + log1pf(expf(-fabsf(x))); }

// the gradients of b1, W2, b2, w3, b3 (the flat layout after W1), then the loss
constexpr int SMALL = MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1;
constexpr int SMALL_L = SMALL + 1;
constexpr int ROWS_NTH = 512;
constexpr int ROWS_CL = 4;                  // blocks of a cluster, whose parts are added in shared memory
constexpr int ROWS_MAXCL = 32;              // clusters of a launch
constexpr int W1_CT = 16;                   // columns of X of a k_w1grad block
constexpr int W1_NTH = 512, W1_G = W1_NTH / 64;   // threads of a k_w1grad block, its row groups
constexpr int W1_RC = 128;                  // rows staged at a time
constexpr int W1_PARTS = 160000;            // floats of the split dW1 (4 x 64 x 625)

// row splits of k_w1grad: up to 160 blocks over the column tiles, as far as the
// parts fit their buffer (3D: 40 tiles by 4, so 8 of 152 SMs hold two blocks)
__host__ __device__ constexpr int w1_tiles(int K) { return (K + W1_CT - 1) / W1_CT; }
__host__ __device__ constexpr int w1_splits(int K) {
    int s = 160 / w1_tiles(K);
    const int fit = W1_PARTS / (MLP_H * K);
    s = s < fit ? s : fit;
    return s < 32 ? s : 32;
}

// Sums v[0 .. M) over the 32 lanes: at each step a lane keeps the half of its
// values that its lane bit names and adds the partner's, so the whole sum
// takes M - 1 (+ the steps left once one value remains) shuffles instead of
// 5 M. Afterwards lane holds the values `base ..`, max(M / 32, 1) of them.
template <int M>
__device__ __forceinline__ int lane_sums(float (&v)[M]) {
    const int lane = threadIdx.x & 31;
    int base = 0, m = M;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        if (m > 1) {
            m >>= 1;
            const bool hi = lane & s;
            if (hi) base += m;
#pragma unroll
            for (int i = 0; i < M / 2; ++i) {
                if (i < m) {
                    const float keep = hi ? v[i + m] : v[i], send = hi ? v[i] : v[i + m];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], s);
        }
    }
    return base;
}

// R rows per tile. Layer 1 is the work: a warp owns 4 of the 64 outputs, its
// lanes run along K (W1 is read once per block, coalesced, from L2, the rows
// from shared memory), and the lanes' sums are added at the end. Bound by the
// L2 latency of the W1 stream and FMA issue. The three launches take 42 us for
// the 3D gradient of 2048 rows; with one thread per (row, output) or weight,
// each looping serially over K or over all the rows, it took 772 us.
template <int D, int R>
__global__ void __cluster_dims__(ROWS_CL, 1, 1) __launch_bounds__(ROWS_NTH)
    k_rows(const float* __restrict__ X, const int* __restrict__ idx, const float* __restrict__ y, long n, float pw,
           const float* __restrict__ w, float* __restrict__ dH1, float* __restrict__ part) {
    constexpr int K = mlp_kin(D), H = MLP_H, P2 = H + 1;
    constexpr int KS = (K + 31) / 32, OW = H / (ROWS_NTH / 32);     // lane steps; outputs per warp
    constexpr int AREA0 = R * K > H * P2 + R * H ? R * K : H * P2 + R * H;
    constexpr int AREA = AREA0 > SMALL_L ? AREA0 : SMALL_L;
    // the rows of X, later W2 (padded rows) and dH1, at the end the block's sums
    __shared__ float area[AREA];
    __shared__ float H1[R * H], H2[R * H];
    __shared__ float dz[R], ls[R];
    float* Xs = area;
    float* W2s = area;
    float* D1 = area + H * P2;
    const float* W1 = w;
    const float* b1 = W1 + H * K;
    const float* W2 = b1 + H;
    const float* b2 = W2 + H * H;
    const float* w3 = b2 + H;
    const float* b3 = w3 + H;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int o = t & (H - 1), rg = t >> 6;                // (output, row group) of the small products
    float aw2[H * H / ROWS_NTH], as = 0.f;                 // this thread's entries of dW2; of the vectors
#pragma unroll
    for (int i = 0; i < H * H / ROWS_NTH; ++i) aw2[i] = 0.f;
    const long tiles = (n + R - 1) / R;
    float w2r[H * H / ROWS_NTH];                           // W2 on its way while layer 1 runs
    for (long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long r0 = tile * R;
        const int nr = (int)(n - r0 < R ? n - r0 : R);
        for (int i = t; i < R * K; i += ROWS_NTH) {
            const int r = i / K, k = i - r * K;
            Xs[i] = r < nr ? X[(long)(idx ? idx[r0 + r] : r0 + r) * K + k] : 0.f;
        }
        __syncthreads();
        {
            float acc[OW * R];
#pragma unroll
            for (int i = 0; i < OW * R; ++i) acc[i] = 0.f;
            // W1 is fetched PF lane steps ahead of its use
            constexpr int PF = KS < 4 ? KS : 4;
            float wv[PF][OW];
            auto fetch = [&](int ks, float (&o)[OW]) {
                const int k = ks * 32 + lane;
#pragma unroll
                for (int j = 0; j < OW; ++j) o[j] = k < K ? W1[(warp * OW + j) * K + k] : 0.f;
            };
#pragma unroll
            for (int b = 0; b < PF; ++b) fetch(b, wv[b]);
#pragma unroll
            for (int i = 0; i < H * H / ROWS_NTH; ++i) w2r[i] = W2[t + i * ROWS_NTH];
#pragma unroll 1
            for (int k0 = 0; k0 < KS; k0 += PF) {
#pragma unroll
                for (int b = 0; b < PF; ++b) {
                    const int ks = k0 + b, k = ks * 32 + lane;
                    if (KS % PF != 0 && ks >= KS) break;
                    const int kk = k < K ? k : K - 1;
                    float wk[OW];
#pragma unroll
                    for (int j = 0; j < OW; ++j) wk[j] = wv[b][j];
                    if (ks + PF < KS) fetch(ks + PF, wv[b]);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float x = Xs[r * K + kk];
                        if (K % 32 != 0 && b == (KS - 1) % PF) x = k < K ? x : 0.f;   // not 0 * inf
#pragma unroll
                        for (int j = 0; j < OW; ++j) acc[j * R + r] = fmaf(x, wk[j], acc[j * R + r]);
                    }
                }
            }
            const int base = lane_sums<OW * R>(acc);
            constexpr int LEFT = OW * R >= 32 ? OW * R / 32 : 1;
#pragma unroll
            for (int i = 0; i < LEFT; ++i) {
                const int j = (base + i) / R, r = (base + i) % R, oo = warp * OW + j;
                H1[r * H + oo] = r < nr ? fmaxf(acc[i] + b1[oo], 0.f) : 0.f;   // rows past the last: 0 throughout
            }
        }
        __syncthreads();                                   // the rows of X are read; H1 is written
#pragma unroll
        for (int i = 0; i < H * H / ROWS_NTH; ++i) {
            const int e = t + i * ROWS_NTH;
            W2s[(e >> 6) * P2 + (e & (H - 1))] = w2r[i];
        }
        __syncthreads();
        for (int r = rg; r < R; r += ROWS_NTH / H) {
            float acc = b2[o];
#pragma unroll 16
            for (int k = 0; k < H; ++k) acc = fmaf(H1[r * H + k], W2s[o * P2 + k], acc);
            H2[r * H + o] = r < nr ? fmaxf(acc, 0.f) : 0.f;
        }
        __syncthreads();
        if (warp < R) {
            float z = H2[warp * H + lane] * w3[lane] + H2[warp * H + lane + 32] * w3[lane + 32];
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) z += __shfl_xor_sync(0xffffffffu, z, s);
            if (lane == 0) {
                z += b3[0];
                float d = 0.f, l = 0.f;
                if (warp < nr) {
                    const float yy = y[idx ? idx[r0 + warp] : r0 + warp];
                    const float sg = 0.5f * (1.f + tanhf(0.5f * z));
                    l = pw * yy * softplus(-z) + (1.f - yy) * softplus(z);
                    d = (pw * yy * (sg - 1.f) + (1.f - yy) * sg) / (float)n;
                }
                dz[warp] = d;
                ls[warp] = l;
            }
        }
        __syncthreads();
        if (t >= 128 && t < 192) {                         // dw3
            for (int r = 0; r < R; ++r) as = fmaf(dz[r], H2[r * H + t - 128], as);
        } else if (t == 192) {
            for (int r = 0; r < R; ++r) as += dz[r];
        } else if (t == 193) {
            for (int r = 0; r < R; ++r) as += ls[r];
        }
        __syncthreads();
        for (int r = rg; r < R; r += ROWS_NTH / H) H2[r * H + o] = H2[r * H + o] > 0.f ? dz[r] * w3[o] : 0.f;   // dH2
        __syncthreads();
        for (int r = rg; r < R; r += ROWS_NTH / H) {
            float acc = 0.f;
#pragma unroll 16
            for (int q = 0; q < H; ++q) acc = fmaf(H2[r * H + q], W2s[q * P2 + o], acc);
            const float d = H1[r * H + o] > 0.f ? acc : 0.f;
            D1[r * H + o] = d;
            if (r < nr) dH1[(r0 + r) * H + o] = d;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float d = H2[r * H + (t >> 3)];
#pragma unroll
            for (int i = 0; i < H * H / ROWS_NTH; ++i) aw2[i] = fmaf(d, H1[r * H + (t & 7) + 8 * i], aw2[i]);
        }
        __syncthreads();
        if (t < 64) {
            for (int r = 0; r < R; ++r) as += D1[r * H + t];
        } else if (t < 128) {
            for (int r = 0; r < R; ++r) as += H2[r * H + t - 64];
        }
        __syncthreads();
    }
    // the block's part, then the cluster's
    if (t < 64) area[t] = as;
    else if (t < 194) area[H * H + t] = as;                // b2, w3, b3, loss follow W2
#pragma unroll
    for (int i = 0; i < H * H / ROWS_NTH; ++i) area[H + (t >> 3) * H + (t & 7) + 8 * i] = aw2[i];
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int rank = (int)cl.block_rank();
    for (int e = rank * ROWS_NTH + t; e < SMALL_L; e += ROWS_CL * ROWS_NTH) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < ROWS_CL; ++q) s += *cl.map_shared_rank(area + e, q);
        part[(long)(blockIdx.x / ROWS_CL) * SMALL_L + e] = s;
    }
    cl.sync();                                             // a block's sums stay until its peers have read them
}

// dW1 of W1_CT columns over one split of the rows: rows are staged 128 at a time
// (the next ones on their way in registers), a thread owns 8 outputs x 2
// columns and every eighth row, so that 16 FMAs share three shared-memory
// loads; the eight row groups are added in order at the end. Bound by the
// latency of those loads: 16 warps per SM, as 8 left the scheduler idle in 60 % of the cycles.
template <int D>
__global__ void __launch_bounds__(W1_NTH) k_w1grad(const float* __restrict__ dH1, const float* __restrict__ X,
                                                const int* __restrict__ idx, long n, float* __restrict__ part) {
    constexpr int K = mlp_kin(D), H = MLP_H, CT = W1_CT, RC = W1_RC;
    constexpr int NTH = W1_NTH, ND = RC * H / 4 / NTH, NX = RC * CT / NTH;
    __shared__ __align__(16) float ds[RC * H];
    __shared__ __align__(16) float xs[RC * CT];
    static_assert(W1_G * H * CT <= RC * H, "the row groups' sums fit the staged rows");
    const int t = threadIdx.x, k0 = blockIdx.x * CT;
    const long per = (n + gridDim.y - 1) / gridDim.y;
    const long lo = blockIdx.y * per, hi = lo + per < n ? lo + per : n;
    float4 rd[ND];
    float rx[NX];
    auto fetch = [&](long b) {
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const int e = t + i * NTH;
            const long r = b + (e >> 4);
            rd[i] = r < hi ? *reinterpret_cast<const float4*>(dH1 + r * H + (e & 15) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < NX; ++i) {
            const int e = t + i * NTH, k = k0 + (e & (CT - 1));
            const long r = b + e / CT;
            rx[i] = (r < hi && k < K) ? X[(long)(idx ? idx[r] : r) * K + k] : 0.f;
        }
    };
    const int g = t >> 6, og = (t & 63) >> 3, kg = t & 7;   // row group, 8 outputs, 2 columns
    float acc[8][2];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0.f;
    fetch(lo);
    for (long b = lo; b < hi; b += RC) {
#pragma unroll
        for (int i = 0; i < ND; ++i) reinterpret_cast<float4*>(ds)[t + i * NTH] = rd[i];
#pragma unroll
        for (int i = 0; i < NX; ++i) xs[t + i * NTH] = rx[i];
        __syncthreads();
        if (b + RC < hi) fetch(b + RC);
        const int rows = hi - b < RC ? (int)(hi - b) : RC;
#pragma unroll 4
        for (int r = g; r < rows; r += W1_G) {
            const float4 a = *reinterpret_cast<const float4*>(ds + r * H + og * 8);
            const float4 c = *reinterpret_cast<const float4*>(ds + r * H + og * 8 + 4);
            const float2 x = *reinterpret_cast<const float2*>(xs + r * CT + kg * 2);
            const float d[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                acc[i][0] = fmaf(d[i], x.x, acc[i][0]);
                acc[i][1] = fmaf(d[i], x.y, acc[i][1]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        ds[(g * H + og * 8 + i) * CT + kg * 2] = acc[i][0];
        ds[(g * H + og * 8 + i) * CT + kg * 2 + 1] = acc[i][1];
    }
    __syncthreads();
    for (int e = t; e < H * CT; e += NTH) {
        const int k = k0 + (e & (CT - 1));
        float sum = ds[e];
#pragma unroll
        for (int q = 1; q < W1_G; ++q) sum += ds[q * H * CT + e];
        if (k < K) part[((long)blockIdx.y * H + e / CT) * K + k] = sum;
    }
}

struct AdamStep {
    float* w;               // nullptr: gradient only
    float* m;
    float* v;
    float lr, c1, c2;
};

// One thread per weight adds its parts in order; the thread past the weights
// adds the loss (scaled; onto *loss where `add`).
__global__ void __launch_bounds__(256) k_gradsum(int K, const float* __restrict__ p1, int s1,
                                                 const float* __restrict__ p2, int s2, float* __restrict__ gr,
                                                 float* loss, float scale, int add, AdamStep a) {
    const int n1 = MLP_H * K;
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n1 + SMALL_L) return;
    const bool first = i < n1;
    const float* p = first ? p1 + i : p2 + (i - n1);
    const int cnt = first ? s1 : s2, step = first ? n1 : SMALL_L;
    float g = 0.f;
#pragma unroll 8
    for (int q = 0; q < cnt; ++q) g += p[(long)q * step];
    if (i == n1 + SMALL) {
        if (loss) loss[0] = add ? loss[0] + g * scale : g * scale;
        return;
    }
    if (gr) gr[i] = g;
    if (a.w) {
        const float mi = 0.9f * a.m[i] + 0.1f * g;
        const float vi = 0.999f * a.v[i] + 0.001f * g * g;
        a.m[i] = mi;
        a.v[i] = vi;
        a.w[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + 1e-8f);
    }
}

// minibatch rows of an epoch: an affine permutation r -> (a r + b) mod n
__global__ void k_perm(int* idx, long n, long a, long b) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i < n) idx[i] = (int)((a * i + b) % n);
}

struct Dev {
    std::vector<void*> p;
    const amr_options_t* opt;
    ~Dev() {
        for (void* q : p) {
            if (opt && opt->dev_free) opt->dev_free(q, opt->user);
            else if (!(opt && opt->dev_alloc)) cudaFree(q);
        }
    }
    template <typename T> T* get(size_t n) {
        void* q = nullptr;
        const size_t bytes = (n * sizeof(T) + 255) / 256 * 256;
        if (opt && opt->dev_alloc) q = opt->dev_alloc(bytes, opt->user);
        else if (cudaMalloc(&q, bytes) != cudaSuccess) q = nullptr;
        if (q) p.push_back(q);
        return reinterpret_cast<T*>(q);
    }
};

cudaStream_t stream_of(const amr_options_t* o) { return o ? reinterpret_cast<cudaStream_t>(o->stream) : nullptr; }

int blocks(long n, int b = 256) { return (int)((n + b - 1) / b); }

// Scratch of a gradient over n rows, in floats: dH1, the clusters' parts of
// k_rows, the splits' parts of k_w1grad
struct GradScratch {
    float *dH1, *small, *w1;
    static constexpr size_t SMALL_PARTS = (size_t)ROWS_MAXCL * SMALL_L;
    static constexpr size_t floats(long n) { return ((size_t)n * MLP_H + 3) / 4 * 4 + SMALL_PARTS + W1_PARTS; }
    GradScratch(float* base, long n) {
        dH1 = base;
        small = base + ((size_t)n * MLP_H + 3) / 4 * 4;
        w1 = small + SMALL_PARTS;
    }
};

// one forward + backward pass over `n` rows; gradient to g (flat layout; may
// be null), loss times loss_scale to *loss (added to it where `add`; may be null)
template <int D>
int fwd_bwd_d(const float* X, const int* idx, const float* y, long n, float pw, const float* w, float* g, float* loss,
              float loss_scale, int add, const GradScratch& sc, const AdamStep& adam, cudaStream_t s) {
    constexpr int K = mlp_kin(D);
    static_assert(w1_splits(K) >= 1 && w1_splits(K) * MLP_H * K <= W1_PARTS, "the parts fit");
    // rows per tile: the fewest that a launch of 128 blocks covers in one pass
    // (a block's time is its W1 stream, then its rows); 16 beyond
    const int R = n <= 4 * ROWS_CL * ROWS_MAXCL ? 4 : (n <= 8 * ROWS_CL * ROWS_MAXCL ? 8 : 16);
    const long tiles = (n + R - 1) / R;
    const int ncl = (int)std::min<long>((tiles + ROWS_CL - 1) / ROWS_CL, ROWS_MAXCL);
    const int grid = ncl * ROWS_CL;
    if (R == 4) k_rows<D, 4><<<grid, ROWS_NTH, 0, s>>>(X, idx, y, n, pw, w, sc.dH1, sc.small);
    else if (R == 8) k_rows<D, 8><<<grid, ROWS_NTH, 0, s>>>(X, idx, y, n, pw, w, sc.dH1, sc.small);
    else k_rows<D, 16><<<grid, ROWS_NTH, 0, s>>>(X, idx, y, n, pw, w, sc.dH1, sc.small);
    const int splits = (int)std::min<long>(w1_splits(K), (n + 63) / 64);
    k_w1grad<D><<<dim3(w1_tiles(K), splits), W1_NTH, 0, s>>>(sc.dH1, X, idx, n, sc.w1);
    k_gradsum<<<(MLP_H * K + SMALL_L + 255) / 256, 256, 0, s>>>(K, sc.w1, splits, sc.small, ncl, g, loss, loss_scale,
                                                                add, adam);
    return cudaGetLastError() == cudaSuccess ? AMR_OK : AMR_ERR_CUDA;
}

int fwd_bwd(int D, const float* X, const int* idx, const float* y, long n, float pw, const float* w, float* g,
            float* loss, float loss_scale, int add, const GradScratch& sc, const AdamStep& adam, cudaStream_t s) {
    switch (D) {
    case 1: return fwd_bwd_d<1>(X, idx, y, n, pw, w, g, loss, loss_scale, add, sc, adam, s);
    case 2: return fwd_bwd_d<2>(X, idx, y, n, pw, w, g, loss, loss_scale, add, sc, adam, s);
    default: return fwd_bwd_d<3>(X, idx, y, n, pw, w, g, loss, loss_scale, add, sc, adam, s);
    }
}

template <int D>
cudaError_t launch_infer(const float* X, long n, const float* w, float* z, int* err, cudaStream_t s) {
    const size_t smem = InferLayout<D>::TOTAL;
    cudaError_t e = cudaFuncSetAttribute(k_infer<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long tiles = (n + TC_M - 1) / TC_M;
    const int grid = (int)std::min<long>(tiles, (long)nsm);
    k_infer<D><<<grid, 512, smem, s>>>(X, n, w, z, err);
    return cudaGetLastError();
}

}  // namespace

extern "C" {

int amr_mlp_k(int dim) { return (dim >= 1 && dim <= 3) ? mlp_kin(dim) : AMR_ERR_ARG; }

int amr_mlp_features(int dim, double gamma, const double* samples, long n, float* X, const amr_options_t* opt) {
    if (dim < 1 || dim > 3 || !samples || !X || n <= 0) return AMR_ERR_ARG;
    cudaStream_t s = stream_of(opt);
    Dev dv{{}, opt};
    const long rows = n * 2 * dim;
    const int K = mlp_kin(dim);
    double* ds = dv.get<double>(n * 15);
    float* dx = dv.get<float>(rows * K);
    if (!ds || !dx) return AMR_ERR_CUDA;
    if (cudaMemcpyAsync(ds, samples, n * 15 * sizeof(double), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return AMR_ERR_CUDA;
    k_features<<<(int)std::min<long>(blocks(rows * K), 65536), 256, 0, s>>>(dim, gamma, ds, n, dx);
    if (cudaGetLastError() != cudaSuccess) return AMR_ERR_CUDA;
    if (cudaMemcpyAsync(X, dx, rows * K * sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess) return AMR_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? AMR_OK : AMR_ERR_CUDA;
}

int amr_mlp_infer(int dim, const float* X, long n, const float* weights, float* logits, const amr_options_t* opt) {
    if (dim < 1 || dim > 3 || !X || !weights || !logits || n <= 0) return AMR_ERR_ARG;
    cudaStream_t s = stream_of(opt);
    Dev dv{{}, opt};
    const int K = mlp_kin(dim);
    const long nw = mlp_n_weights(dim);
    float* dx = dv.get<float>(n * K);
    float* dw = dv.get<float>(nw);
    float* dz = dv.get<float>(n);
    int* derr = dv.get<int>(1);
    if (!dx || !dw || !dz || !derr) return AMR_ERR_CUDA;
    cudaMemcpyAsync(dx, X, n * K * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dw, weights, nw * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(dz, 0xFF, n * sizeof(float), s);           // NaN until written
    cudaMemsetAsync(derr, 0, sizeof(int), s);
    cudaError_t e = dim == 1 ? launch_infer<1>(dx, n, dw, dz, derr, s)
                  : dim == 2 ? launch_infer<2>(dx, n, dw, dz, derr, s) : launch_infer<3>(dx, n, dw, dz, derr, s);
    if (e != cudaSuccess) return AMR_ERR_CUDA;
    int herr = 0;
    cudaMemcpyAsync(logits, dz, n * sizeof(float), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(&herr, derr, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) return AMR_ERR_CUDA;
    return herr ? AMR_ERR_TIMEOUT : AMR_OK;
}

int amr_mlp_grad(int dim, const float* X, const float* y, long n, float pw, const float* weights, float* grad,
                 float* loss, const amr_options_t* opt) {
    if (dim < 1 || dim > 3 || !X || !y || !weights || !grad || n <= 0 || n > (1 << 24)) return AMR_ERR_ARG;
    cudaStream_t s = stream_of(opt);
    Dev dv{{}, opt};
    const int K = mlp_kin(dim);
    const long nw = mlp_n_weights(dim);
    float* dx = dv.get<float>(n * K);
    float* dy = dv.get<float>(n);
    float* dw = dv.get<float>(nw);
    float* dg = dv.get<float>(nw);
    float* scr = dv.get<float>(GradScratch::floats(n));
    float* la = dv.get<float>(1);
    if (!dx || !dy || !dw || !dg || !scr || !la) return AMR_ERR_CUDA;
    cudaMemcpyAsync(dx, X, n * K * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dy, y, n * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dw, weights, nw * sizeof(float), cudaMemcpyHostToDevice, s);
    if (fwd_bwd(dim, dx, nullptr, dy, n, pw, dw, dg, la, 1.0f / (float)n, 0, GradScratch(scr, n), AdamStep{}, s))
        return AMR_ERR_CUDA;
    cudaMemcpyAsync(grad, dg, nw * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (loss) cudaMemcpyAsync(loss, la, sizeof(float), cudaMemcpyDeviceToHost, s);
    return cudaStreamSynchronize(s) == cudaSuccess ? AMR_OK : AMR_ERR_CUDA;
}

int amr_mlp_train(int dim, const float* X, const float* y, long n, float pw, int epochs, int batch, float lr,
                  uint64_t seed, float* weights, float* loss_hist, const amr_options_t* opt) {
    if (dim < 1 || dim > 3 || !X || !y || !weights || n <= 0 || epochs <= 0 || batch <= 0 || n > (1L << 30))
        return AMR_ERR_ARG;
    cudaStream_t s = stream_of(opt);
    Dev dv{{}, opt};
    const int K = mlp_kin(dim);
    const long nw = mlp_n_weights(dim);
    const int B = (int)std::min<long>(batch, n);
    float* dx = dv.get<float>(n * K);
    float* dy = dv.get<float>(n);
    float* dw = dv.get<float>(nw);
    float* m = dv.get<float>(nw);
    float* v = dv.get<float>(nw);
    int* idx = dv.get<int>(n);
    float* scr = dv.get<float>(GradScratch::floats(B));
    float* la = dv.get<float>(epochs);
    if (!dx || !dy || !dw || !m || !v || !idx || !scr || !la) return AMR_ERR_CUDA;
    const GradScratch sc(scr, B);
    cudaMemcpyAsync(dx, X, n * K * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dy, y, n * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dw, weights, nw * sizeof(float), cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(m, 0, nw * sizeof(float), s);
    cudaMemsetAsync(v, 0, nw * sizeof(float), s);
    cudaMemsetAsync(la, 0, epochs * sizeof(float), s);
    long step = 0;
    const long nb = n / B;            // full minibatches per epoch
    for (int ep = 0; ep < epochs; ++ep) {
        // affine permutation with a multiplier coprime to n, from a SplitMix64 stream
        uint64_t z = seed + (uint64_t)(ep + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        long a = (long)(z % (uint64_t)n) | 1;
        auto gcd = [](long p, long q) { while (q) { long r = p % q; p = q; q = r; } return p; };
        while (gcd(a, n) != 1) a += 2;
        const long b = (long)((z >> 32) % (uint64_t)n);
        k_perm<<<blocks(n), 256, 0, s>>>(idx, n, a % n, b);
        for (long bi = 0; bi < nb; ++bi) {
            ++step;
            const AdamStep adam{dw, m, v, lr, 1.f - powf(0.9f, (float)step), 1.f - powf(0.999f, (float)step)};
            if (fwd_bwd(dim, dx, idx + bi * B, dy, B, pw, dw, nullptr, la + ep, 1.0f / (float)(B * nb), 1, sc, adam, s))
                return AMR_ERR_CUDA;
        }
    }
    if (cudaGetLastError() != cudaSuccess) return AMR_ERR_CUDA;
    cudaMemcpyAsync(weights, dw, nw * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (loss_hist) cudaMemcpyAsync(loss_hist, la, epochs * sizeof(float), cudaMemcpyDeviceToHost, s);
    return cudaStreamSynchronize(s) == cudaSuccess ? AMR_OK : AMR_ERR_CUDA;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free gradient: amr_mlp_grad_noalloc.
//
// Some callers cannot allocate device memory: code running inside a task-based
// runtime that owns the whole device memory (a task there only gets the
// buffers the runtime maps for it, and an allocation behind the runtime's back
// can fail or fragment its pool), code issuing work while a CUDA stream
// capture is in progress (allocation is not allowed there), and real-time
// loops where an allocation may synchronise the device. For them the scratch
// of the forward/backward pass lives in the fixed array below, which every GPU
// that loads this library holds until the process exits: GradScratch of 2048
// rows (2048 x 64 + 32 x 4290 + 160000 floats, about 1.7 MB).
// ---------------------------------------------------------------------------
namespace {
constexpr long NOALLOC_ROWS = AMR_MLP_NOALLOC_MAX_ROWS;
constexpr size_t NOALLOC_FLOATS = GradScratch::floats(NOALLOC_ROWS);
}  // namespace

static __device__ __align__(256) float g_noalloc_scratch[NOALLOC_FLOATS];

namespace {
std::mutex g_noalloc_mu;
constexpr int NOALLOC_MAX_DEVICES = 64;
float* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of the scratch array on device `dev` (current). In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device with cudaGetSymbolAddress and cached.
float* noalloc_scratch(int dev) {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (dev >= 0 && dev < NOALLOC_MAX_DEVICES && g_noalloc_ptr[dev]) return g_noalloc_ptr[dev];
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return nullptr;
    if (dev >= 0 && dev < NOALLOC_MAX_DEVICES) g_noalloc_ptr[dev] = reinterpret_cast<float*>(p);
    return reinterpret_cast<float*>(p);
}
}  // namespace

extern "C" int amr_mlp_grad_noalloc(int dim, const float* X, const float* y, long n, float pos_weight,
                                    const float* weights, float* grad, float* loss, void* stream) {
    if (dim < 1 || dim > 3 || !X || !y || !weights || !grad || !loss || n <= 0) return AMR_ERR_ARG;
    if (n > AMR_MLP_NOALLOC_MAX_ROWS) return AMR_ERR_ARG;      // beyond the fixed scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return AMR_ERR_CUDA;
    float* base = noalloc_scratch(dev);
    if (!base) return AMR_ERR_CUDA;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return fwd_bwd(dim, X, nullptr, y, n, pos_weight, weights, grad, loss, 1.0f / (float)n, 0, GradScratch(base, n),
                   AdamStep{}, s);
}
