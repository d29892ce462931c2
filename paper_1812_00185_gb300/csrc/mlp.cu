// Learned initial guess for the coarse Poisson solve (not in the paper): a per-vertex MLP
// on the pressure-increment mesh with 1-ring mean aggregation, 3 layers, widths
// 4 -> 64 -> 64 -> 1, bfloat16 weights with FP32 arithmetic, FP32 master weights and Adam.
//
//   f_i   = (r_i / s_r, q_i / s_q, x_i, y_i)       r: coarse rhs, q: previous Phi_c, s: RMS
//   a_l,i = W_l [h_{l-1,i}; mean_{j in N(i), j != i} h_{l-1,j}] + b_l,   h_l = relu(a_l) (l < 3)
//   Phi0_i = q_i + s_q * a_3,i
//   loss  = mean over samples and vertices of (a_3,i - clip((Phi*_i - q_i) / s_q, -10, 10))^2
//           (the clip keeps transient steps, where Phi changes by many times its own size,
//           from dominating the fit; there the residual judge falls back to q anyway)
//
// Activations are stored feature-major per sample ([sample][feature][vertex]) so that a
// warp's 32 vertices read consecutive addresses.  Weight gradients are reduced in two
// deterministic passes (per-block partials, then a fixed-order sum).
#include <cuda_bf16.h>

#include <algorithm>

#include "flows.cuh"
#include "mlp.cuh"
#include "solver.cuh"

namespace cgp {

// ---------------------------------------------------------------- forward kernels
// per-sample RMS of r and q: kScaleBlocks blocks per sample write partial sums of squares,
// then one warp per sample adds them in block order (deterministic)
__global__ void __launch_bounds__(kBlock) k_mlp_scales(int n, const double* __restrict__ r, const double* __restrict__ q,
                                                     double* __restrict__ spart) {
    const int b = blockIdx.y;
    double a0 = 0.0, a1 = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double rv = r[(size_t)b * n + i], qv = q[(size_t)b * n + i];
        a0 += rv * rv;
        a1 += qv * qv;
    }
    __shared__ double sm[kBlock / 32][2];
    a0 = warp_sum(a0);
    a1 = warp_sum(a1);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sm[wid][0] = a0;
        sm[wid][1] = a1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            s0 += sm[w][0];
            s1 += sm[w][1];
        }
        spart[((size_t)b * gridDim.x + blockIdx.x) * 2] = s0;
        spart[((size_t)b * gridDim.x + blockIdx.x) * 2 + 1] = s1;
    }
}

__global__ void k_mlp_scales_fin(int n, int nblk, const double* __restrict__ spart, float* __restrict__ scale) {
    const int b = blockIdx.x, lane = threadIdx.x;
    double s0 = 0.0, s1 = 0.0;
    for (int k = lane; k < nblk; k += 32) {
        s0 += spart[((size_t)b * nblk + k) * 2];
        s1 += spart[((size_t)b * nblk + k) * 2 + 1];
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane == 0) {
        const double sr = sqrt(s0 / n), sq = sqrt(s1 / n);
        scale[2 * b] = sr > 0.0 ? (float)sr : 1.0f;
        scale[2 * b + 1] = sq > 0.0 ? (float)sq : 1.0f;
    }
}

__global__ void k_mlp_features(int n, int batch, const double* __restrict__ r, const double* __restrict__ q,
                               const double* __restrict__ xy, const float* __restrict__ scale, float* __restrict__ h0) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * batch) return;
    const int b = (int)(t / n), i = (int)(t % n);
    float* o = h0 + (size_t)b * 4 * n;
    o[i] = (float)(r[t] / (double)scale[2 * b]);
    o[n + i] = (float)(q[t] / (double)scale[2 * b + 1]);
    o[2 * n + i] = (float)xy[2 * i];
    o[3 * n + i] = (float)xy[2 * i + 1];
}

// m[b][f][i] = mean over the 1-ring (i excluded) of act(h[b][f][j]); act = relu if RELU
template <int F, bool RELU>
__global__ void k_mlp_nmean(int n, int batch, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                            const float* __restrict__ h, float* __restrict__ m) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * batch) return;
    const int b = (int)(t / n), i = (int)(t % n);
    const float* hb = h + (size_t)b * F * n;
    float* mb = m + (size_t)b * F * n;
    float acc[F];
#pragma unroll
    for (int f = 0; f < F; ++f) acc[f] = 0.0f;
    int deg = 0;
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int j = col[e];
        if (j == i) continue;
        ++deg;
#pragma unroll
        for (int f = 0; f < F; ++f) {
            float v = hb[(size_t)f * n + j];
            acc[f] += RELU ? fmaxf(v, 0.0f) : v;
        }
    }
    const float inv = deg ? 1.0f / deg : 0.0f;
#pragma unroll
    for (int f = 0; f < F; ++f) mb[(size_t)f * n + i] = acc[f] * inv;
}

// The 64-wide 1-ring means read vertex-major: a feature-major gather reads one 4-byte value
// per 32-byte sector for each (neighbour, feature); a vertex-major one reads each neighbour's
// 64 features as one 256-byte run.  The dense layer that produces the features also writes
// this copy, hv[b][i][f] = relu(a[b][f][i]).
// Sum over the 1-ring of vertex i (i excluded, CSR order) of the vertex-major rows vb[j], two
// features per lane; a warp per vertex.  The lanes hold the ring's indices, so eight rows are
// in flight at a time instead of one row after each index.
__device__ __forceinline__ int ring_sum64(int i, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                          const float2* __restrict__ vb, int lane, float& ax, float& ay) {
    const int rb = rowptr[i], cnt = rowptr[i + 1] - rb;
    int deg = 0;
    for (int e0 = 0; e0 < cnt; e0 += 32) {
        const int m = min(32, cnt - e0), c = lane < m ? col[rb + e0 + lane] : i;
        deg += __popc(__ballot_sync(0xffffffffu, c != i));
        for (int e = 0; e < m; e += 8) {
            float2 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = __shfl_sync(0xffffffffu, c, (e + u) & 31);
                x[u] = make_float2(0.0f, 0.0f);
                if (e + u < m && j != i) x[u] = vb[(size_t)j * (kHid / 2) + lane];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                ax += x[u].x;
                ay += x[u].y;
            }
        }
    }
    return deg;
}

// m[b][f][i] = mean over the 1-ring (i excluded) of hv[b][j][f] for 32 vertices per block: a
// warp per vertex (neighbours in CSR order as in k_mlp_nmean), written back feature-major
// through shared memory
__global__ void __launch_bounds__(256) k_mlp_nmean64(int n, const int32_t* __restrict__ rowptr,
                                                    const int32_t* __restrict__ col, const float* __restrict__ hv,
                                                    float* __restrict__ m) {
    static_assert(kHid == 64, "two features per lane");
    __shared__ float tile[kHid][33];
    const int b = blockIdx.y, i0 = blockIdx.x * 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float2* vb = reinterpret_cast<const float2*>(hv + (size_t)b * n * kHid);
    for (int v = wid; v < 32; v += 8) {
        const int i = i0 + v;
        float ax = 0.0f, ay = 0.0f;
        const int deg = i < n ? ring_sum64(i, rowptr, col, vb, lane, ax, ay) : 0;
        const float inv = deg ? 1.0f / deg : 0.0f;
        tile[2 * lane][v] = ax * inv;
        tile[2 * lane + 1][v] = ay * inv;
    }
    __syncthreads();
    float* mb = m + (size_t)b * kHid * n;
    for (int f = wid; f < kHid; f += 8) {
        const int i = i0 + lane;
        if (i < n) mb[(size_t)f * n + i] = tile[f][lane];
    }
}

// Its transpose, fused with the ReLU's: gh[b][f][j] += sum over the neighbours i of j of
// gv[b][i][f] (vertex-major, already divided by i's degree), then gh = 0 where a_prev <= 0.
// (A feature-major gather of gm read one 4-byte value per 32-byte sector.)
__global__ void __launch_bounds__(256) k_mlp_nmean64_bwd(int n, const int32_t* __restrict__ rowptr,
                                                        const int32_t* __restrict__ col, const float* __restrict__ gv,
                                                        const float* __restrict__ a_prev, float* __restrict__ gh) {
    __shared__ float tile[kHid][33];
    const int b = blockIdx.y, i0 = blockIdx.x * 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float2* vb = reinterpret_cast<const float2*>(gv + (size_t)b * n * kHid);
    for (int v = wid; v < 32; v += 8) {
        const int i = i0 + v;
        float ax = 0.0f, ay = 0.0f;
        if (i < n) ring_sum64(i, rowptr, col, vb, lane, ax, ay);
        tile[2 * lane][v] = ax;
        tile[2 * lane + 1][v] = ay;
    }
    __syncthreads();
    const size_t o = (size_t)b * kHid * n + i0 + lane;
    if (i0 + lane < n)
#pragma unroll
        for (int f = wid; f < kHid; f += 8) {
            const size_t at = o + (size_t)f * n;
            gh[at] = a_prev[at] > 0.0f ? gh[at] + tile[f][lane] : 0.0f;
        }
}

// a[b][o][i] = sum_k W[o][k] x_k + bias[o], x = [act(h); m] (2*FIN inputs), summed in k
// order; with VOUT also hv[b][i][o] = relu(a[b][o][i]) (the vertex-major copy the next
// 1-ring mean gathers).  W (bf16, row-major FOUT x 2*FIN) is staged per block as FP32
// columns wt[k][o]: lane l of a warp loads 8 consecutive k of row o = l (16 bytes) and
// writes them down column l, so the transposed writes are free of bank conflicts.
// Two threads share a vertex (the first half of the block takes outputs
// [0, FOUT/2), the second half the rest, so a warp reads one wt row as a broadcast), and each
// thread has two vertices, so a weight read from shared memory feeds two FMAs (one read per
// FMA held the kernel at the shared-memory pipe's rate).  Each thread loads its inputs in
// chunks, the next chunk while it multiplies the current one, so the latency of the
// feature-major input loads overlaps the FMAs.
constexpr int kDenseVertices = 128;   // per block of 128 threads

template <int FIN, int FOUT, bool RELU_IN, bool VOUT>
__global__ void __launch_bounds__(128) k_mlp_dense(int n, int batch, const __nv_bfloat16* __restrict__ W,
                                                   const float* __restrict__ bias, const float* __restrict__ h,
                                                   const float* __restrict__ m, float* __restrict__ a,
                                                   float* __restrict__ hv) {
    constexpr int K = 2 * FIN;
    constexpr int OS = 2;                               // threads per vertex
    constexpr int V = OS * kDenseVertices / 128;        // vertices per thread
    constexpr int FO = FOUT / OS;                       // outputs per thread
    constexpr int LD = FOUT + 4;                        // row stride of wt (16-byte rows)
    constexpr int KC = FIN < 8 ? FIN : 8;               // inputs loaded per chunk
    constexpr int NV8 = K * FOUT / 8;                   // 16-byte pieces of W
    static_assert(FOUT % OS == 0 && FO % 4 == 0 && FIN % KC == 0 && K % 8 == 0, "dense layer shape");
    __shared__ __align__(16) float wt[K][LD];
    const uint4* W8 = reinterpret_cast<const uint4*>(W);
#pragma unroll
    for (int r = 0; r < (NV8 + 127) / 128; ++r) {
        const int f = threadIdx.x + 128 * r;
        if (f < NV8) {
            const int o = f % FOUT, k0 = 8 * (f / FOUT);
            const uint4 u = __ldg(W8 + (o * K + k0) / 8);
            const uint32_t wd[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 w2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&wd[j]));
                wt[k0 + 2 * j][o] = w2.x;
                wt[k0 + 2 * j + 1][o] = w2.y;
            }
        }
    }
    __syncthreads();
    constexpr int TV = 128 / OS;                        // threads over the vertices
    const int part = threadIdx.x / TV;
    const int o0 = part * FO;
    int b[V], i[V];
    bool in[V];
    const float *hb[V], *mb[V];
    float acc[V][FO];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int64_t t = blockIdx.x * (int64_t)kDenseVertices + threadIdx.x % TV + v * TV;
        in[v] = t < (int64_t)n * batch;
        b[v] = in[v] ? (int)(t / n) : 0;
        i[v] = in[v] ? (int)(t % n) : 0;
        hb[v] = h + (size_t)b[v] * FIN * n + i[v];
        mb[v] = m + (size_t)b[v] * FIN * n + i[v];
#pragma unroll
        for (int o = 0; o < FO; ++o) acc[v][o] = bias[o0 + o];
    }
    // chunk c holds inputs k = c KC .. c KC + KC - 1: the first FIN / KC chunks come from h
    // (with the ReLU when RELU_IN), the rest from m; two register buffers alternate, so the
    // loads of chunk c + 1 are in flight while chunk c is multiplied
    constexpr int NCH = K / KC;
    static_assert(NCH % 2 == 0, "chunks come in pairs");
    auto load = [&](float (&xs)[V][KC], int c) {
        const bool from_h = c < FIN / KC;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float* src = from_h ? hb[v] + (size_t)c * KC * n : mb[v] + (size_t)(c - FIN / KC) * KC * n;
#pragma unroll
            for (int u = 0; u < KC; ++u) {
                const float x = src[(size_t)u * n];
                xs[v][u] = (RELU_IN && from_h) ? fmaxf(x, 0.0f) : x;
            }
        }
    };
    auto mul = [&](const float (&xs)[V][KC], int c) {
#pragma unroll
        for (int u = 0; u < KC; ++u) {
            const float* wr = &wt[c * KC + u][o0];
#pragma unroll
            for (int o = 0; o < FO; o += 4) {
                const float4 w4 = *reinterpret_cast<const float4*>(wr + o);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    acc[v][o] += w4.x * xs[v][u];
                    acc[v][o + 1] += w4.y * xs[v][u];
                    acc[v][o + 2] += w4.z * xs[v][u];
                    acc[v][o + 3] += w4.w * xs[v][u];
                }
            }
        }
    };
    float xa[V][KC], xb[V][KC];
    load(xa, 0);
    for (int c = 0; c < NCH; c += 2) {
        load(xb, c + 1);
        mul(xa, c);
        if (c + 2 < NCH) load(xa, c + 2);
        mul(xb, c + 1);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if (!in[v]) continue;
        float* ab = a + (size_t)b[v] * FOUT * n;
#pragma unroll
        for (int o = 0; o < FO; ++o) ab[(size_t)(o0 + o) * n + i[v]] = acc[v][o];
        if constexpr (VOUT) {
            float4* vr = reinterpret_cast<float4*>(hv + ((size_t)b[v] * n + i[v]) * FOUT + o0);
#pragma unroll
            for (int o = 0; o < FO; o += 4)
                vr[o / 4] = make_float4(fmaxf(acc[v][o], 0.0f), fmaxf(acc[v][o + 1], 0.0f), fmaxf(acc[v][o + 2], 0.0f),
                                        fmaxf(acc[v][o + 3], 0.0f));
        }
    }
}

// ---------------------------------------------------------------- backward kernels
constexpr double kTargetClip = 10.0;

// ---- layer 3 (one output) in training.  Its 1-ring mean commutes with the weights, so no
// 64-wide mean is formed: with p = W3h . h2 and z = W3m . h2 per vertex,
//   a3_i = b3 + p_i + mean_{j in N(i)} z_j,
// and with g3 = dL/da3 and S_j = sum over the neighbours i of j of g3_i / deg(i),
//   dL/dh2_j = W3h g3_j + W3m S_j,  dW3h = sum_j g3_j h2_j,  dW3m = sum_j S_j h2_j.
// (The mean, its transpose and the products over it read and wrote 64 values per vertex eight
// times: 620 us of a step of 32,489 vertices and 8 samples; these four kernels take about 90.)
__global__ void __launch_bounds__(kBlock) k_mlp_l3_pz(int n, int batch, const __nv_bfloat16* __restrict__ W,
                                                     const float* __restrict__ a2, float2* __restrict__ pz) {
    __shared__ float2 w[kHid];
    if (threadIdx.x < kHid)
        w[threadIdx.x] = make_float2(__bfloat162float(W[threadIdx.x]), __bfloat162float(W[kHid + threadIdx.x]));
    __syncthreads();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * batch) return;
    const float* ab = a2 + (size_t)(t / n) * kHid * n + t % n;
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll 16
    for (int f = 0; f < kHid; ++f) {
        const float v = fmaxf(ab[(size_t)f * n], 0.0f);
        s.x += w[f].x * v;
        s.y += w[f].y * v;
    }
    pz[t] = s;
}

// a3 from p and z, g3 = dL/da3 = 2 (a3 - clip((t - q)/s_q)) / (n * batch); loss partials per block
__global__ void __launch_bounds__(kBlock) k_mlp_loss(int n, int batch, const int32_t* __restrict__ rowptr,
                                                   const int32_t* __restrict__ col, const float* __restrict__ bias,
                                                   const float2* __restrict__ pz, const double* __restrict__ q,
                                                   const double* __restrict__ tgt, const float* __restrict__ scale,
                                                   float* __restrict__ g3, double* __restrict__ partials,
                                                   unsigned int* ticket, float* __restrict__ loss) {
    double acc[1] = {0.0};
    const int64_t total = (int64_t)n * batch;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(t / n), i = (int)(t % n);
        float z = 0.0f;
        int deg = 0;
        for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
            const int j = col[e];
            if (j == i) continue;
            ++deg;
            z += pz[(size_t)b * n + j].y;
        }
        const float out = bias[0] + pz[t].x + z * (deg ? 1.0f / deg : 0.0f);
        const double tn = fmin(fmax((tgt[t] - q[t]) / (double)scale[2 * b + 1], -kTargetClip), kTargetClip);
        const double d = (double)out - tn;
        acc[0] += d * d;
        g3[t] = (float)(2.0 * d / (double)total);
    }
    double tot[1];
    if (grid_sum<1>(acc, partials, ticket, tot) && threadIdx.x == 0) *loss = (float)(tot[0] / (double)total);
}

// (g3_j, S_j) per vertex and g2 = dL/da2 = (W3h g3 + W3m S) where a2 > 0
__global__ void __launch_bounds__(kBlock) k_mlp_l3_bwd(int n, int batch, const int32_t* __restrict__ rowptr,
                                                      const int32_t* __restrict__ col,
                                                      const __nv_bfloat16* __restrict__ W, const float* __restrict__ g3,
                                                      const float* __restrict__ a2, float2* __restrict__ gs,
                                                      float* __restrict__ g2) {
    __shared__ float2 w[kHid];
    if (threadIdx.x < kHid)
        w[threadIdx.x] = make_float2(__bfloat162float(W[threadIdx.x]), __bfloat162float(W[kHid + threadIdx.x]));
    __syncthreads();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * batch) return;
    const int b = (int)(t / n), j = (int)(t % n);
    const float g = g3[t];
    float s = 0.0f;
    for (int e = rowptr[j]; e < rowptr[j + 1]; ++e) {
        const int i = col[e];
        if (i != j) s += g3[(size_t)b * n + i] * (1.0f / (float)(rowptr[i + 1] - rowptr[i] - 1));
    }
    gs[t] = make_float2(g, s);
    const size_t at = (size_t)b * kHid * n + j;
#pragma unroll 16
    for (int f = 0; f < kHid; ++f) {
        const size_t x = at + (size_t)f * n;
        g2[x] = a2[x] > 0.0f ? w[f].x * g + w[f].y * s : 0.0f;
    }
}

// per-block partials of dW3h, dW3m, db3: blocks of kRowsPerBlock vertices of one sample; a warp
// takes every eighth feature, its lanes the vertices
constexpr int kRowsPerBlock = 1024;

__global__ void __launch_bounds__(256) k_mlp_wgrad3(int n, const float2* __restrict__ gs, const float* __restrict__ a2,
                                                   float* __restrict__ partials) {
    __shared__ float2 g[kRowsPerBlock];
    const int b = blockIdx.y, i0 = blockIdx.x * kRowsPerBlock, cnt = min(kRowsPerBlock, n - i0);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = threadIdx.x; r < kRowsPerBlock; r += 256)
        g[r] = r < cnt ? gs[(size_t)b * n + i0 + r] : make_float2(0.0f, 0.0f);
    __syncthreads();
    float* out = partials + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (2 * kHid + 1);
    for (int f = wid; f < kHid; f += 8) {
        const float* ab = a2 + ((size_t)b * kHid + f) * n + i0;
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll 8
        for (int r = lane; r < kRowsPerBlock; r += 32) {
            const float v = r < cnt ? fmaxf(ab[r], 0.0f) : 0.0f;
            s0 += g[r].x * v;
            s1 += g[r].y * v;
        }
        s0 = warp_sum(s0);
        s1 = warp_sum(s1);
        if (lane == 0) {
            out[f] = s0;
            out[kHid + f] = s1;
        }
    }
    if (wid == 0) {
        float s = 0.0f;
        for (int r = lane; r < kRowsPerBlock; r += 32) s += g[r].x;
        s = warp_sum(s);
        if (lane == 0) out[2 * kHid] = s;
    }
}

// per-block partials of layer 1's 64 x 8 weight gradient and bias, same blocks: the 8 inputs in
// shared memory, a warp takes 8 outputs in two groups of 4, so an input read feeds 4 FMAs
__global__ void __launch_bounds__(256) k_mlp_wgrad1(int n, const float* __restrict__ ga, const float* __restrict__ h,
                                                   const float* __restrict__ m, float* __restrict__ partials) {
    __shared__ float x[8][kRowsPerBlock];
    const int b = blockIdx.y, i0 = blockIdx.x * kRowsPerBlock, cnt = min(kRowsPerBlock, n - i0);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < 8 * kRowsPerBlock; e += 256) {
        const int k = e / kRowsPerBlock, r = e % kRowsPerBlock;
        const float* src = (k < 4 ? h : m) + ((size_t)b * 4 + (k & 3)) * n + i0;
        x[k][r] = r < cnt ? src[r] : 0.0f;
    }
    __syncthreads();
    float* out = partials + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (kHid * 9);
    for (int o0 = 4 * wid; o0 < kHid; o0 += 32) {
        float s[4][9];
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int k = 0; k < 9; ++k) s[o][k] = 0.0f;
        const float* gb = ga + ((size_t)b * kHid + o0) * n + i0;
#pragma unroll 4
        for (int r = lane; r < kRowsPerBlock; r += 32) {
            float g[4];
#pragma unroll
            for (int o = 0; o < 4; ++o) g[o] = r < cnt ? gb[(size_t)o * n + r] : 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float v = x[k][r];
#pragma unroll
                for (int o = 0; o < 4; ++o) s[o][k] += g[o] * v;
            }
#pragma unroll
            for (int o = 0; o < 4; ++o) s[o][8] += g[o];
        }
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const float t = warp_sum(s[o][k]);
                if (lane == 0) out[(o0 + o) * 9 + k] = t;
            }
    }
}

// gx = W^T ga: gh (the h part, k < FIN; feature-major) and gv (the mean part divided by the
// vertex's degree, vertex-major, for k_mlp_nmean64_bwd).  Two vertices per thread, so a weight
// read from shared memory feeds two FMAs.
template <int FIN, int FOUT>
__global__ void __launch_bounds__(128) k_mlp_dense_bwd(int n, int batch, const int32_t* __restrict__ rowptr,
                                                       const __nv_bfloat16* __restrict__ W,
                                                       const float* __restrict__ ga, float* __restrict__ gh,
                                                       float* __restrict__ gv) {
    constexpr int K = 2 * FIN, V = 2, KC = 4;
    static_assert(FIN % KC == 0, "whole chunks");
    __shared__ __align__(16) float w[K][FOUT];
    for (int e = threadIdx.x; e < K * FOUT; e += blockDim.x) {
        const int o = e / K, k = e % K;
        w[k][o] = __bfloat162float(W[e]);
    }
    __syncthreads();
    int b[V], i[V];
    bool in[V];
    float inv[V], g[V][FOUT];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int64_t t = blockIdx.x * (int64_t)(128 * V) + threadIdx.x + 128 * v;
        in[v] = t < (int64_t)n * batch;
        b[v] = in[v] ? (int)(t / n) : 0;
        i[v] = in[v] ? (int)(t % n) : 0;
        inv[v] = 1.0f / (float)(rowptr[i[v] + 1] - rowptr[i[v]] - 1);
#pragma unroll
        for (int o = 0; o < FOUT; ++o) g[v][o] = ga[((size_t)b[v] * FOUT + o) * n + i[v]];
    }
    for (int k0 = 0; k0 < K; k0 += KC) {
        float s[V][KC];
#pragma unroll
        for (int u = 0; u < KC; ++u) {
#pragma unroll
            for (int v = 0; v < V; ++v) s[v][u] = 0.0f;
#pragma unroll
            for (int o = 0; o < FOUT; ++o) {
                const float wv = w[k0 + u][o];
#pragma unroll
                for (int v = 0; v < V; ++v) s[v][u] += wv * g[v][o];
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (!in[v]) continue;
            if (k0 < FIN) {
#pragma unroll
                for (int u = 0; u < KC; ++u) gh[((size_t)b[v] * FIN + k0 + u) * n + i[v]] = s[v][u];
            } else {
                *reinterpret_cast<float4*>(gv + ((size_t)b[v] * n + i[v]) * FIN + (k0 - FIN)) =
                    make_float4(s[v][0] * inv[v], s[v][1] * inv[v], s[v][2] * inv[v], s[v][3] * inv[v]);
            }
        }
    }
}

// Weight gradients are reduced in two deterministic passes: per-block partials [block][o][k]
// (k = 2 FIN: the bias), then a fixed-order sum in FP64.
constexpr int kTile = 32;

// The 64 x 128 weight gradient of layer 2 (and its bias) as a register-tiled product: 256
// threads hold 8 x 4 outputs each (o = og + 8 j, k = kg + 32 j), so 12 16-byte shared-memory
// reads feed 128 FMAs; two CTAs per SM.  Sums of 32 rows are added to the running ones, those of
// at most kRowsPerBlock rows, which keeps the rounding of a two-level sum: beyond kWgradBlocks
// CTAs of that many rows (311,296) there are more CTAs, not longer FP32 sums.  (8.4M rows with 304
// CTAs: equal terms added up to 1.3e-5 off, against 9e-7.)
constexpr int kWgradBlocks = 304;

inline int wgrad64_rows(int64_t rows) {   // rows per CTA, whole tiles
    const int64_t r = (rows + kWgradBlocks - 1) / kWgradBlocks;
    return (int)std::min<int64_t>((r + kTile - 1) / kTile * kTile, kRowsPerBlock);
}
inline int wgrad64_blocks(int64_t rows) {
    const int r = wgrad64_rows(rows);
    return (int)((rows + r - 1) / r);
}

__global__ void __launch_bounds__(256, 2) k_mlp_wgrad64(int n, int batch, int rows, const float* __restrict__ ga,
                                                       const float* __restrict__ h, const float* __restrict__ m,
                                                       float* __restrict__ partials) {
    constexpr int K = 2 * kHid, LD = kTile + 4;   // 16-byte rows on distinct banks
    __shared__ __align__(16) float gt[kHid][LD];
    __shared__ __align__(16) float xt[K][LD];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int og = lane & 7, kg = 4 * wid + (lane >> 3);
    float acc[8][4], accb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        accb[j] = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
    }
    const int64_t total = (int64_t)n * batch, r0 = (int64_t)blockIdx.x * rows;
    for (int64_t rt = r0; rt < r0 + rows && rt < total; rt += kTile) {
        const int64_t row = rt + lane;
        const bool in = row < total;
        const int b = in ? (int)(row / n) : 0, i = in ? (int)(row % n) : 0;
        const size_t at = (size_t)b * kHid * n + i;
        float v[24];
#pragma unroll
        for (int u = 0; u < 24; ++u) {
            const int f = wid + 8 * u;   // 0..63: ga, 64..127: h, 128..191: m
            const float* src = u < 8 ? ga : (u < 16 ? h : m);
            v[u] = in ? src[at + (size_t)(f & (kHid - 1)) * n] : 0.0f;
        }
        __syncthreads();   // the previous tile is consumed
#pragma unroll
        for (int u = 0; u < 24; ++u) {
            const int f = wid + 8 * u;
            if (u < 8) gt[f][lane] = v[u];
            else xt[f - kHid][lane] = u < 16 ? fmaxf(v[u], 0.0f) : v[u];
        }
        __syncthreads();
        float s[8][4], sb[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            sb[j] = 0.0f;
#pragma unroll
            for (int q = 0; q < 4; ++q) s[j][q] = 0.0f;
        }
#pragma unroll 1
        for (int r = 0; r < kTile; r += 4) {
            float4 x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = *reinterpret_cast<const float4*>(&xt[kg + 32 * q][r]);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 g = *reinterpret_cast<const float4*>(&gt[og + 8 * j][r]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    s[j][q] += g.x * x[q].x;
                    s[j][q] += g.y * x[q].y;
                    s[j][q] += g.z * x[q].z;
                    s[j][q] += g.w * x[q].w;
                }
                if (wid == 0) sb[j] += (g.x + g.y) + (g.z + g.w);
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            accb[j] += sb[j];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[j][q] += s[j][q];
        }
    }
    float* out = partials + (size_t)blockIdx.x * kHid * (K + 1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int o = og + 8 * j;
#pragma unroll
        for (int q = 0; q < 4; ++q) out[o * (K + 1) + kg + 32 * q] = acc[j][q];
        if (kg == 0) out[o * (K + 1) + K] = accb[j];
    }
}

// grad[W offset + o*K + k] / grad[b offset + o] = sum over blocks (fixed order) of the partials
// (eight threads per output take every eighth block, then their sums are added in order)
__global__ void __launch_bounds__(256) k_mlp_wgrad_reduce(int nblk, int fout, int K, const float* __restrict__ partials,
                                                         float* __restrict__ gW, float* __restrict__ gb) {
    __shared__ double part[8][32];
    const int nout = fout * (K + 1), lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int qi = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (qi < nout)
#pragma unroll 4
        for (int c = grp; c < nblk; c += 8) s += partials[(size_t)c * nout + qi];
    part[grp][lane] = s;
    __syncthreads();
    if (grp || qi >= nout) return;
    for (int k = 1; k < 8; ++k) s += part[k][lane];
    const int o = qi / (K + 1), k = qi % (K + 1);
    if (k < K) gW[o * K + k] = (float)s;
    else gb[o] = (float)s;
}

__global__ void k_mlp_adam(int np, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int t, float lr, __nv_bfloat16* __restrict__ pbf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.0f - powf(b1, (float)t));
    const float vh = vi / (1.0f - powf(b2, (float)t));
    const float pi = p[i] - lr * mh / (sqrtf(vh) + eps);
    p[i] = pi;
    pbf[i] = __float2bfloat16_rn(pi);
}

__global__ void k_mlp_to_bf16(int np, const float* __restrict__ p, __nv_bfloat16* __restrict__ pbf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < np) pbf[i] = __float2bfloat16_rn(p[i]);
}

// ---------------------------------------------------------------- host side
size_t MlpBuffers::bytes(int n, int batch) {
    Carve cv(nullptr);
    MlpBuffers B;
    B.carve(cv, n, batch);
    return cv.off;
}

void MlpBuffers::carve(Carve& cv, int n_, int batch) {
    n = n_;
    maxb = batch;
    const size_t nb = (size_t)n * batch;
    scale = cv.take<float>(2 * (size_t)batch);
    spart = cv.take<double>(2 * (size_t)kScaleBlocks * batch);
    h0 = cv.take<float>(4 * nb);
    m0 = cv.take<float>(4 * nb);
    a1 = cv.take<float>(kHid * nb);
    m1 = cv.take<float>(kHid * nb);
    a2 = cv.take<float>(kHid * nb);
    pz = cv.take<float2>(nb);
    hv = cv.take<float>(kHid * nb);
    params_bf = cv.take<__nv_bfloat16>(kMlpParams);
    params = cv.take<float>(kMlpParams);
}

// the training forward pass up to layer 3's (p, z): every activation kept
// (feature-major) for mlp_backward
static int mlp_forward_train(const MlpBuffers& B, const Level& L, const double* r, const double* q, int batch,
                             cudaStream_t st) {
    const int n = B.n;
    const int64_t nb = (int64_t)n * batch;
    const int g = blocks_for(nb);
    const int gh = blocks_for(nb, kDenseVertices);
    k_mlp_scales<<<dim3(kScaleBlocks, batch), kBlock, 0, st>>>(n, r, q, B.spart);
    k_mlp_scales_fin<<<batch, 32, 0, st>>>(n, kScaleBlocks, B.spart, B.scale);
    k_mlp_features<<<g, kBlock, 0, st>>>(n, batch, r, q, L.xy, B.scale, B.h0);
    k_mlp_nmean<4, false><<<g, kBlock, 0, st>>>(n, batch, L.rowptr, L.col, B.h0, B.m0);
    k_mlp_dense<4, kHid, false, true><<<gh, 128, 0, st>>>(n, batch, B.params_bf + kOffW1, B.params + kOffB1, B.h0,
                                                           B.m0, B.a1, B.hv);
    const dim3 gm((n + 31) / 32, batch);
    k_mlp_nmean64<<<gm, 256, 0, st>>>(n, L.rowptr, L.col, B.hv, B.m1);
    k_mlp_dense<kHid, kHid, true, false><<<gh, 128, 0, st>>>(n, batch, B.params_bf + kOffW2, B.params + kOffB2, B.a1,
                                                              B.m1, B.a2, nullptr);
    k_mlp_l3_pz<<<g, kBlock, 0, st>>>(n, batch, B.params_bf + kOffW3, B.a2, B.pz);
    CGP_LAUNCH_CHECK();
    return CGP_OK;
}

}  // namespace cgp

using namespace cgp;

struct cgp_mlp {
    const cgp_mesh* mesh = nullptr;
    int level = 0;
    MlpBuffers B;
    void* mem = nullptr;          // one cudaMalloc: buffers + training state
    float *grad = nullptr, *adam_m = nullptr, *adam_v = nullptr, *wpart = nullptr;
    float *gA = nullptr, *gB = nullptr, *gM = nullptr, *g3 = nullptr, *loss = nullptr;
    double* partials = nullptr;
    unsigned int* ticket = nullptr;
    int adam_t = 0;
};

extern "C" int cgp_mlp_param_count(void) { return kMlpParams; }

extern "C" int cgp_mlp_create(const cgp_mesh* mesh, int32_t level, int32_t max_batch, cgp_mlp** out) {
    clear_error();
    if (!mesh || !out || level < 0 || level > mesh->n_levels || max_batch < 1) {
        set_error("cgp_mlp_create: bad arguments");
        return CGP_EINVAL;
    }
    *out = nullptr;
    cgp_mlp* m = new cgp_mlp();
    m->mesh = mesh;
    m->level = level;
    const int n = mesh->lev[level].nv;
    const int64_t nb = (int64_t)n * max_batch;
    const size_t nblk = (size_t)((n + kRowsPerBlock - 1) / kRowsPerBlock) * max_batch;   // blocks of layers 1 and 3
    auto layout = [&](Carve& cv) {
        m->B.carve(cv, n, max_batch);
        m->grad = cv.take<float>(kMlpParams);
        m->adam_m = cv.take<float>(kMlpParams);
        m->adam_v = cv.take<float>(kMlpParams);
        m->wpart = cv.take<float>(std::max((size_t)std::max(kWgradBlocks, wgrad64_blocks(nb)) * kHid * (2 * kHid + 1), nblk * kHid * 9));
        m->gA = cv.take<float>(kHid * nb);
        m->gB = cv.take<float>(kHid * nb);
        m->gM = cv.take<float>(kHid * nb);
        m->g3 = cv.take<float>(nb);
        m->loss = cv.take<float>(1);
        m->partials = cv.take<double>(4096);
        m->ticket = cv.take<unsigned int>(4);
    };
    Carve c0(nullptr);
    layout(c0);
    cudaError_t e = cudaMalloc(&m->mem, c0.off + 256);
    if (e != cudaSuccess) {
        set_error("cudaMalloc(%zu) failed: %s", c0.off, cudaGetErrorString(e));
        delete m;
        return CGP_ENOMEM;
    }
    Carve c1((void*)(((uintptr_t)m->mem + 255) & ~(uintptr_t)255));
    layout(c1);
    if (cudaMemset(m->adam_m, 0, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMemset(m->adam_v, 0, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMemset(m->ticket, 0, 4 * sizeof(unsigned int)) != cudaSuccess ||
        cudaMemset(m->B.params, 0, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMemset(m->B.params_bf, 0, sizeof(__nv_bfloat16) * kMlpParams) != cudaSuccess) {
        set_error("cgp_mlp_create: initialisation failed");
        cudaFree(m->mem);
        delete m;
        return CGP_ECUDA;
    }
    {
        const int rc = mlp_infer_setup();
        if (rc != CGP_OK) {
            cudaFree(m->mem);
            delete m;
            return rc;
        }
    }
    *out = m;
    return CGP_OK;
}

extern "C" void cgp_mlp_destroy(cgp_mlp* m) {
    if (!m) return;
    if (m->mem) cudaFree(m->mem);
    delete m;
}

extern "C" int cgp_mlp_set_params(cgp_mlp* m, const float* params, int32_t where, cgp_stream_t stream) {
    clear_error();
    if (!m || !params) {
        set_error("cgp_mlp_set_params: null argument");
        return CGP_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CGP_CUDA(cudaMemcpyAsync(m->B.params, params, sizeof(float) * kMlpParams,
                             where == CGP_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st));
    k_mlp_to_bf16<<<blocks_for(kMlpParams), kBlock, 0, st>>>(kMlpParams, m->B.params, m->B.params_bf);
    CGP_LAUNCH_CHECK();
    CGP_CUDA(cudaMemsetAsync(m->adam_m, 0, sizeof(float) * kMlpParams, st));
    CGP_CUDA(cudaMemsetAsync(m->adam_v, 0, sizeof(float) * kMlpParams, st));
    m->adam_t = 0;
    if (where == CGP_HOST) CGP_CUDA(cudaStreamSynchronize(st));
    return CGP_OK;
}

extern "C" int cgp_mlp_copy_state(cgp_mlp* dst, const cgp_mlp* src, cgp_stream_t stream) {
    clear_error();
    if (!dst || !src) {
        set_error("cgp_mlp_copy_state: null argument");
        return CGP_EINVAL;
    }
    if (dst == src) return CGP_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t fb = sizeof(float) * kMlpParams;
    CGP_CUDA(cudaMemcpyAsync(dst->B.params, src->B.params, fb, cudaMemcpyDeviceToDevice, st));
    CGP_CUDA(cudaMemcpyAsync(dst->B.params_bf, src->B.params_bf, sizeof(__nv_bfloat16) * kMlpParams,
                             cudaMemcpyDeviceToDevice, st));
    CGP_CUDA(cudaMemcpyAsync(dst->adam_m, src->adam_m, fb, cudaMemcpyDeviceToDevice, st));
    CGP_CUDA(cudaMemcpyAsync(dst->adam_v, src->adam_v, fb, cudaMemcpyDeviceToDevice, st));
    dst->adam_t = src->adam_t;
    return CGP_OK;
}

extern "C" int cgp_mlp_get_params(cgp_mlp* m, float* params, int32_t where, cgp_stream_t stream) {
    clear_error();
    if (!m || !params) {
        set_error("cgp_mlp_get_params: null argument");
        return CGP_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CGP_CUDA(cudaMemcpyAsync(params, m->B.params, sizeof(float) * kMlpParams,
                             where == CGP_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
    if (where == CGP_HOST) CGP_CUDA(cudaStreamSynchronize(st));
    return CGP_OK;
}

extern "C" int cgp_mlp_forward(cgp_mlp* m, const double* r, const double* q, int32_t batch, double* pred,
                               cgp_stream_t stream) {
    clear_error();
    if (!m || !r || !q || !pred || batch < 1 || batch > m->B.maxb) {
        set_error("cgp_mlp_forward: bad arguments");
        return CGP_EINVAL;
    }
    return mlp_forward(m->B, m->mesh->lev[m->level], r, q, batch, pred, (cudaStream_t)stream);
}

// loss and gradient (into m->grad); shared by cgp_mlp_grad and cgp_mlp_train_step
static int mlp_backward(cgp_mlp* m, const double* r, const double* q, const double* tgt, int batch,
                        cudaStream_t st) {
    const Level& L = m->mesh->lev[m->level];
    MlpBuffers& B = m->B;
    const int n = B.n;
    const int64_t nb = (int64_t)n * batch;
    CGP_TRY(mlp_forward_train(B, L, r, q, batch, st));
    const int g = blocks_for(nb), g256 = blocks_for(nb, 256);   // two vertices per thread of 128
    const dim3 gm((n + 31) / 32, batch), gw((n + kRowsPerBlock - 1) / kRowsPerBlock, batch);
    const int rows64 = wgrad64_rows(nb), nblk64 = wgrad64_blocks(nb);
    const int nblk = (int)(gw.x * gw.y);
    int gl = (int)(nb / kBlock + 1);
    if (gl > 1024) gl = 1024;
    float2* gs = reinterpret_cast<float2*>(m->gM);   // free until layer 2's mean part
    k_mlp_loss<<<gl, kBlock, 0, st>>>(n, batch, L.rowptr, L.col, B.params + kOffB3, B.pz, q, tgt, B.scale, m->g3,
                                      m->partials, m->ticket, m->loss);
    // layer 3: gA = dL/da2, then dW3, db3
    k_mlp_l3_bwd<<<g, kBlock, 0, st>>>(n, batch, L.rowptr, L.col, B.params_bf + kOffW3, m->g3, B.a2, gs, m->gA);
    k_mlp_wgrad3<<<gw, 256, 0, st>>>(n, gs, B.a2, m->wpart);
    k_mlp_wgrad_reduce<<<blocks_for(2 * kHid + 1, 32), 256, 0, st>>>(nblk, 1, 2 * kHid, m->wpart, m->grad + kOffW3,
                                                                    m->grad + kOffB3);
    // layer 2
    k_mlp_wgrad64<<<nblk64, 256, 0, st>>>(n, batch, rows64, m->gA, B.a1, B.m1, m->wpart);
    k_mlp_wgrad_reduce<<<blocks_for(kHid * (2 * kHid + 1), 32), 256, 0, st>>>(nblk64, kHid, 2 * kHid, m->wpart,
                                                                             m->grad + kOffW2, m->grad + kOffB2);
    k_mlp_dense_bwd<kHid, kHid><<<g256, 128, 0, st>>>(n, batch, L.rowptr, B.params_bf + kOffW2, m->gA, m->gB, m->gM);
    k_mlp_nmean64_bwd<<<gm, 256, 0, st>>>(n, L.rowptr, L.col, m->gM, B.a1, m->gB);   // gB = dL/da1
    // layer 1
    k_mlp_wgrad1<<<gw, 256, 0, st>>>(n, m->gB, B.h0, B.m0, m->wpart);
    k_mlp_wgrad_reduce<<<blocks_for(kHid * 9, 32), 256, 0, st>>>(nblk, kHid, 8, m->wpart, m->grad + kOffW1,
                                                                m->grad + kOffB1);
    CGP_LAUNCH_CHECK();
    return CGP_OK;
}

extern "C" int cgp_mlp_grad(cgp_mlp* m, const double* r, const double* q, const double* target, int32_t batch,
                            float* grad, float* loss, cgp_stream_t stream) {
    clear_error();
    if (!m || !r || !q || !target || !grad || batch < 1 || batch > m->B.maxb) {
        set_error("cgp_mlp_grad: bad arguments");
        return CGP_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CGP_TRY(mlp_backward(m, r, q, target, batch, st));
    CGP_CUDA(cudaMemcpyAsync(grad, m->grad, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, st));
    float l = 0.f;
    CGP_CUDA(cudaMemcpyAsync(&l, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
    CGP_CUDA(cudaStreamSynchronize(st));
    if (loss) *loss = l;
    return CGP_OK;
}

extern "C" int cgp_mlp_train_step(cgp_mlp* m, const double* r, const double* q, const double* target, int32_t batch,
                                  float lr, float* loss, cgp_stream_t stream) {
    clear_error();
    if (!m || !r || !q || !target || batch < 1 || batch > m->B.maxb || !(lr > 0)) {
        set_error("cgp_mlp_train_step: bad arguments");
        return CGP_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CGP_TRY(mlp_backward(m, r, q, target, batch, st));
    m->adam_t += 1;
    k_mlp_adam<<<blocks_for(kMlpParams), kBlock, 0, st>>>(kMlpParams, m->B.params, m->grad, m->adam_m, m->adam_v,
                                                         m->adam_t, lr, m->B.params_bf);
    CGP_LAUNCH_CHECK();
    if (loss) {
        CGP_CUDA(cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        CGP_CUDA(cudaStreamSynchronize(st));
    }
    return CGP_OK;
}

extern "C" int cgp_guess_set(cgp_solver* h, const cgp_mlp* m, cgp_stream_t stream) {
    clear_error();
    if (!h || !m) {
        set_error("cgp_guess_set: null argument");
        return CGP_EINVAL;
    }
    Solver& s = h->s;
    if (!s.mlp.params || m->mesh != s.mesh || m->level != s.lc) {
        set_error("cgp_guess_set: the solver was not assembled with CGP_GUESS_LEARNED, or the network belongs to "
                  "another mesh level");
        return CGP_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CGP_CUDA(cudaMemcpyAsync(s.mlp.params, m->B.params, sizeof(float) * kMlpParams, cudaMemcpyDeviceToDevice, st));
    CGP_CUDA(cudaMemcpyAsync(s.mlp.params_bf, m->B.params_bf, sizeof(__nv_bfloat16) * kMlpParams,
                             cudaMemcpyDeviceToDevice, st));
    CGP_CUDA(cudaStreamSynchronize(st));
    s.guess_ready = true;
    return CGP_OK;
}
