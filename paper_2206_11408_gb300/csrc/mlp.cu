// Learned angle predictor (an extension of FINGER; the paper has no learned
// predictor): training data harvest, training kernels and weight upload.
//
// The predictor maps the r + 4 features of a (q, c, d) triple (see
// features_row in search_impl.cuh) to cos(q_res, d_res) with a 64-64 ReLU MLP
// and replaces the distribution matching of Algorithm 3 in the MLP search mode.
// Weights are stored in BF16 (W1, W2, w3) with FP32 biases; training keeps FP32
// master weights and runs the forward pass exactly as inference does (BF16
// weights, hidden-layer inputs rounded to BF16, FP32 accumulation), with the
// roundings passed straight through in the backward pass.
//
// Kernels, two per mini-batch of B rows:
//   k_rows      a block per 32 rows, lane = row, warp = 8 of the 64 units of a layer:
//               x~, h1~ = bf16(relu(W1 x~ + b1)), h2 = relu(W2 h1~ + b2),
//               y = w3 . h2 + b3; training also dy = 2 (y - t) / B,
//               dz2 = dy w3 [h2 > 0], dz1 = W2^T dz2 [h1 > 0] and the squared errors
//   k_weights   thread per weight: sums of dz1 x~, dz2 h1~, dy h2 over the batch (a
//               bias is the weight of a constant 1), then Adam on the FP32 master
// Every sum of outputs and gradients runs in a fixed order (units, inputs and rows
// ascending); the reported losses and eps' add their blocks' sums as they come, in 64 bits.  Weights are
// rounded to BF16 as they are read.  Between the two kernels a quantity is stored
// unit-major (one row of B values per unit), so that both sides move 16 bytes per
// lane.  A step of 4,096 rows with r = 24 took 500 us as six kernels (the weight
// sums alone over 400: 48 blocks of strided loads); the sums' chain of B dependent
// FMAs (8.5 us) bounds it now.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <numeric>
#include <random>
#include <vector>

#include "internal.cuh"

using namespace fg;

finger_status fg_make_plan(finger_index* ix, int mode, int ef_max, int64_t nq, SearchPlan* p,
                           int wpb, int H, int occ = 0, int shape = 0);
finger_status fg_run_search(finger_index* ix, const SearchPlan& p, SearchArgs& a, cudaStream_t s);
SearchArgs fg_base_args(finger_index* ix, const SearchPlan& p);
void fg_drop_captures(const finger_index* ix);

namespace {

constexpr int HID = MLP_H;

__host__ __device__ inline int64_t wcount(int nf) { return (int64_t)HID * nf + HID + HID * HID + HID + HID + 1; }

struct Off {
    int64_t W1, b1, W2, b2, w3, b3;
    __host__ __device__ explicit Off(int nf) {
        W1 = 0;
        b1 = W1 + (int64_t)HID * nf;
        W2 = b1 + HID;
        b2 = W2 + HID * HID;
        w3 = b2 + HID;
        b3 = w3 + HID;
    }
};

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

constexpr int RB = 32;        // rows per block of k_rows
constexpr int RT = 256;       // its threads: a warp per 8 units
constexpr int WTJ = 8, WTK = 16, WTB = 128;   // weights per block of k_weights, rows per stage
constexpr int WLD = WTB + 4;  // its row stride in shared memory (conflict-free 16-byte reads)

size_t rows_smem(int nf, bool train) {
    return sizeof(float) * ((size_t)nf * (HID + RB) + HID * HID + 2 * HID * RB + HID + RB +
                            (train ? HID * HID + HID * RB : 0));
}

// per-unit arrays of a batch: nf, 64, 64, 64, 64 and 1 rows of Bp values
struct Batch {
    float *x, *h1, *h2, *dz1, *dz2, *dy;
    int64_t Bp;
};

// rows idx[0 .. B) (or 0 .. B - 1) of X (N x nf).  TRAIN: a block per 32 rows.  Forward only:
// the block goes on to further ones with its weights in place (2M rows, r = 24: 1.08 ms; 2.43
// with a block per 32 rows, which spent it on the weights; 1.78 for a thread per row).
template <bool TRAIN>
__global__ void __launch_bounds__(RT) k_rows(const float* __restrict__ w, int nf,
                                             const float* __restrict__ X, const float* __restrict__ T,
                                             const int64_t* __restrict__ idx, int B, Batch g,
                                             float* res, float* y_out, double* sq) {
    extern __shared__ __align__(16) float sw[];
    float* W1t = sw;                       // nf x 64: W1 transposed
    float* W2t = W1t + nf * HID;           // 64 x 64: W2 transposed
    float* xs = W2t + HID * HID;           // nf x 32
    float* h1 = xs + nf * RB;              // 64 x 32
    float* h2 = h1 + HID * RB;             // 64 x 32
    float* w3 = h2 + HID * RB;             // 64
    float* dyv = w3 + HID;                 // 32
    float* W2s = dyv + RB;                 // (TRAIN) 64 x 64: W2
    float* dz = W2s + HID * HID;           // (TRAIN) 64 x 32
    const Off o(nf);
    const int t = threadIdx.x, lane = t & 31, u0 = (t >> 5) * 8;
    for (int i = t; i < HID * nf; i += RT) W1t[(i % nf) * HID + i / nf] = bf(w[o.W1 + i]);
    for (int i = t; i < HID * HID; i += RT) {
        const float v = bf(w[o.W2 + i]);
        if (TRAIN) W2s[i] = v;
        W2t[(i % HID) * HID + i / HID] = v;
    }
    if (t < HID) w3[t] = bf(w[o.w3 + t]);

    // out[u0 .. u0 + 7][lane] = init + sum over i of M[i][u] v[i][lane], i ascending
    auto layer = [&](const float* M, const float* v, int n, float (&z)[8]) {
#pragma unroll 4
        for (int i = 0; i < n; ++i) {
            const float a = v[i * RB + lane];
            const float4 m0 = *reinterpret_cast<const float4*>(M + i * HID + u0);
            const float4 m1 = *reinterpret_cast<const float4*>(M + i * HID + u0 + 4);
            z[0] = fmaf(m0.x, a, z[0]);
            z[1] = fmaf(m0.y, a, z[1]);
            z[2] = fmaf(m0.z, a, z[2]);
            z[3] = fmaf(m0.w, a, z[3]);
            z[4] = fmaf(m1.x, a, z[4]);
            z[5] = fmaf(m1.y, a, z[5]);
            z[6] = fmaf(m1.z, a, z[6]);
            z[7] = fmaf(m1.w, a, z[7]);
        }
    };
    for (int r0 = blockIdx.x * RB; r0 < B; r0 += gridDim.x * RB) {
        const int b = r0 + lane;
        for (int i = t; i < RB * nf; i += RT) {   // consecutive threads: consecutive features of a row
            const int r = i / nf, f = i % nf, br = r0 + r;
            xs[f * RB + r] = br < B ? bf(X[(idx ? idx[br] : (int64_t)br) * nf + f]) : 0.f;
        }
        __syncthreads();
        if (TRAIN && b < B)
            for (int f = t >> 5; f < nf; f += RT / 32) g.x[f * g.Bp + b] = xs[f * RB + lane];
        float z[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) z[q] = w[o.b1 + u0 + q];
        layer(W1t, xs, nf, z);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float h = bf(fmaxf(z[q], 0.f));
            h1[(u0 + q) * RB + lane] = h;
            if (TRAIN && b < B) g.h1[(u0 + q) * g.Bp + b] = h;
            z[q] = w[o.b2 + u0 + q];
        }
        __syncthreads();
        layer(W2t, h1, HID, z);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float h = fmaxf(z[q], 0.f);
            h2[(u0 + q) * RB + lane] = h;
            if (TRAIN && b < B) g.h2[(u0 + q) * g.Bp + b] = h;
        }
        __syncthreads();
        if (t < 32) {
            float y = w[o.b3];
#pragma unroll 8
            for (int k = 0; k < HID; ++k) y = fmaf(w3[k], h2[k * RB + lane], y);
            float e = 0.f;
            if (b < B) {
                if (y_out) y_out[b] = y;
                e = y - (T ? T[idx ? idx[b] : (int64_t)b] : 0.f);
                if (res) res[b] = e;
            }
            if (TRAIN) {
                const float dy = 2.f * e / (float)B;
                dyv[lane] = dy;
                if (b < B) g.dy[b] = dy;
                double a = (double)e * e;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
                if (lane == 0) atomicAdd(sq, a);
            }
        }
        if (!TRAIN) continue;   // (the next rows' barriers keep h2 until it is read)
        __syncthreads();
        const float dy = dyv[lane];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = u0 + q;
            const float d = h2[k * RB + lane] > 0.f ? dy * w3[k] : 0.f;
            dz[k * RB + lane] = d;
            if (b < B) g.dz2[k * g.Bp + b] = d;
            z[q] = 0.f;
        }
        __syncthreads();
        layer(W2s, dz, HID, z);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (b < B) g.dz1[(u0 + q) * g.Bp + b] = h1[(u0 + q) * RB + lane] > 0.f ? z[q] : 0.f;
        break;
    }
}

__device__ __forceinline__ void adam(float* w, float* m, float* v, int64_t i, float gi, float lr,
                                     float b1, float b2, float c1, float c2) {
    m[i] = b1 * m[i] + (1.f - b1) * gi;
    v[i] = b2 * v[i] + (1.f - b2) * gi * gi;
    const float mh = m[i] / c1, vh = v[i] / c2;
    w[i] -= lr * mh / (sqrtf(vh) + 1e-8f);
}

// One weight per thread: its gradient summed over the batch's rows in order, written to
// `grad` (when not null) and applied by Adam (when w is not null).  Blocks of 8 x 16
// weights of the three outer products dz1 x [x~, 1], dz2 x [h1~, 1], dy x [h2, 1]; their 24
// rows of values pass through shared memory 128 batch rows at a time.
__global__ void __launch_bounds__(WTJ * WTK)
    k_weights(int nf, int B, Batch g, float* grad, float* w, float* m, float* v, float lr, float b1,
              float b2, float c1, float c2) {
    __shared__ __align__(16) float s[2][WTJ + WTK][WLD];
    const Off o(nf);
    const int n1 = (nf + 1 + WTK - 1) / WTK, n2 = (HID + 1 + WTK - 1) / WTK;
    int blk = blockIdx.x;
    const float *A, *C;   // rows of the outer product's sides
    int nj = HID, nk = HID;
    int64_t wb, bb;
    if (blk < n1 * (HID / WTJ)) {
        A = g.dz1;
        C = g.x;
        nk = nf;
        wb = o.W1;
        bb = o.b1;
    } else if ((blk -= n1 * (HID / WTJ)) < n2 * (HID / WTJ)) {
        A = g.dz2;
        C = g.h1;
        wb = o.W2;
        bb = o.b2;
    } else {
        blk -= n2 * (HID / WTJ);
        A = g.dy;
        C = g.h2;
        nj = 1;
        wb = o.w3;
        bb = o.b3;
    }
    const int nt = nk == nf && A == g.dz1 ? n1 : n2;
    const int j0 = blk / nt * WTJ, k0 = blk % nt * WTK;
    const int t = threadIdx.x, jj = t / WTK, kk = t % WTK;
    const int j = j0 + jj, k = k0 + kk;
    // 16-byte asynchronous copies; rows that do not exist and values past B read as 0
    auto stage = [&](int st, int lo) {
        for (int i = t; i < (WTJ + WTK) * (WTB / 4); i += WTJ * WTK) {
            const int r = i / (WTB / 4), c = i % (WTB / 4) * 4;
            const bool side = r < WTJ;
            const int row = side ? j0 + r : k0 + r - WTJ;
            const bool ok = row < (side ? nj : nk) && lo + c < B;
            const float* src = ok ? (side ? A : C) + (size_t)row * g.Bp + lo + c : A;
            const int bytes = ok ? min(16, 4 * (B - lo - c)) : 0;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&s[st][r][c])),
                         "l"(src), "r"(bytes));
        }
        asm volatile("cp.async.commit_group;");
    };
    float acc = 0.f;
    const bool bias = k == nk;
    stage(0, 0);
    for (int lo = 0, st = 0; lo < B; lo += WTB, st ^= 1) {
        if (lo + WTB < B) stage(st ^ 1, lo + WTB);
        else asm volatile("cp.async.commit_group;");
        asm volatile("cp.async.wait_group 1;");
        __syncthreads();
        const float* a = s[st][jj];
        const float* c = s[st][WTJ + kk];
#pragma unroll 8
        for (int i = 0; i < WTB; i += 4) {
            const float4 x = *reinterpret_cast<const float4*>(a + i);
            float4 y = *reinterpret_cast<const float4*>(c + i);
            if (bias) y = make_float4(1.f, 1.f, 1.f, 1.f);
            acc = fmaf(x.x, y.x, acc);
            acc = fmaf(x.y, y.y, acc);
            acc = fmaf(x.z, y.z, acc);
            acc = fmaf(x.w, y.w, acc);
        }
        __syncthreads();
    }
    if (j >= nj || k > nk) return;
    const int64_t i = bias ? bb + j : wb + (int64_t)j * nk + k;
    if (grad) grad[i] = acc;
    if (w) adam(w, m, v, i, acc, lr, b1, b2, c1, c2);
}

__global__ void k_abs_sum(const float* res, int n, double* out) {
    __shared__ double s[256];
    double a = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        a += fabs((double)res[i]);
    s[threadIdx.x] = a;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out, s[0]);
}

struct Buf {
    std::vector<void*> ptrs;
    template <class T>
    T* get(size_t count) {
        void* p = nullptr;
        if (cudaMalloc(&p, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) return nullptr;
        ptrs.push_back(p);
        return static_cast<T*>(p);
    }
    ~Buf() {
        for (void* p : ptrs) cudaFree(p);
    }
};

bool get_batch(Buf& buf, int nf, int64_t B, Batch* g) {
    g->Bp = (B + 3) & ~int64_t(3);
    g->x = buf.get<float>((size_t)g->Bp * nf);
    g->h1 = buf.get<float>((size_t)g->Bp * HID);
    g->h2 = buf.get<float>((size_t)g->Bp * HID);
    g->dz1 = buf.get<float>((size_t)g->Bp * HID);
    g->dz2 = buf.get<float>((size_t)g->Bp * HID);
    g->dy = buf.get<float>((size_t)g->Bp);
    return g->x && g->h1 && g->h2 && g->dz1 && g->dz2 && g->dy;
}

// g.x == nullptr: forward only
cudaError_t run_rows(int num_sms, const float* w, int nf, const float* X, const float* T, const int64_t* idx,
                     int B, const Batch& g, float* res, float* y, double* sq, cudaStream_t s) {
    const bool train = g.x != nullptr;
    const int smem = (int)rows_smem(nf, train), tiles = (B + RB - 1) / RB;
    const cudaError_t e =
        train ? cudaFuncSetAttribute(k_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
              : cudaFuncSetAttribute(k_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (train) {
        k_rows<true><<<tiles, RT, smem, s>>>(w, nf, X, T, idx, B, g, res, y, sq);
    } else {   // (227 KB of shared memory, 8 blocks of 256 threads)
        const int blocks = num_sms * std::min(8, 227 * 1024 / (smem + 1024));
        k_rows<false><<<std::min(tiles, blocks), RT, smem, s>>>(w, nf, X, T, idx, B, g, res, y, sq);
    }
    return cudaGetLastError();
}

cudaError_t run_weights(int nf, int B, const Batch& g, float* grad, float* w, float* m, float* v,
                        float lr, float b1, float b2, float c1, float c2, cudaStream_t s) {
    const int n1 = (nf + 1 + WTK - 1) / WTK, n2 = (HID + 1 + WTK - 1) / WTK;
    k_weights<<<(n1 + n2) * (HID / WTJ) + n2, WTJ * WTK, 0, s>>>(nf, B, g, grad, w, m, v, lr, b1, b2,
                                                                c1, c2);
    return cudaGetLastError();
}

}  // namespace

// upload a flat FP32 predictor (the order of finger.h) as the inference copy
finger_status finger_load_mlp_internal(finger_index* ix, const float* w, int64_t count, float eps) {
    if (!ix || !w || ix->r < 1) return ix && ix->r < 1 ? FINGER_ERR_NOT_BUILT : FINGER_ERR_INVALID_ARG;
    const int nf = ix->r + 4;
    if (count != wcount(nf)) return FINGER_ERR_INVALID_ARG;
    const Off o(nf);
    const int kp = (nf + 15) & ~15;
    std::vector<__nv_bfloat16> W1((size_t)HID * kp), W2((size_t)HID * HID);
    for (int j = 0; j < HID; ++j)
        for (int i = 0; i < kp; ++i)
            W1[(size_t)j * kp + i] = __float2bfloat16_rn(i < nf ? w[o.W1 + (int64_t)j * nf + i] : 0.f);
    for (int i = 0; i < HID * HID; ++i) W2[i] = __float2bfloat16_rn(w[o.W2 + i]);
    // fragment-major B operands of m16n8k16 (row n = 8 nt + g of the weight
    // matrix, k pairs 16 ks + 2t and 16 ks + 2t + 8 of that row; g = lane / 4,
    // t = lane % 4): one uint2 per lane per (nt, ks)
    auto frag = [](const std::vector<__nv_bfloat16>& Wm, int K) {
        const int nk = K / 16;
        std::vector<uint2> f((size_t)8 * nk * 32);
        auto bits = [&](int row, int col) {
            __nv_bfloat16 v = Wm[(size_t)row * K + col];
            uint16_t u;
            memcpy(&u, &v, 2);
            return (uint32_t)u;
        };
        for (int nt = 0; nt < 8; ++nt)
            for (int ks = 0; ks < nk; ++ks)
                for (int lane = 0; lane < 32; ++lane) {
                    const int n = 8 * nt + (lane >> 2), c = 16 * ks + 2 * (lane & 3);
                    f[((size_t)nt * nk + ks) * 32 + lane] =
                        make_uint2(bits(n, c) | bits(n, c + 1) << 16,
                                   bits(n, c + 8) | bits(n, c + 9) << 16);
                }
        return f;
    };
    const std::vector<uint2> W1f = frag(W1, kp), W2f = frag(W2, HID);
    std::vector<float> w3(HID), b1(w + o.b1, w + o.b1 + HID), b2(w + o.b2, w + o.b2 + HID);
    for (int k = 0; k < HID; ++k) w3[k] = __bfloat162float(__float2bfloat16_rn(w[o.w3 + k]));
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ix->device);
    cudaFree(ix->W1f);
    cudaFree(ix->W2f);
    cudaFree(ix->w3);
    cudaFree(ix->b1);
    cudaFree(ix->b2);
    ix->W1f = ix->W2f = nullptr;
    ix->w3 = ix->b1 = ix->b2 = nullptr;
    bool ok = cudaMalloc(&ix->W1f, W1f.size() * sizeof(uint2)) == cudaSuccess &&
              cudaMalloc(&ix->W2f, W2f.size() * sizeof(uint2)) == cudaSuccess &&
              cudaMalloc(&ix->w3, HID * 4) == cudaSuccess &&
              cudaMalloc(&ix->b1, HID * 4) == cudaSuccess &&
              cudaMalloc(&ix->b2, HID * 4) == cudaSuccess;
    ok = ok &&
         cudaMemcpy(ix->W1f, W1f.data(), W1f.size() * sizeof(uint2), cudaMemcpyHostToDevice) ==
             cudaSuccess &&
         cudaMemcpy(ix->W2f, W2f.data(), W2f.size() * sizeof(uint2), cudaMemcpyHostToDevice) ==
             cudaSuccess &&
         cudaMemcpy(ix->w3, w3.data(), HID * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(ix->b1, b1.data(), HID * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(ix->b2, b2.data(), HID * 4, cudaMemcpyHostToDevice) == cudaSuccess;
    cudaSetDevice(prev);
    if (!ok) {
        cudaGetLastError();
        return FINGER_ERR_OOM;
    }
    ix->b3 = w[o.b3];
    ix->mlp_eps = eps;
    ix->mlp_kp = kp;
    ix->h_mlp.assign(w, w + count);
    ix->has_mlp = 1;
    fg_drop_captures(ix);
    return FINGER_OK;
}

extern "C" {

int64_t finger_mlp_size(int r) { return r < 1 ? -1 : wcount(r + 4); }

finger_status finger_set_predictor(finger_index* ix, const float* weights, int64_t count,
                                   float eps) {
    return finger_load_mlp_internal(ix, weights, count, eps);
}

finger_status finger_set_predictor_gate(finger_index* ix, float delta) {
    if (!ix || !(delta == delta)) return FINGER_ERR_INVALID_ARG;
    if (ix->mlp_delta != delta) fg_drop_captures(ix);   // captured launches hold the index view
    ix->mlp_delta = delta;
    return FINGER_OK;
}

finger_status finger_get_predictor(const finger_index* ix, float* weights, float* eps) {
    if (!ix) return FINGER_ERR_INVALID_ARG;
    if (!ix->has_mlp) return FINGER_ERR_NOT_BUILT;
    if (weights) memcpy(weights, ix->h_mlp.data(), ix->h_mlp.size() * sizeof(float));
    if (eps) *eps = ix->mlp_eps;
    return FINGER_OK;
}

finger_status finger_harvest(finger_index* ix, const float* queries, int64_t nq, int ef,
                             int64_t cap, float* feat, float* target, int32_t* triples,
                             int64_t* count, void* stream) {
    if (!ix || !queries || nq < 1 || ef < 1 || ef > MAX_EF || cap < 1 || !feat || !target ||
        !triples || !count)
        return FINGER_ERR_INVALID_ARG;
    if (!ix->adj0 || !ix->edge_u) return FINGER_ERR_NOT_BUILT;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ix->device);
    cudaStream_t s = (cudaStream_t)stream;
    finger_status st;
    SearchPlan p;
    Buf buf;
    int64_t* ids = buf.get<int64_t>((size_t)nq);
    float* ds = buf.get<float>((size_t)nq);
    unsigned long long* cnt = buf.get<unsigned long long>(1);
    if (!ids || !ds || !cnt) {
        cudaSetDevice(prev);
        return FINGER_ERR_OOM;
    }
    st = fg_make_plan(ix, MODE_HARVEST, ef, nq, &p, 4, 0);
    if (st == FINGER_OK) {
        SearchArgs a = fg_base_args(ix, p);
        a.Q = queries;
        a.nq = nq;
        a.K = 1;
        a.ef = ef;
        a.out_ids = ids;
        a.out_d = ds;
        a.hv_feat = feat;
        a.hv_target = target;
        a.hv_trip = triples;
        a.hv_count = cnt;
        a.hv_cap = cap;
        if (cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s) != cudaSuccess) st = FINGER_ERR_CUDA;
        else st = fg_run_search(ix, p, a, s);
        unsigned long long h = 0;
        if (st == FINGER_OK &&
            (cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
             cudaStreamSynchronize(s) != cudaSuccess))
            st = FINGER_ERR_CUDA;
        *count = (int64_t)std::min<unsigned long long>(h, (unsigned long long)cap);
    }
    cudaGetLastError();
    cudaSetDevice(prev);
    return st;
}

finger_status finger_mlp_loss_grad(finger_index* ix, int nf, const float* weights,
                                   const float* feat, const float* target, int64_t n, float* grad,
                                   double* loss, void* stream) {
    if (!ix || nf < 1 || nf > 96 || !weights || !feat || !target || n < 1 || n > (1 << 24) || !grad)
        return FINGER_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ix->device);
    cudaStream_t s = (cudaStream_t)stream;
    const int B = (int)n;
    const int64_t nw = wcount(nf);
    Buf buf;
    float* w = buf.get<float>(nw);
    float* g = buf.get<float>(nw);
    double* acc = buf.get<double>(1);
    Batch bt;
    finger_status st = FINGER_OK;
    if (!w || !g || !acc || !get_batch(buf, nf, B, &bt)) {
        st = FINGER_ERR_OOM;
    } else {
        double h = 0;
        bool ok = cudaMemcpyAsync(w, weights, nw * 4, cudaMemcpyHostToDevice, s) == cudaSuccess;
        ok = ok && cudaMemsetAsync(acc, 0, 8, s) == cudaSuccess;
        ok = ok && run_rows(ix->num_sms, w, nf, feat, target, nullptr, B, bt, nullptr, nullptr, acc, s) == cudaSuccess;
        ok = ok && run_weights(nf, B, bt, g, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, 1.f, 1.f, s) ==
                       cudaSuccess;
        ok = ok && cudaMemcpyAsync(grad, g, nw * 4, cudaMemcpyDeviceToHost, s) == cudaSuccess;
        ok = ok && cudaMemcpyAsync(&h, acc, 8, cudaMemcpyDeviceToHost, s) == cudaSuccess;
        ok = ok && cudaStreamSynchronize(s) == cudaSuccess;
        if (!ok) st = FINGER_ERR_CUDA;
        if (loss) *loss = h / B;
    }
    cudaGetLastError();
    cudaSetDevice(prev);
    return st;
}

finger_status finger_mlp_predict(finger_index* ix, const float* feat, int64_t n, float* out,
                                 void* stream) {
    if (!ix || !feat || !out || n < 0) return FINGER_ERR_INVALID_ARG;
    if (!ix->has_mlp) return FINGER_ERR_NOT_BUILT;
    if (n == 0) return FINGER_OK;
    const int nf = ix->r + 4;
    const int64_t nw = wcount(nf);
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ix->device);
    cudaStream_t s = (cudaStream_t)stream;
    Buf buf;
    float* w = buf.get<float>(nw);
    finger_status st = FINGER_OK;
    if (!w) {
        st = FINGER_ERR_OOM;
    } else {
        bool ok = cudaMemcpyAsync(w, ix->h_mlp.data(), nw * 4, cudaMemcpyHostToDevice, s) == cudaSuccess;
        for (int64_t lo = 0; lo < n && ok; lo += 1 << 20) {
            const int B = (int)std::min<int64_t>(n - lo, 1 << 20);
            ok = run_rows(ix->num_sms, w, nf, feat + lo * nf, nullptr, nullptr, B, Batch{}, nullptr, out + lo, nullptr,
                          s) == cudaSuccess;
        }
        ok = ok && cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(s) == cudaSuccess;
        if (!ok) st = FINGER_ERR_CUDA;
    }
    cudaGetLastError();
    cudaSetDevice(prev);
    return st;
}

finger_status finger_train_predictor(finger_index* ix, const finger_train_params* p, float* losses,
                                     void* stream) {
    if (!ix || !p || !p->feat || !p->target || p->n_train < 1 || p->n_val < 0 || p->epochs < 1 ||
        p->batch < 1 || p->batch > (1 << 20) || !(p->lr > 0))
        return FINGER_ERR_INVALID_ARG;
    if (ix->r < 1) return FINGER_ERR_NOT_BUILT;
    const int nf = ix->r + 4;
    const int64_t nw = wcount(nf);
    const Off o(nf);
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ix->device);
    cudaStream_t s = (cudaStream_t)stream;
    const int B = p->batch;
    Buf buf;
    float* w = buf.get<float>(nw);
    float* m1 = buf.get<float>(nw);
    float* m2 = buf.get<float>(nw);
    float* res = buf.get<float>(B);
    int64_t* idx = buf.get<int64_t>((size_t)p->n_train);
    double* acc = buf.get<double>(1);
    Batch bt;
    if (!w || !m1 || !m2 || !res || !idx || !acc || !get_batch(buf, nf, B, &bt)) {
        cudaSetDevice(prev);
        return FINGER_ERR_OOM;
    }
    // He-uniform initialisation of the masters (seeded), zero biases
    std::vector<float> hw((size_t)nw, 0.f);
    std::mt19937_64 rng(p->seed);
    std::uniform_real_distribution<float> U(-1.f, 1.f);
    const float s1 = sqrtf(6.f / nf), s2 = sqrtf(6.f / HID);
    for (int64_t i = 0; i < (int64_t)HID * nf; ++i) hw[o.W1 + i] = U(rng) * s1;
    for (int64_t i = 0; i < HID * HID; ++i) hw[o.W2 + i] = U(rng) * s2;
    for (int64_t i = 0; i < HID; ++i) hw[o.w3 + i] = U(rng) * s2;
    bool ok = cudaMemcpyAsync(w, hw.data(), nw * 4, cudaMemcpyHostToDevice, s) == cudaSuccess &&
              cudaMemsetAsync(m1, 0, nw * 4, s) == cudaSuccess &&
              cudaMemsetAsync(m2, 0, nw * 4, s) == cudaSuccess;
    std::vector<int64_t> perm((size_t)p->n_train);
    std::iota(perm.begin(), perm.end(), 0);
    int64_t step = 0;
    const float b1 = 0.9f, b2 = 0.999f;
    std::shuffle(perm.begin(), perm.end(), rng);
    for (int ep = 0; ep < p->epochs && ok; ++ep) {
        ok = cudaMemcpyAsync(idx, perm.data(), perm.size() * 8, cudaMemcpyHostToDevice, s) == cudaSuccess &&
             cudaStreamSynchronize(s) == cudaSuccess;
        double sq = 0;
        ok = ok && cudaMemsetAsync(acc, 0, 8, s) == cudaSuccess;
        for (int64_t lo = 0; lo + B <= p->n_train && ok; lo += B) {
            step++;
            const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
            ok = run_rows(ix->num_sms, w, nf, p->feat, p->target, idx + lo, B, bt, nullptr, nullptr, acc, s) ==
                     cudaSuccess &&
                 run_weights(nf, B, bt, nullptr, w, m1, m2, p->lr, b1, b2, c1, c2, s) == cudaSuccess;
        }
        // the next epoch's order while this one runs
        if (ep + 1 < p->epochs) std::shuffle(perm.begin(), perm.end(), rng);
        ok = ok && cudaMemcpyAsync(&sq, acc, 8, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
             cudaStreamSynchronize(s) == cudaSuccess;
        if (losses) losses[ep] = (float)(sq / std::max<int64_t>(1, (p->n_train / B) * B));
    }
    // eps' = mean |prediction - target| on the held-out rows (inference semantics)
    float eps = 0.f;
    if (ok) {
        ok = cudaMemsetAsync(acc, 0, 8, s) == cudaSuccess;
        const int64_t v0 = p->n_train, nv = p->n_val;
        for (int64_t lo = 0; lo < nv && ok; lo += B) {
            const int nb = (int)std::min<int64_t>(B, nv - lo);
            ok = run_rows(ix->num_sms, w, nf, p->feat + (v0 + lo) * nf, p->target + v0 + lo, nullptr, nb, Batch{}, res,
                          nullptr, nullptr, s) == cudaSuccess;
            k_abs_sum<<<16, 256, 0, s>>>(res, nb, acc);
        }
        double sa = 0;
        ok = ok && cudaMemcpyAsync(&sa, acc, 8, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
             cudaStreamSynchronize(s) == cudaSuccess;
        eps = nv > 0 ? (float)(sa / nv) : 0.f;
    }
    if (ok) ok = cudaMemcpy(hw.data(), w, nw * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    cudaGetLastError();
    cudaSetDevice(prev);
    if (!ok) return FINGER_ERR_CUDA;
    return finger_load_mlp_internal(ix, hw.data(), nw, eps);
}

}  // extern "C"
