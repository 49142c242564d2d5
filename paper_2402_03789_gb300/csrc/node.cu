// Node-level kernels of the interaction blocks and the readout.
//
//  * per-irrep linears (linear_1, self-connection, linear_2; Figure 2b and the
//    self-connection-as-linear of Sec. 5.1): out[v, m, :] = in[v, m, :] @ W,
//    W pre-scaled by 1/sqrt(fan_in); rows are (atom, m) pairs.
//  * gate (NequIP's equivariant nonlinearity, Sec. 3.2) and its adjoint.
//  * embedding h1 = W_emb[Z] and the atomwise readout (Eq. 1).
//  * forces F_v = sum_w (F_vw - F_wv) (Eq. 6) from the per-edge gradients
//    F_vw = dE/dd_vw accumulated over blocks (Eq. 5), and the atom virials
//    -sum_e F_e (x) d_e, both summed in FP64.
#include "internal.h"

#include <algorithm>

namespace sn {

__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ float silu_(float x) { return x * sigm(x); }
__device__ __forceinline__ float dsilu_(float x) {
    float s = sigm(x);
    return s * (1.0f + x * (1.0f - s));
}

// ---------------------------------------------------------------- FP32 GEMM
// TM x TN output tile, 4 x 4 per thread, K slices of 16 through a ring of four
// stages filled by cp.async (a slice waited for its loads before: 17 us a launch
// for cells of any size up to some hundred atoms).  Small problems take 32 x 32
// tiles, which spread them over more SMs.  k runs in ascending order either way, so
// a row's result does not depend on the batch it is in.
constexpr int GK = 16, GST = 4;

__device__ __forceinline__ void g_cp16(void* s, const void* g, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g),
                 "r"(valid ? 16 : 0) : "memory");
}

template <int TM, int TN>
__global__ void __launch_bounds__(TM * TN / 16)
gemm_f32_kernel(const __grid_constant__ GemmBatch batch) {
    constexpr int NT = TM * TN / 16, NA = TM * GK / 4 / NT, NB = TN * GK / 4 / NT;
    const GemmProb& P = batch.p[blockIdx.z];
    const int64_t rows = P.n_atoms * P.R;
    const int64_t r0 = (int64_t)blockIdx.x * TM;
    const int n0 = blockIdx.y * TN;
    if (r0 >= rows || n0 >= P.N) return;
    __shared__ __align__(16) float sA[GST][TM][GK + 4];
    __shared__ __align__(16) float sB[GST][GK][TN];
    const int t = threadIdx.x;
    const int tr = t / (TN / 4), tc = t % (TN / 4);
    float acc[4][4] = {};
    // loaders: A row (t + i NT) / 4, k quad % 4; B row (t + i NT) / (TN / 4)
    const float* aptr[NA][2];
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        const int64_t ar = r0 + (t + i * NT) / 4, v = (ar < rows ? ar : 0) / P.R;
        const int mm = (int)((ar < rows ? ar : 0) % P.R);
        aptr[i][0] = P.A + v * P.lda + P.a_off + (int64_t)mm * P.K;
        aptr[i][1] = P.K2 ? P.A2 + v * P.lda2 + P.a_off2 + (int64_t)mm * P.K2 : nullptr;
    }
    const int s1 = P.K / GK, slices = s1 + P.K2 / GK;
    auto load = [&](int sl) {
        const bool two = sl >= s1;
        const int k0 = (two ? sl - s1 : sl) * GK, b = sl % GST;
        const float* B = two ? P.B2 : P.B;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int q = t + i * NT;
            g_cp16(&sA[b][q / 4][4 * (q % 4)], aptr[i][two] + k0 + 4 * (q % 4), r0 + q / 4 < rows);
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int q = t + i * NT, kk = q / (TN / 4), col = n0 + 4 * (q % (TN / 4));
            g_cp16(&sB[b][kk][4 * (q % (TN / 4))], B + (int64_t)(k0 + kk) * P.N + (col < P.N ? col : 0), col < P.N);
        }
    };
#pragma unroll
    for (int i = 0; i < GST - 1; ++i) {
        if (i < slices) load(i);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int sl = 0; sl < slices; ++sl) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(GST - 2) : "memory");
        __syncthreads();
        if (sl + GST - 1 < slices) load(sl + GST - 1);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        const int b = sl % GST;
#pragma unroll
        for (int k4 = 0; k4 < GK / 4; ++k4) {
            float aa[4][4], bb[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 q = *reinterpret_cast<const float4*>(&sA[b][4 * tr + i][4 * k4]);
                aa[i][0] = q.x; aa[i][1] = q.y; aa[i][2] = q.z; aa[i][3] = q.w;
                const float4 p = *reinterpret_cast<const float4*>(&sB[b][4 * k4 + i][4 * tc]);
                bb[i][0] = p.x; bb[i][1] = p.y; bb[i][2] = p.z; bb[i][3] = p.w;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(aa[i][kk], bb[kk][j], acc[i][j]);
        }
    }
    const int col = n0 + 4 * tc;
    if (col >= P.N) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t row = r0 + 4 * tr + i;
        if (row >= rows) break;
        const int64_t v = row / P.R;
        const int mm = (int)(row % P.R);
        float* cp = P.C + v * P.ldc + (P.c_blk ? P.c_blk[col >> 5] + 32 * mm + (col & 31) : P.c_off + mm * P.N + col);
        float4 o = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        if (P.accumulate) {
            const float4 c = *reinterpret_cast<const float4*>(cp);
            o.x += c.x; o.y += c.y; o.z += c.z; o.w += c.w;
        }
        *reinterpret_cast<float4*>(cp) = o;
    }
}

// ---------------------------------------------------------------- BF16 GEMM
// Tensor cores (mma.sync m16n8k16, BF16 operands, FP32 accumulate).  A is read
// as FP32 and rounded to BF16 in the fragment; B is the BF16 [N][K] copy.
// Activations and weights both enter as hi + lo BF16 pairs; three MMAs
// (hi*hi, lo*hi, hi*lo) keep about 16 mantissa bits of each operand.
constexpr bool GEMM_SPLIT_ACT = true;

__device__ __forceinline__ void split_bf16_n(float x, float y, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

__device__ __forceinline__ void mma_bf16_n(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// 128 x 64 output tile, 8 warps as 4 (rows) x 2 (cols), each warp 32 rows x 32
// cols (2 m tiles x 4 n tiles); for N <= 32 the warps stack 8 x 1 over 256 x 32.
// K runs in blocks of 32 under one k permutation of both operands (the
// reduction order inside an MMA is free): lane tq owns
// k = kb + 8 tq + [0, 8), k step ks takes kb + 8 tq + 4 ks + [0, 4).  Its A
// values are then one float4 per row and k step, and its B words (hi and lo)
// one 16-byte load per n row and k block.  K and N are multiples of 32.
// PF: the next k block's operands are loaded before this one's MMAs (small
// problems, one CTA or fewer per SM: their k blocks otherwise wait for memory one
// after another); large problems hide it behind the other CTA of the SM instead.
// DUAL: some problem has a second product.
template <bool PF, bool DUAL>
__global__ void __launch_bounds__(256, PF ? 1 : 2)
gemm_bf16_kernel(const __grid_constant__ GemmBatch batch) {
    const GemmProb& P = batch.p[blockIdx.z];
    const int64_t rows = P.n_atoms * P.R;
    // N <= 32: the 8 warps stack as 8 x 1 over a 256 x 32 tile (the grid's extra
    // row blocks exit); otherwise 4 x 2 over 128 x 64
    const bool narrow = P.N <= 32;
    const int64_t r0 = (int64_t)blockIdx.x * (narrow ? 256 : 128);
    const int n0 = blockIdx.y * 64;
    if (r0 >= rows || n0 >= P.N) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, tq = lane & 3;
    const int wr = narrow ? warp : (warp & 3), wc = narrow ? 0 : (warp >> 2);
    const int nbase = n0 + wc * 32;
    if (nbase >= P.N) return;
    const float* pr[2][2];
    float c[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int j = 0; j < 4; ++j) c[mt][j][0] = c[mt][j][1] = c[mt][j][2] = c[mt][j][3] = 0.0f;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    struct Ops {
        uint4 bh[4], bl[4];
        float4 av[2][2][2];                                // [m tile][row half][k step]
    };
#pragma unroll 1
    for (int seg = 0; seg < (DUAL ? 2 : 1); ++seg) {
        const int K = seg ? P.K2 : P.K;
        if (DUAL && K == 0) break;
        const __nv_bfloat16* Bh = seg ? P.Bh2 : P.Bh;
        const int64_t lo_off = (int64_t)K * P.N;           // bf16 elements
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t r = r0 + wr * 32 + mt * 16 + h * 8 + g;
                pr[mt][h] = r < rows ? (seg ? P.A2 + P.a_off2 : P.A + P.a_off) + r / P.R * (seg ? P.lda2 : P.lda) +
                                           (int64_t)(int)(r % P.R) * K
                                     : nullptr;
            }
        auto load = [&](int kb, Ops& o) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat16* br = Bh + (int64_t)(nbase + j * 8 + g) * K + kb + 8 * tq;
                o.bh[j] = __ldg(reinterpret_cast<const uint4*>(br));
                o.bl[j] = __ldg(reinterpret_cast<const uint4*>(br + lo_off));
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
                        o.av[mt][h][ks] = pr[mt][h] ? *reinterpret_cast<const float4*>(pr[mt][h] + kb + 8 * tq + 4 * ks) : z4;
        };
        auto mul = [&](const Ops& o) {
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    uint32_t a[4], al[4];
                    split_bf16_n(o.av[mt][0][ks].x, o.av[mt][0][ks].y, a[0], al[0]);
                    split_bf16_n(o.av[mt][1][ks].x, o.av[mt][1][ks].y, a[1], al[1]);
                    split_bf16_n(o.av[mt][0][ks].z, o.av[mt][0][ks].w, a[2], al[2]);
                    split_bf16_n(o.av[mt][1][ks].z, o.av[mt][1][ks].w, a[3], al[3]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t* wh = reinterpret_cast<const uint32_t*>(&o.bh[j]);
                        const uint32_t* wl = reinterpret_cast<const uint32_t*>(&o.bl[j]);
                        const uint32_t b[2] = {wh[2 * ks], wh[2 * ks + 1]};
                        const uint32_t b2[2] = {wl[2 * ks], wl[2 * ks + 1]};
                        mma_bf16_n(c[mt][j], a, b);
                        if (GEMM_SPLIT_ACT) mma_bf16_n(c[mt][j], al, b);
                        mma_bf16_n(c[mt][j], a, b2);
                    }
                }
            }
        };
        if constexpr (PF) {
            Ops o0, o1;
            load(0, o0);
            for (int kb = 0; kb < K; kb += 64) {
                if (kb + 32 < K) load(kb + 32, o1);
                mul(o0);
                if (kb + 32 >= K) break;
                if (kb + 64 < K) load(kb + 64, o0);
                mul(o1);
            }
        } else {
            for (int kb = 0; kb < K; kb += 32) {
                Ops o;
                load(kb, o);
                mul(o);
            }
        }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t r = r0 + wr * 32 + mt * 16 + h * 8 + g;
            if (r >= rows) continue;
            const int64_t v = r / P.R;
            const int mm = (int)(r % P.R);
            float* cp = P.C + v * P.ldc + (P.c_blk ? P.c_blk[nbase >> 5] + 32 * mm - nbase : P.c_off + mm * P.N);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = nbase + j * 8 + 2 * tq;
                float2 o = make_float2(c[mt][j][2 * h], c[mt][j][2 * h + 1]);
                if (P.accumulate) {
                    const float2 q = *reinterpret_cast<const float2*>(cp + col);
                    o.x += q.x;
                    o.y += q.y;
                }
                *reinterpret_cast<float2*>(cp + col) = o;
            }
        }
}

void launch_gemm(const GemmBatch& b, sevennet_precision prec, cudaStream_t st) {
    if (b.n == 0) return;
    int64_t max_rows = 0;
    int max_n = 0;
    for (int i = 0; i < b.n; ++i) {
        max_rows = std::max<int64_t>(max_rows, b.p[i].n_atoms * b.p[i].R);
        max_n = std::max(max_n, b.p[i].N);
    }
    if (max_rows == 0) return;
    int dev = 0;
    cudaGetDevice(&dev);
    const int64_t sms = num_sms(dev);
    if (prec == SEVENNET_BF16) {
        const dim3 grid((unsigned)((max_rows + 127) / 128), (unsigned)((max_n + 63) / 64), (unsigned)b.n);
        bool dual = false;
        for (int i = 0; i < b.n; ++i) dual = dual || b.p[i].K2 > 0;
        const bool pf = (int64_t)grid.x * grid.y * grid.z <= sms;
        if (pf && dual) gemm_bf16_kernel<true, true><<<grid, 256, 0, st>>>(b);
        else if (pf) gemm_bf16_kernel<true, false><<<grid, 256, 0, st>>>(b);
        else if (dual) gemm_bf16_kernel<false, true><<<grid, 256, 0, st>>>(b);
        else gemm_bf16_kernel<false, false><<<grid, 256, 0, st>>>(b);
    } else {
        const dim3 grid((unsigned)((max_rows + 63) / 64), (unsigned)((max_n + 63) / 64), (unsigned)b.n);
        if ((int64_t)grid.x * grid.y * grid.z < 2 * sms) {
            const dim3 small((unsigned)((max_rows + 31) / 32), (unsigned)((max_n + 31) / 32), (unsigned)b.n);
            gemm_f32_kernel<32, 32><<<small, 64, 0, st>>>(b);
        } else {
            gemm_f32_kernel<64, 64><<<grid, 256, 0, st>>>(b);
        }
    }
}

// ---------------------------------------------------------------- embedding
__device__ __forceinline__ int clamp_species(int s, int ns) { return s < 0 ? 0 : (s >= ns ? ns - 1 : s); }

// Out-of-range species are clamped here (no out-of-bounds read) and reported
// as an error by the host after the evaluation.
__global__ void embed_kernel(const float* __restrict__ table, const int* __restrict__ species,
                             int64_t n, int mul0, int n_species, float* __restrict__ h) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * mul0) return;
    const int64_t v = i / mul0;
    const int u = (int)(i % mul0);
    h[i] = table[(int64_t)clamp_species(species[v], n_species) * mul0 + u];
}

void launch_embed(const float* table, const int* species, int64_t n, int mul0, int n_species, float* h,
                  cudaStream_t st) {
    const int64_t tot = n * mul0;
    if (tot == 0) return;
    embed_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(table, species, n, mul0, n_species, h);
}

// ---------------------------------------------------------------- gate
struct GateDims {
    int mul0, ng, lmax, y_dim, h_dim;
    int mul[NL], y_off[NL], h_off[NL], goff[NL];
    int last;
};

// Entry l (1..3) of a per-irrep array of the kernel parameter, by selects: a
// dynamic index into a by-value parameter array would copy it to local memory.
__device__ __forceinline__ int irrep_sel(const int (&a)[NL], int l) {
    return l == 1 ? a[1] : (l == 2 ? a[2] : a[3]);
}

static GateDims gate_dims(const LayerDev& L, int mul0, const int* mul, int lmax) {
    GateDims g{};
    g.mul0 = mul0;
    g.lmax = lmax;
    g.y_dim = L.y_dim;
    g.h_dim = L.h_out_dim;
    g.last = L.last ? 1 : 0;
    int go = 0;
    for (int l = 0; l < NL; ++l) {
        g.mul[l] = (l <= lmax) ? mul[l] : 0;
        g.y_off[l] = L.y_off[l];
        g.h_off[l] = L.out_off[l];
        if (l >= 1 && l <= lmax) { g.goff[l] = go; go += mul[l]; }
    }
    g.ng = go;
    return g;
}

// The gate kernels walk atoms (grid-stride) with the CTA's threads over one
// atom's row, so no element index is divided by a row length.
static inline unsigned gate_grid(int64_t n) {
    int dev = 0;
    cudaGetDevice(&dev);
    const int64_t g = (int64_t)8 * num_sms(dev);
    return (unsigned)(n < g ? n : g);
}

__global__ void gate_fwd_kernel(const GateDims G, int64_t n, const float* __restrict__ y,
                                float* __restrict__ h) {
    for (int64_t v = blockIdx.x; v < n; v += gridDim.x) {
        const float* yr = y + v * G.y_dim;
        float* hr = h + v * G.h_dim;
        for (int j = threadIdx.x; j < G.h_dim; j += blockDim.x) {
            if (G.last || j < G.mul0) {
                hr[j] = silu_(yr[j]);
                continue;
            }
            const int l = 1 + (G.lmax >= 2 && j >= G.h_off[2]) + (G.lmax >= 3 && j >= G.h_off[3]);
            const int r = j - irrep_sel(G.h_off, l);
            const int u = r % irrep_sel(G.mul, l);
            const float gate = silu_(yr[G.mul0 + irrep_sel(G.goff, l) + u]);
            hr[j] = yr[irrep_sel(G.y_off, l) + r] * gate;
        }
    }
}

void launch_gate_fwd(const LayerDev& L, int mul0, const int* mul, int lmax, int64_t n,
                     const float* y, float* h, cudaStream_t st) {
    const GateDims G = gate_dims(L, mul0, mul, lmax);
    if (n == 0 || G.h_dim == 0) return;
    gate_fwd_kernel<<<gate_grid(n), 256, 0, st>>>(G, n, y, h);
}

// gy = dE/dy from gh = dE/dh (or, for the last block, the readout vector)
__global__ void gate_bwd_kernel(const GateDims G, int64_t n, const float* __restrict__ y,
                                const float* __restrict__ gh, const float* __restrict__ readout,
                                float* __restrict__ gy) {
    for (int64_t v = blockIdx.x; v < n; v += gridDim.x) {
        const float* yr = y + v * G.y_dim;
        const float* ghr = gh + v * G.h_dim;
        float* gyr = gy + v * G.y_dim;
        for (int j = threadIdx.x; j < G.y_dim; j += blockDim.x) {
            if (G.last) {
                gyr[j] = readout[j] * dsilu_(yr[j]);
                continue;
            }
            if (j < G.mul0) {
                gyr[j] = ghr[j] * dsilu_(yr[j]);
                continue;
            }
            if (j < G.mul0 + G.ng) {               // a gate scalar
                const int gidx = j - G.mul0;
                const int l = 1 + (G.lmax >= 2 && gidx >= G.goff[2]) + (G.lmax >= 3 && gidx >= G.goff[3]);
                const int u = gidx - irrep_sel(G.goff, l);
                const int ml = irrep_sel(G.mul, l), ho = irrep_sel(G.h_off, l), yo = irrep_sel(G.y_off, l);
                float s = 0.0f;
                for (int mm = 0; mm < 2 * l + 1; ++mm) {
                    const int off = mm * ml + u;
                    s = fmaf(ghr[ho + off], yr[yo + off], s);
                }
                gyr[j] = s * dsilu_(yr[j]);
                continue;
            }
            const int l = 1 + (G.lmax >= 2 && j >= G.y_off[2]) + (G.lmax >= 3 && j >= G.y_off[3]);
            const int r = j - irrep_sel(G.y_off, l);
            const int u = r % irrep_sel(G.mul, l);
            gyr[j] = ghr[irrep_sel(G.h_off, l) + r] * silu_(yr[G.mul0 + irrep_sel(G.goff, l) + u]);
        }
    }
}

void launch_gate_bwd(const LayerDev& L, int mul0, const int* mul, int lmax, int64_t n,
                     const float* y, const float* gh, const float* readout, float* gy,
                     cudaStream_t st) {
    const GateDims G = gate_dims(L, mul0, mul, lmax);
    if (n == 0 || G.y_dim == 0) return;
    gate_bwd_kernel<<<gate_grid(n), 256, 0, st>>>(G, n, y, gh, readout, gy);
}

// ---------------------------------------------------------------- readout
__global__ void readout_kernel(const float* __restrict__ h, int h_dim, const float* __restrict__ c,
                               const double* __restrict__ shift, const int* __restrict__ species,
                               int64_t n, int mul0, int n_species, double* __restrict__ e_atom) {
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (v >= n) return;
    float s = 0.0f;
    for (int u = lane; u < mul0; u += 32) s = fmaf(h[v * h_dim + u], c[u], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) e_atom[v] = (double)s + shift[clamp_species(species[v], n_species)];
}

void launch_readout(const float* h, int h_dim, const float* c, const double* shift,
                    const int* species, int64_t n, int mul0, int n_species, double* e_atom, cudaStream_t st) {
    if (n == 0) return;
    const int64_t threads = n * 32;
    readout_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(h, h_dim, c, shift, species,
                                                                      n, mul0, n_species, e_atom);
}

// ---------------------------------------------------------------- forces / virial
// Eight lanes an atom (one walked its edges one after another: 41 us for any cell
// up to some thousand atoms); each sums every eighth edge, then a fixed tree.
constexpr int FL = 8;

__global__ void __launch_bounds__(128)
forces_kernel(int64_t n, const int* __restrict__ row_ptr, const int* __restrict__ rev,
              const float* __restrict__ gd, const float4* __restrict__ geom,
              double* __restrict__ f, double* __restrict__ w) {
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / FL;
    const int j = threadIdx.x & (FL - 1);
    double acc[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};      // force, then virial
    if (v < n)
        for (int e = row_ptr[v] + j; e < row_ptr[v + 1]; e += FL) {
            const float* g = gd + (int64_t)e * 3;
            const float* gr = gd + (int64_t)rev[e] * 3;
            const float4 d = geom[e];
            const double gg[3] = {g[0], g[1], g[2]}, dd[3] = {d.x, d.y, d.z};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                acc[a] += gg[a] - (double)gr[a];
#pragma unroll
                for (int b = 0; b < 3; ++b) acc[3 + a * 3 + b] -= gg[a] * dd[b];
            }
        }
#pragma unroll
    for (int k = 0; k < 12; ++k)
#pragma unroll
        for (int o = FL / 2; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (v < n && j == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) f[v * 3 + k] = acc[k];
#pragma unroll
        for (int k = 0; k < 9; ++k) w[v * 9 + k] = acc[3 + k];
    }
}

void launch_forces(int64_t n, const int* row_ptr, const int* rev, const float* gd,
                   const float4* geom, double* f_s, double* w_atom, cudaStream_t st) {
    if (n == 0) return;
    forces_kernel<<<(unsigned)((n * FL + 127) / 128), 128, 0, st>>>(n, row_ptr, rev, gd, geom, f_s, w_atom);
}

// FP64 sums of atom energies and virials per structure in a fixed order that
// depends on the structure alone: a CTA per 512 atoms of a structure (two a thread,
// a shuffle tree per warp, the warps in order), then a warp per structure over its
// CTAs' partial sums.  One CTA per structure took 90 us for 24,000 atoms.
constexpr int RS_ATOMS = 512, RS_THREADS = 256;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// first partial of structure s: structures never share one
__device__ __forceinline__ int64_t partial_base(const int64_t* __restrict__ atom_off, int s) {
    return atom_off[s] / RS_ATOMS + s;
}

__global__ void __launch_bounds__(RS_THREADS) reduce_partials_kernel(int s0,
                                                                     const int64_t* __restrict__ atom_off,
                                                                     const double* __restrict__ e_atom,
                                                                     const double* __restrict__ w_atom,
                                                                     double* __restrict__ partial) {
    const int s = s0 + blockIdx.y;
    const int64_t a0 = atom_off[s] + (int64_t)blockIdx.x * RS_ATOMS, a1 = min(atom_off[s + 1], a0 + RS_ATOMS);
    if (a0 >= a1) return;
    double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t v = a0 + threadIdx.x; v < a1; v += RS_THREADS) {
        acc[0] += e_atom[v];
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[1 + k] += w_atom[v * 9 + k];
    }
    __shared__ double red[RS_THREADS / 32][10];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        const double w = warp_sum_d(acc[k]);
        if (lane == 0) red[warp][k] = w;
    }
    __syncthreads();
    if (threadIdx.x < 10) {
        double t = 0.0;
        for (int i = 0; i < RS_THREADS / 32; ++i) t += red[i][threadIdx.x];
        partial[(partial_base(atom_off, s) + blockIdx.x) * 10 + threadIdx.x] = t;
    }
}

__global__ void reduce_structs_kernel(int n_structs, const int64_t* __restrict__ atom_off,
                                      const double* __restrict__ partial, double* __restrict__ energy,
                                      double* __restrict__ virial) {
    const int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= n_structs) return;
    const int64_t n = (atom_off[s + 1] - atom_off[s] + RS_ATOMS - 1) / RS_ATOMS, b = partial_base(atom_off, s);
    double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t i = lane; i < n; i += 32)
#pragma unroll
        for (int k = 0; k < 10; ++k) acc[k] += partial[(b + i) * 10 + k];
#pragma unroll
    for (int k = 0; k < 10; ++k) acc[k] = warp_sum_d(acc[k]);
    if (lane == 0) {
        if (energy) energy[s] = acc[0];
        if (virial)
            for (int k = 0; k < 9; ++k) virial[s * 9 + k] = acc[1 + k];
    }
}

void launch_reduce_structs(int32_t n_structs, int64_t max_atoms, const int64_t* atom_off, const double* e_atom,
                           const double* w_atom, double* partial, double* energy, double* virial, cudaStream_t st) {
    if (n_structs == 0) return;
    const unsigned chunks = (unsigned)((max_atoms + RS_ATOMS - 1) / RS_ATOMS);
    for (int32_t s0 = 0; chunks > 0 && s0 < n_structs; s0 += 65535) {    // grid.y is at most 65,535
        const dim3 grid(chunks, (unsigned)std::min<int32_t>(65535, n_structs - s0));
        reduce_partials_kernel<<<grid, RS_THREADS, 0, st>>>(s0, atom_off, e_atom, w_atom, partial);
    }
    reduce_structs_kernel<<<(unsigned)((n_structs * 32 + 127) / 128), 128, 0, st>>>(n_structs, atom_off, partial, energy,
                                                                                    virial);
}

__global__ void scatter_forces_kernel(int64_t n, const int* __restrict__ perm,
                                      const double* __restrict__ f_s, double* __restrict__ forces) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t o = perm[i];
    forces[o * 3 + 0] = f_s[i * 3 + 0];
    forces[o * 3 + 1] = f_s[i * 3 + 1];
    forces[o * 3 + 2] = f_s[i * 3 + 2];
}

void launch_scatter_forces(int64_t n, const int* perm, const double* f_s, double* forces,
                           cudaStream_t st) {
    if (n == 0 || !forces) return;
    scatter_forces_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, perm, f_s, forces);
}

}  // namespace sn
