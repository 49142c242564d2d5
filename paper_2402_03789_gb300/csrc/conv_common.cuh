// Shared device code of the tensor-product convolution (forward: conv_fwd.cu,
// adjoint: conv_bwd.cu).
//
// Tensor-product convolution of one interaction block and its adjoint.
//
// Forward (paper Eq. 3, Figure 2b; SevenNet-0 details Sec. 5.1):
//   m_v[p][m3, u] = sum_{e into v} w_e[p, u] sum_{m1} x_src(e)[l1][m1, u] G_e^p[m1, m3]
//   G_e^p[m1, m3] = sum_{m2} C_p[m1, m2, m3] Y_l2(d_e)[m2],
//   w_e = MLP(Bessel(r_e) * envelope(r_e))  (the 1/avg_num_neigh factor is folded into
//   the last MLP weight matrix on the host).
// Adjoint (Eqs. 5-8): given g_m = dE/dm, each edge produces dE/dx_src (scattered
// to the sender as 64-bit fixed-point sums), dE/dw_e -> back through the
// MLP to dE/dr_e, and dE/dY_e; together dE/dd_e, accumulated over blocks.
//
// Forward: one CTA owns a contiguous range of receivers (balanced by edge
// count) and walks its edges, sorted by receiver, in chunks of EC edges.
// Adjoint: one CTA per tile of up to 4 chunks, tiles in edge order.  Per chunk:
//   A  geometry: r, unit vector, Y (l <= 3), Bessel basis x envelope  (FP32)
//   B  radial MLP hidden layers
//   C  G matrices of every path for every edge of the chunk
//   D  w = H2 @ W3 for all W columns into shared memory   (tensor cores)
//   E  forward: each warp owns 32-channel groups of paths and walks the edges,
//      keeping the running sum of the current receiver in registers and writing
//      it once when the receiver changes (segmented sum, no atomics);
//      adjoint: each warp owns edges and walks all paths of that edge.
#pragma once

#include "internal.h"
#include "cg_tables.cuh"

#include <utility>

namespace sn {

struct ConvSmem {
    int w, stage, A1, A2, H2, gH, G, Y, B, gY, src, dst, first, W1, geo, gdp, total;
};

__host__ __device__ inline int rup4(int x) { return (x + 3) & ~3; }

// Index of element (k, e) of an [H][EC] activation tile (EC = 16).  Rows k and
// k + 1 share one 32-word line, and the line is XOR-permuted in 8-word steps by
// t(k) = (4 k / H + k / 2) mod 4.  The MMA fragment loads (the four tq lanes
// read rows H/4 apart) and the accumulator stores (rows 2 tq, 2 tq + 1) then
// touch 32 distinct banks, and four consecutive e stay contiguous and aligned.
template <int H>
__device__ __forceinline__ int hk(int k, int e) {
    const int t = ((k * 4 / H) + (k >> 1)) & 3;
    return ((k >> 1) << 5) | ((((k & 1) << 4) | e) ^ (t << 3));
}

// The staging region holds H1 and dE/dbasis.  dE/dH2 (adjoint) reuses H2, which is
// dead once phase D has run.  The BF16 kernels stay under 97 KB so two CTAs leave
// about 60 KB of each SM's 256 KB to the L1 cache.
__host__ __device__ inline ConvSmem conv_smem_layout(int Wpad, int WpadB, int H, int nG, int ys, bool bwd, bool bf) {
    ConvSmem s;
    int o = 0;
    // [EC][row stride]: BF16 in the BF16 forward; the adjoint also keeps three
    // [H][EC] partials of phase F there
    const int w_bwd = EC * Wpad > 3 * H * EC ? EC * Wpad : 3 * H * EC;
    s.w = o;     o += bwd ? w_bwd : (bf ? EC * WpadB / 2 : EC * Wpad);
    s.stage = o; o += H * EC > MAX_NB * EC ? H * EC : MAX_NB * EC;
    s.A1 = o;    o += H * EC;
    s.A2 = o;    o += H * EC;
    s.H2 = o;    o += H * EC;
    s.gH = s.H2;
    s.G = o;     o += rup4(EC * nG);
    s.Y = o;     o += EC * ys;
    s.B = o;     o += MAX_NB * EC;
    s.gY = o;    o += bwd ? EC * ys : 0;
    s.src = o;   o += EC;
    s.dst = o;   o += EC;
    s.first = o; o += EC;
    s.W1 = o;    o += MAX_NB * H;          // radial MLP input layer, loaded once per CTA
    s.geo = o;   o += 4 * EC;              // (d, r) of the chunk's edges
    s.gdp = o;   o += bwd ? 3 * EC : 0;    // dE/dd of earlier blocks, prefetched (adjoint)
    s.total = o;
    return s;
}

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ float siluf_(float x) { return x * sigmoidf_(x); }
__device__ __forceinline__ float dsiluf_(float x) {
    float s = sigmoidf_(x);
    return s * (1.0f + x * (1.0f - s));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Envelope u(x) and du/dx for x = r / r_c (polynomial cutoff of order p).
__device__ __forceinline__ void envelope(const ConvDesc& D, float xr, float& u, float& du) {
    if (xr >= 1.0f) { u = 0.0f; du = 0.0f; return; }
    float xp1 = 1.0f;                       // x^(p-1)
    for (int i = 0; i < D.poly_p - 1; ++i) xp1 *= xr;
    float xp = xp1 * xr, xp2 = xp * xr, xp3 = xp2 * xr;
    const float p = (float)D.poly_p;
    u = 1.0f - D.env_a * xp + D.env_b * xp2 - D.env_c * xp3;
    du = -D.env_a * p * xp1 + D.env_b * (p + 1.0f) * xp - D.env_c * (p + 2.0f) * xp2;
}

// Real harmonics of degree 1..LMAX of the unit vector (x, y, z), component
// normalised, m = -l..l: Y[0..2] degree 1, Y[3..7] degree 2, Y[8..14] degree 3.
template <int LMAX>
__device__ __forceinline__ void edge_harmonics(float x, float y, float z, float* Y) {
    const float s3 = 1.7320508075688772f, s15 = 3.872983346207417f, s5 = 2.23606797749979f;
    Y[0] = s3 * y; Y[1] = s3 * z; Y[2] = s3 * x;
    if constexpr (LMAX >= 2) {
        Y[3] = s15 * x * y;
        Y[4] = s15 * y * z;
        Y[5] = 0.5f * s5 * (3.0f * z * z - 1.0f);
        Y[6] = s15 * x * z;
        Y[7] = 0.5f * s15 * (x * x - y * y);
    }
    if constexpr (LMAX >= 3) {   // degree 3: the standard real harmonics times sqrt(4 pi)
        const float a3 = 2.0916500663351889f, b3 = 10.246950765959598f;    // sqrt(70)/4, sqrt(105)
        const float c3 = 1.6201851746019651f, d3 = 1.3228756555322954f;    // sqrt(42)/4, sqrt(7)/2
        const float zz5 = 5.0f * z * z;
        Y[8] = a3 * y * (3.0f * x * x - y * y);
        Y[9] = b3 * x * y * z;
        Y[10] = c3 * y * (zz5 - 1.0f);
        Y[11] = d3 * z * (zz5 - 3.0f);
        Y[12] = c3 * x * (zz5 - 1.0f);
        Y[13] = 0.5f * b3 * z * (x * x - y * y);
        Y[14] = a3 * x * (x * x - 3.0f * y * y);
    }
}

// Phase A: Y_l(d/r) (component normalised, m = -l..l) and the enveloped basis.
template <int LMAX>
__device__ __forceinline__ void edge_features(const ConvDesc& D, float4 g, float* Y, float* Bcol,
                                              int bstride) {
    const float r = g.w;
    const float inv = 1.0f / r;
    const float x = g.x * inv, y = g.y * inv, z = g.z * inv;
    Y[0] = 1.0f;
    edge_harmonics<LMAX>(x, y, z, Y + 1);
    if constexpr (LMAX < 2) Y[4] = Y[5] = Y[6] = Y[7] = Y[8] = 0.0f;
    float u, du;
    envelope(D, r / D.r_cut, u, du);
    const float th = 3.14159265358979f * r / D.r_cut;
    float s1, c1;
    sincosf(th, &s1, &c1);
    const float pref = 2.0f / D.r_cut * inv * u;
    float sm = 0.0f, sn = s1;                 // sin((n-1) th), sin(n th)
    for (int n = 0; n < D.n_basis; ++n) {
        Bcol[n * bstride] = pref * sn;
        float nx = 2.0f * c1 * sn - sm;
        sm = sn;
        sn = nx;
    }
}

// G matrices of one path for one edge.
// Floats per edge of the Y and dE/dY tiles (also ConvDesc::ys).
template <int LMAX>
constexpr int y_stride() { return LMAX >= 3 ? 16 : 9; }

// Only the couplings a kernel of degree LMAX can meet are compiled in.
template <int LMAX>
__device__ __forceinline__ void path_G(int kind, const float* Y, float* g) {
#define SN_G(a, b, c) case coupling_kind(a, b, c): CG<a, b, c>::G(Y + (b) * (b), g); break;
    if constexpr (LMAX <= 2) {
        switch (kind) {
            SN_FOR_EACH_COUPLING_L2(SN_G)
            default: break;
        }
    } else {
        switch (kind) {
            SN_FOR_EACH_COUPLING(SN_G)
            default: break;
        }
    }
#undef SN_G
}

// 4-byte asynchronous global -> shared copy (no register staging).
__device__ __forceinline__ void cp_async4(float* s, const float* g) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(s);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async16(float4* s, const float4* g) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(s);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Compile-time loop and the compile-time path list of one input irrep.
template <typename F, int... Is>
__device__ __forceinline__ void static_for_impl(F& f, std::integer_sequence<int, Is...>) {
    (f(std::integral_constant<int, Is>{}), ...);
}

template <int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

template <int L1, int LMAX, int KIND>
struct BlockPaths {
    static constexpr PathList list = path_list(L1, LMAX, KIND);
    static constexpr int begin = path_begin(L1, LMAX, KIND);
};

// ---- phases D and F on tensor cores (mma.sync m16n8k16, FP32 accumulate)
// The per-edge weight tile holds BF16 values in the BF16 forward kernel and
// FP32 values otherwise (the adjoint keeps dE/dw in FP32 beside w).
template <bool BF>
struct WTile {
    using T = float;
};
template <>
struct WTile<true> {
    using T = __nv_bfloat16;
};
__device__ __forceinline__ float wload(const float* p) { return *p; }
__device__ __forceinline__ float wload(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void wstore(float* p, float v) { *p = v; }
__device__ __forceinline__ void wstore(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// The four floats of two packed BF16 pairs (a = (x, y), b = (z, w)).
__device__ __forceinline__ float4 unpack_bf16x4(uint32_t a, uint32_t b) {
    return make_float4(__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u), __uint_as_float(b << 16),
                       __uint_as_float(b & 0xffff0000u));
}

// Operands enter the tensor cores as sums of BF16 terms, each the BF16 value
// nearest to what the terms before it leave.  BF16 path: one term for the
// activations and W3, two for the hidden-layer weights W2 (a single BF16 W2 raised
// the virial error fivefold).  FP32 path: three terms of everything, 24 mantissa
// bits.  Products of terms i and j are taken while i + j is below the larger number
// of terms (six for three terms; those left out are below 2^-24).  The tensor cores
// truncate where an FP32 unit rounds, so the FP32 path keeps their chains short: the
// leading products of a k step start from zero and are added by FADD, the small
// ones run in a chain of their own (in one chain dE/dd was 2.0e-6 off in FP32,
// twice the error of FFMA sums).
template <int NT>
__device__ __forceinline__ void bf16_terms(float x, float y, uint32_t (&t)[NT]) {
#pragma unroll
    for (int z = 0; z < NT; ++z) {
        t[z] = pack_bf16(x, y);
        x -= __uint_as_float(t[z] << 16);
        y -= __uint_as_float(t[z] & 0xffff0000u);
    }
}

// threadIdx.x for one chunk: opaque, so that the addresses made from it are not kept in
// registers across the adjoint's chunks (its BF16 kernel fills 128 a thread, and what
// spills leaves the small L1: 24,000 atoms, adjoints 12.23 ms without, 11.9 ms with it).
__device__ __forceinline__ int chunk_tid() {
    int t = threadIdx.x;
    asm volatile("" : "+r"(t));
    return t;
}

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The reduction order inside one MMA k step is free, so the BF16 products
// below permute k identically in the A and B fragments: lane (g, tq) owns the
// 32-bit words [tq * 2 KSN, (tq + 1) * 2 KSN) of every B row, which makes its B
// operand two contiguous 16-byte loads; k step ks then uses words
// w0 = tq * 2 KSN + 2 ks (first half of the fragment) and w0 + 1 (second half).

// Phase D: w[e][c] = sum_k H2[k][e] W3[k][c]; B operand W3T, NT terms of [W][H].
// Each warp loads the B fragments of BATCH n tiles at once.  FP32: FFMA took 61,440
// multiply-adds an edge on FP32 lanes, more than half of the FP32 adjoint's time.
template <int H, int NT, bool BFT>
__device__ __forceinline__ void chunk_w_gemm(const ConvDesc& D, const ConvSmem& L, float* smem,
                                             const __nv_bfloat16* __restrict__ W3T) {
    constexpr int KSN = H / 16;                // k steps (4 or 2)
    constexpr int NV = KSN / 2;                // 16-byte loads per lane, n tile and term
    constexpr int BATCH = NT == 1 ? 4 : 1;
    static_assert(EC == 16, "one m tile of edges");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, tq = lane & 3;
    const float* s_H2 = smem + L.H2;
    uint32_t af[NT][KSN][4];
#pragma unroll
    for (int ks = 0; ks < KSN; ++ks)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = 2 * (tq * 2 * KSN + 2 * ks) + 2 * (q >> 1), e = g + 8 * (q & 1);
            uint32_t tt[NT];
            bf16_terms<NT>(s_H2[hk<H>(k, e)], s_H2[hk<H>(k + 1, e)], tt);
#pragma unroll
            for (int z = 0; z < NT; ++z) af[z][ks][q] = tt[z];
        }
    const int ntiles = D.W / 8;
    const size_t term = (size_t)D.W * H;
    for (int nb = warp; nb < ntiles; nb += BATCH * CONV_WARPS) {
        uint4 bv[BATCH][NT][NV];
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            const int nt = nb + j * CONV_WARPS;
            if (nt < ntiles) {
#pragma unroll
                for (int z = 0; z < NT; ++z) {
                    const uint4* row = reinterpret_cast<const uint4*>(W3T + z * term + (size_t)(nt * 8 + g) * H);
#pragma unroll
                    for (int v = 0; v < NV; ++v) bv[j][z][v] = __ldg(row + tq * NV + v);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            const int nt = nb + j * CONV_WARPS;
            if (nt >= ntiles) break;
            float c[4] = {}, cs[4] = {};       // leading and small products
#pragma unroll
            for (int ks = 0; ks < KSN; ++ks) {
                float ct[4] = {};
#pragma unroll
                for (int o = NT - 1; o >= 0; --o)
#pragma unroll
                    for (int z = 0; z <= o; ++z) {
                        const uint32_t* bw = reinterpret_cast<const uint32_t*>(bv[j][o - z]);
                        const uint32_t b[2] = {bw[2 * ks], bw[2 * ks + 1]};
                        mma_bf16(o > 0 ? cs : (NT == 3 ? ct : c), af[z][ks], b);
                    }
                if constexpr (NT == 3) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[q] += ct[q];
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] += cs[q];
            const int col = nt * 8 + 2 * tq;
            if constexpr (BFT) {         // BF16 tile [EC][WpadB]
                __nv_bfloat16* s_w = reinterpret_cast<__nv_bfloat16*>(smem + L.w);
                *reinterpret_cast<__nv_bfloat162*>(s_w + g * D.WpadB + col) = __floats2bfloat162_rn(c[0], c[1]);
                *reinterpret_cast<__nv_bfloat162*>(s_w + (g + 8) * D.WpadB + col) =
                    __floats2bfloat162_rn(c[2], c[3]);
            } else {                     // FP32 tile [EC][Wpad]
                float* s_w = smem + L.w;
                *reinterpret_cast<float2*>(s_w + g * D.Wpad + col) = make_float2(c[0], c[1]);
                *reinterpret_cast<float2*>(s_w + (g + 8) * D.Wpad + col) = make_float2(c[2], c[3]);
            }
        }
    }
    __syncthreads();
}

// Phase F: gA2[k][e] = silu'(A2[k][e]) sum_c gw[e][c] W3[c][k]; A operand dE/dw in AT terms, B
// operand W3 in BT terms of [H][W].
// K (the W columns, in blocks of 32) is split between four groups of two warps;
// within a group each warp owns H/16 n tiles of 8 hidden units for the group's
// whole K range, so every output has one writer per group.  Group 0 writes
// dE/dH2; groups 1-3 write partials into the dE/dw tile once every warp is done
// reading it (the adjoint's tile holds at least three [H][EC] partials),
// and the partials are added in group order, so the result does not depend on
// the warps' timing.
// The pair kernel's BF16 dE/dw takes two terms (it is the sum of two directions).
template <int H, int AT, int BT>
__device__ __forceinline__ void chunk_gw_gemm(const ConvDesc& D, const ConvSmem& L, float* smem,
                                              const __nv_bfloat16* __restrict__ W3h) {
    constexpr int G = 4, WPG = CONV_WARPS / G, MT = AT > BT ? AT : BT;
    constexpr int NTW = (H / 8) / WPG;         // n tiles per warp (4 or 2)
    static_assert(EC == 16, "one m tile of edges");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, tq = lane & 3;
    const int grp = warp / WPG, wq = warp % WPG;
    float* s_w = smem + L.w;                   // dE/dw, [EC][Wpad]
    float* s_gH = smem + L.gH;                 // [H][EC]
    const int W = D.W, nkb = W / 32;
    const size_t term = (size_t)W * H;
    const int kb0 = nkb * grp / G, kb1 = nkb * (grp + 1) / G;
    __syncthreads();                           // every warp's dE/dw of phase E is in s_w
    float c[NTW][4];
#pragma unroll
    for (int j = 0; j < NTW; ++j) c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
    for (int kb = kb0; kb < kb1; ++kb) {
        uint4 bv[NTW][BT];
#pragma unroll
        for (int j = 0; j < NTW; ++j)
#pragma unroll
            for (int z = 0; z < BT; ++z)
                bv[j][z] = __ldg(reinterpret_cast<const uint4*>(W3h + z * term + (size_t)((wq * NTW + j) * 8 + g) * W + kb * 32) + tq);
        float ct[NTW][4] = {}, cs[NTW][4] = {};    // FP32: leading and small products of this block
        // k step ks covers words kb*16 + 4 tq + 2 ks (+1): columns 32 kb + 8 tq + 4 ks .. + 3
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            const int c0 = kb * 32 + 8 * tq + 4 * ks;
            const float4 r0 = *reinterpret_cast<const float4*>(s_w + g * D.Wpad + c0);
            const float4 r1 = *reinterpret_cast<const float4*>(s_w + (g + 8) * D.Wpad + c0);
            uint32_t a[4][AT];
            bf16_terms<AT>(r0.x, r0.y, a[0]);
            bf16_terms<AT>(r1.x, r1.y, a[1]);
            bf16_terms<AT>(r0.z, r0.w, a[2]);
            bf16_terms<AT>(r1.z, r1.w, a[3]);
#pragma unroll
            for (int o = MT - 1; o >= 0; --o)
#pragma unroll
                for (int z = 0; z <= o; ++z) {
                    if (z >= AT || o - z >= BT) continue;
                    const uint32_t az[4] = {a[0][z < AT ? z : 0], a[1][z < AT ? z : 0], a[2][z < AT ? z : 0], a[3][z < AT ? z : 0]};
#pragma unroll
                    for (int j = 0; j < NTW; ++j) {
                        const uint32_t* bw = reinterpret_cast<const uint32_t*>(&bv[j][o - z < BT ? o - z : 0]);
                        const uint32_t b[2] = {bw[2 * ks], bw[2 * ks + 1]};
                        mma_bf16(MT < 3 ? c[j] : (o > 0 ? cs[j] : ct[j]), az, b);
                    }
                }
        }
        if constexpr (MT == 3) {
#pragma unroll
            for (int j = 0; j < NTW; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) c[j][q] += ct[j][q] + cs[j][q];
        }
    }
    __syncthreads();                           // the partials overwrite s_w
    float* out = grp == 0 ? s_gH : s_w + (grp - 1) * H * EC;
#pragma unroll
    for (int j = 0; j < NTW; ++j) {
        const int k = (wq * NTW + j) * 8 + 2 * tq;
        out[hk<H>(k, g)] = c[j][0];
        out[hk<H>(k + 1, g)] = c[j][1];
        out[hk<H>(k, g + 8)] = c[j][2];
        out[hk<H>(k + 1, g + 8)] = c[j][3];
    }
    __syncthreads();
    for (int i = t; i < H * EC; i += CONV_THREADS)
        s_gH[i] = (((s_gH[i] + s_w[i]) + s_w[H * EC + i]) + s_w[2 * H * EC + i]) * dsiluf_(smem[L.A2 + i]);
    __syncthreads();
}

// Hidden layer of the radial MLP on tensor cores:
//   out[k_out][e] = sum_k in[k][e] B[k][k_out], B given N-major ([k_out][k]) in BT
//   terms, the input in AT terms.
// The 16 edges of the chunk are one m tile; warps take n tiles of 8 outputs.
template <int H, int BT = 2>
struct HiddenB {                                   // B fragments of one n tile
    uint4 b[BT][H / 32];
};

template <int H, int BT>
__device__ __forceinline__ void hidden_load(const __nv_bfloat16* __restrict__ Bn, int nt, HiddenB<H, BT>& b) {
    constexpr int NV = H / 32;
    const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int z = 0; z < BT; ++z) {
        const uint4* p = reinterpret_cast<const uint4*>(Bn + (size_t)z * H * H + (size_t)(nt * 8 + g) * H) + tq * NV;
#pragma unroll
        for (int v = 0; v < NV; ++v) b.b[z][v] = __ldg(p + v);
    }
}

template <int H, int AT = 1, int BT = 2>
__device__ __forceinline__ void hidden_mma(const float* __restrict__ s_in, const HiddenB<H, BT>& bf, float (&c)[4]) {
    constexpr int KSN = H / 16, MT = AT > BT ? AT : BT;
    const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
    c[0] = c[1] = c[2] = c[3] = 0.f;
    float cs[4] = {};
#pragma unroll
    for (int ks = 0; ks < KSN; ++ks) {
        float ct[4] = {};
        uint32_t a[4][AT];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = 2 * (tq * 2 * KSN + 2 * ks) + 2 * (q >> 1), e = g + 8 * (q & 1);
            bf16_terms<AT>(s_in[hk<H>(k, e)], s_in[hk<H>(k + 1, e)], a[q]);
        }
#pragma unroll
        for (int o = MT - 1; o >= 0; --o)
#pragma unroll
            for (int z = 0; z <= o; ++z) {
                if (z >= AT || o - z >= BT) continue;
                const uint32_t* w = reinterpret_cast<const uint32_t*>(bf.b[o - z < BT ? o - z : 0]);
                const uint32_t az[4] = {a[0][z < AT ? z : 0], a[1][z < AT ? z : 0], a[2][z < AT ? z : 0], a[3][z < AT ? z : 0]};
                const uint32_t b[2] = {w[2 * ks], w[2 * ks + 1]};
                mma_bf16(MT < 3 ? c : (o > 0 ? cs : ct), az, b);
            }
        if constexpr (MT == 3) {
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] += ct[q];
        }
    }
    if constexpr (MT == 3) {
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] += cs[q];
    }
}

// Edge data of one chunk, fetched one chunk ahead by threads 0..EC-1.
struct EdgePrefetch {
    int src = 0, dst = -1, first = 0;           // first: index of the receiver's first edge
    float4 geom = make_float4(0.f, 0.f, 0.f, 1.f);
    __device__ __forceinline__ void fetch(int c0, int E1, const int* __restrict__ dsts,
                                          const int* __restrict__ srcs, const float4* __restrict__ geoms,
                                          const int* __restrict__ row_ptr) {
        const int ge = c0 + (int)threadIdx.x;
        if ((int)threadIdx.x < EC && ge < E1) {
            src = srcs[ge];
            dst = dsts[ge];
            geom = geoms[ge];
            first = __ldg(row_ptr + dst);
        }
    }
};

// Radial MLP input layer into shared memory (once per CTA; the first chunk's
// barrier publishes it).
template <int H>
__device__ __forceinline__ void load_W1(const ConvDesc& D, const ConvSmem& L, float* smem,
                                        const float* __restrict__ W1) {
    for (int i = threadIdx.x; i < D.n_basis * H; i += CONV_THREADS) smem[L.W1 + i] = W1[i];
}

// Phase A: edge records, harmonics and basis of a chunk, thread i < EC edge i
// (published by the next barrier).
template <int LMAX>
__device__ __forceinline__ void chunk_features(const ConvDesc& D, const ConvSmem& L, float* smem, int i,
                                               int c0, int ne, const EdgePrefetch& pf) {
    int* s_src = reinterpret_cast<int*>(smem + L.src);
    int* s_dst = reinterpret_cast<int*>(smem + L.dst);
    float* s_Y = smem + L.Y;
    float* s_B = smem + L.B;       // [NB][EC]
    if (i < ne) {
        s_src[i] = pf.src;
        s_dst[i] = pf.dst;
        reinterpret_cast<int*>(smem + L.first)[i] = pf.first >= c0;   // receiver starts here
        reinterpret_cast<float4*>(smem + L.geo)[i] = pf.geom;
        edge_features<LMAX>(D, pf.geom, s_Y + i * y_stride<LMAX>(), s_B + i, EC);
    } else {
        s_src[i] = 0;
        s_dst[i] = -1;
        reinterpret_cast<float4*>(smem + L.geo)[i] = make_float4(0.f, 0.f, 0.f, 1.f);
        for (int n = 0; n < y_stride<LMAX>(); ++n) s_Y[i * y_stride<LMAX>() + n] = 0.0f;
        for (int n = 0; n < D.n_basis; ++n) s_B[n * EC + i] = 0.0f;
    }
}

// Phases B and C.  Leaves A1/A2/H2/G filled.
template <int H, bool BF, int LMAX>
__device__ __forceinline__ void chunk_hidden(const ConvDesc& D, const ConvSmem& L, float* smem,
                                             const __nv_bfloat16* __restrict__ W2T_h) {
    const int t = threadIdx.x, warp = t >> 5;
    float* s_Y = smem + L.Y;
    float* s_B = smem + L.B;       // [NB][EC]
    constexpr int AT = BF ? 1 : 3, BT = BF ? 2 : 3;
    HiddenB<H, BT> hb;
    // B: A1 = B @ W1 (layout [H][EC]); H1 = silu(A1) lives in the staging area until
    // phase D.  Thread (j, edge group): hidden unit j for EPT consecutive edges.
    float* s_A1 = smem + L.A1;
    float* s_A2 = smem + L.A2;
    float* s_H2 = smem + L.H2;
    float* s_H1 = smem + L.stage;
    {
        constexpr int EPT = EC * H / CONV_THREADS;
        static_assert(EPT == 4 || EPT == 2, "edges per thread of the input layer");
        static_assert(H / 8 <= CONV_WARPS, "one hidden n tile per warp");
        const int j = t % H, e0 = (t / H) * EPT;
        float a[EPT];
#pragma unroll
        for (int q = 0; q < EPT; ++q) a[q] = 0.0f;
        for (int n = 0; n < D.n_basis; ++n) {
            const float wv = smem[L.W1 + n * H + j];
            const float* bn = s_B + n * EC + e0;
#pragma unroll
            for (int q = 0; q < EPT; ++q) a[q] = fmaf(bn[q], wv, a[q]);
        }
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
            const int o = hk<H>(j, e0 + q);
            s_A1[o] = a[q];
            s_H1[o] = siluf_(a[q]);
        }
    }
    // C: G matrices (independent of B)
    float* s_G = smem + L.G;
    for (int i = t; i < EC * D.n_paths; i += CONV_THREADS) {
        const int e = i % EC, p = i / EC;
        path_G<LMAX>(D.paths[p].kind, s_Y + e * y_stride<LMAX>(), s_G + e * D.nG + D.paths[p].g_off);
    }
    __syncthreads();
    if (warp < H / 8) {          // A2 = H1 @ W2, H2 = silu(A2)
        const int lane = t & 31, g = lane >> 2, tq = lane & 3, nt = warp;
        float c[4];
        hidden_load<H, BT>(W2T_h, nt, hb);
        hidden_mma<H, AT, BT>(s_H1, hb, c);
        const int j = nt * 8 + 2 * tq;
        const int o[4] = {hk<H>(j, g), hk<H>(j + 1, g), hk<H>(j, g + 8), hk<H>(j + 1, g + 8)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s_A2[o[q]] = c[q];
            s_H2[o[q]] = siluf_(c[q]);
        }
    }
    __syncthreads();
}

// Receiver range of this CTA, balanced by edges.  The edge count is taken from
// row_ptr[n_atoms] (the host may not know it: asynchronous neighbour builds).
__device__ __forceinline__ void cta_range(int n_atoms, int /*n_edges*/, const int* __restrict__ row_ptr,
                                          int* s_range) {
    if (threadIdx.x == 0) {
        const int n_edges = row_ptr[n_atoms];
        const int nb = gridDim.x, b = blockIdx.x;
        auto lb = [&](long long key) {
            int lo = 0, hi = n_atoms;      // first v in [0, n_atoms] with row_ptr[v] >= key
            while (lo < hi) {
                int mid = (lo + hi) >> 1;
                if ((long long)row_ptr[mid] < key) lo = mid + 1; else hi = mid;
            }
            return lo;
        };
        const long long elo = (long long)n_edges * b / nb;
        const long long ehi = (long long)n_edges * (b + 1) / nb;
        const int v0 = (b == 0) ? 0 : lb(elo);
        const int v1 = (b == nb - 1) ? n_atoms : lb(ehi);
        s_range[0] = v0;
        s_range[1] = v1;
    }
    __syncthreads();
}

// G matrix of one path into registers with 16-byte shared-memory loads
// (every path's G starts on a 16-byte boundary).
template <int NG>
__device__ __forceinline__ void load_G(const float* __restrict__ src, float* G) {
    const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int i = 0; i < (NG + 3) / 4; ++i) {
        const float4 v = s4[i];
        G[4 * i] = v.x;
        G[4 * i + 1] = v.y;
        G[4 * i + 2] = v.z;
        G[4 * i + 3] = v.w;
    }
}

static inline size_t smem_bytes(const ConvDesc& D, int H, bool bwd, bool bf) {
    return (size_t)conv_smem_layout(D.Wpad, D.WpadB, H, D.nG, D.ys, bwd, bf).total * sizeof(float);
}

static inline int conv_grid(int64_t n_atoms, int ctas_per_sm) {
    int dev = 0;
    cudaGetDevice(&dev);
    int g = ctas_per_sm * num_sms(dev);
    if (n_atoms < g) g = (int)(n_atoms > 0 ? n_atoms : 1);
    return g;
}

// Opt a kernel into `need` bytes of dynamic shared memory (never lowering a
// limit granted before in this process).
static inline sevennet_status conv_set_smem(const void* fn, size_t need, size_t* granted) {
    int dev = 0, optin = 0;
    SN_CUDA(cudaGetDevice(&dev));
    SN_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    need = need > *granted ? need : *granted;
    cudaFuncAttributes a{};
    SN_CUDA(cudaFuncGetAttributes(&a, fn));
    SN_CHECK(need + a.sharedSizeBytes <= (size_t)optin, SEVENNET_EINVAL,
             "convolution needs %zu bytes of shared memory, the device allows %d", need, optin);
    SN_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need));
    *granted = need;
    return SEVENNET_OK;
}

}  // namespace sn
