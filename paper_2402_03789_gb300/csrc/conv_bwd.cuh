// Adjoint of the tensor-product convolution (Eqs. 5 and 8): given dE/dm,
// dE/dx of the senders and dE/dd of every edge through the tensor product, the
// radial MLP and the edge embedding.  Shared phases live in conv_common.cuh;
// conv_bwd.cu instantiates the per-edge kernel, conv_bwd_pair.cu the one over
// unordered pairs.
#pragma once
#include "conv_common.cuh"

namespace sn {

// ------------------------------------------------------------- adjoint
// Fixed-point add of one dE/dx contribution (order-independent sums); the
// conversion after the kernel reports a sum that received the sentinel.
__device__ __forceinline__ void gx_fixed_add(unsigned long long* p, float v) {
    const long long q = fabsf(v) < GX_LIMIT ? __float2ll_rn(v * GX_SCALE) : GX_SENTINEL;   // exact scaling by 2^36
    atomicAdd(p, (unsigned long long)q);
}

// ------------------------------------------------------------- tensor product
// Units are edges (DIRS = 1) or unordered pairs (DIRS = 2).  An edge e (receiver v,
// sender w, d = r_w + S cell - r_v) and its reverse (receiver w, sender v, -d) share
// the radial weights w_e, which depend on |d| only, and Y_l(-d/r) = (-1)^l Y_l(d/r),
// so G of the reverse is (-1)^l2 G.  The pair kernel runs the radial MLP, the G
// matrices and their adjoints once per pair and the tensor product once per
// direction: direction 0 is e itself, direction 1 takes dE/dm of w times (-1)^l2 and
// x of v, which gives the reverse edge's products expressed through Y(d/r).  dE/dw,
// and dE/dY w.r.t. Y(d/r), are the sums over both directions.
//
// One path, a channel per lane:
//   t[m1] = sum_{m3} G[m1][m3] g[m3],  dE/dw += x[m1] t[m1],  dE/dx[m1] += w t[m1],
//   S[m1][m3] += w x[m1] g[m3] over both directions, and dE/dY += C : S once
// (the coupling applied per direction cost two instructions a coefficient, half of
// the phase's arithmetic).  Y of degree 0 is constant: no S for l2 = 0.
template <int L1, int L2, int L3, int DIRS, int NCH, int OFF, int NG>
__device__ __forceinline__ void tp_bwd_path(const PathDesc& P, int u0, int e, const float (&x)[DIRS * NCH][2 * L1 + 1],
                                            float (&gx)[DIRS * NCH][2 * L1 + 1], const float (&g)[DIRS * NCH][NG],
                                            float* gY, float* s_w, int Wpad, const float* s_G, int nG) {
    constexpr int N1 = 2 * L1 + 1, N3 = 2 * L3 + 1;
    float* wr = s_w + e * Wpad + P.col0 + u0;
    float wv[NCH], gw[NCH];
#pragma unroll
    for (int h = 0; h < NCH; ++h) {
        wv[h] = wr[32 * h];
        gw[h] = 0.0f;
    }
    float G[((N1 * N3 + 3) / 4) * 4];
    load_G<N1 * N3>(s_G + e * nG + P.g_off, G);
    float S[N1 * N3];
#pragma unroll
    for (int a = 0; a < N1; ++a)
#pragma unroll
        for (int k = 0; k < DIRS * NCH; ++k) {
            const int h = k % NCH;
            const bool neg = k >= NCH && (L2 & 1);       // G of the reverse edge
            float t = 0.0f;
#pragma unroll
            for (int c = 0; c < N3; ++c) t = fmaf(G[a * N3 + c], g[k][OFF + c], t);
            if (neg) t = -t;
            gw[h] = fmaf(x[k][a], t, gw[h]);
            gx[k][a] = fmaf(wv[h], t, gx[k][a]);
            if constexpr (L2 > 0) {
                const float wx = (neg ? -wv[h] : wv[h]) * x[k][a];
#pragma unroll
                for (int c = 0; c < N3; ++c)
                    S[a * N3 + c] = k == 0 ? wx * g[0][OFF + c] : fmaf(wx, g[k][OFF + c], S[a * N3 + c]);
            }
        }
    if constexpr (L2 > 0) CG<L1, L2, L3>::S(S, gY + L2 * L2);
#pragma unroll
    for (int h = 0; h < NCH; ++h) wr[32 * h] = gw[h];    // dE/dw of the unit replaces w (same thread, same slot)
}

template <int L1, int LMAX, int KIND>
__host__ __device__ constexpr int tp_g_off(int i) {        // dE/dm values of the paths before path i
    const PathList p = path_list(L1, LMAX, KIND);
    int o = 0;
    for (int k = 0; k < i; ++k) o += 2 * p.l3[k] + 1;
    return o;
}

// All paths of one input irrep l1 over 32 channels of one unit: the channel loads,
// the path descriptors and the CG code resolve at compile time.  Every dE/dm value
// of the block is loaded before the first path.  The pair kernel reads blocked rows
// of dE/dm ([l1][32 channels][path, m3][channel], written by the linear_2 adjoint):
// in the message layout the address arithmetic of its loads was a fifth of the
// kernel's instructions.  24,000 atoms BF16, adjoints of 5 layers: 12.84 ms with a
// load wave per path and C applied per direction, 13.18 ms with S and loads up front
// in the message layout, 12.25 ms with blocked rows.  The per-edge kernel gets dE/dm
// from its caller, in the message layout.  Scalars (at most 3 x 2 registers a path)
// run two channels a lane where 64 are left, which halves their reads of G.
template <int L1, int LMAX, int KIND, int DIRS, int NCH>
__device__ __forceinline__ void tp_bwd_block(const ConvDesc& D, int u0, int e, const int (&recv)[DIRS],
                                             const int (&send)[DIRS], float* gY, float* s_w, const float* s_G,
                                             const float* __restrict__ x, const float* __restrict__ gm,
                                             unsigned long long* __restrict__ gxo) {
    using BP = BlockPaths<L1, LMAX, KIND>;
    constexpr int N1 = 2 * L1 + 1, NG = tp_g_off<L1, LMAX, KIND>(BP::list.n), K = DIRS * NCH;
    const int mul = D.mul_in[L1];
    float xv[K][N1], gx[K][N1], g[K][NG];
#pragma unroll
    for (int q = 0; q < DIRS; ++q) {
        if constexpr (DIRS == 2) {               // blocked rows
            const int lane = u0 & 31;
            const float* gr = gm + (size_t)recv[q] * D.m_dim + D.gb_off[L1] + (u0 - lane) * NG + lane;
#pragma unroll
            for (int h = 0; h < NCH; ++h)
#pragma unroll
                for (int j = 0; j < NG; ++j) g[q * NCH + h][j] = __ldg(gr + 32 * (h * NG + j));
        } else {
            const float* gr = gm + (size_t)recv[q] * D.m_dim + u0;
            static_for<BP::list.n>([&](auto I) {
                constexpr int i = decltype(I)::value, o = tp_g_off<L1, LMAX, KIND>(i), N3 = 2 * BP::list.l3[i] + 1;
                const PathDesc& P = D.paths[BP::begin + i];
#pragma unroll
                for (int c = 0; c < N3; ++c)
#pragma unroll
                    for (int h = 0; h < NCH; ++h)
                        g[q * NCH + h][o + c] = __ldg(gr + P.m_off + P.m_ch0 + c * P.m_mul + 32 * h);
            });
        }
        const float* xr = x + (size_t)send[q] * D.x_dim + D.x_off[L1] + u0;
#pragma unroll
        for (int a = 0; a < N1; ++a)
#pragma unroll
            for (int h = 0; h < NCH; ++h) {
                xv[q * NCH + h][a] = __ldg(xr + a * mul + 32 * h);
                gx[q * NCH + h][a] = 0.0f;
            }
    }
    static_for<BP::list.n>([&](auto I) {
        constexpr int i = decltype(I)::value;
        tp_bwd_path<L1, BP::list.l2[i], BP::list.l3[i], DIRS, NCH, tp_g_off<L1, LMAX, KIND>(i), NG>(
            D.paths[BP::begin + i], u0, e, xv, gx, g, gY, s_w, D.Wpad, s_G, D.nG);
    });
    if (gxo) {                                   // null: the block's dE/dx is not needed
#pragma unroll
        for (int q = 0; q < DIRS; ++q) {
            unsigned long long* o = gxo + (size_t)send[q] * D.x_dim + D.x_off[L1] + u0;
#pragma unroll
            for (int a = 0; a < N1; ++a)
#pragma unroll
                for (int h = 0; h < NCH; ++h) gx_fixed_add(o + a * mul + 32 * h, gx[q * NCH + h][a]);
        }
    }
}

// Phase E for every unit of the chunk, a warp per unit (slot e: receiver s_dst[e],
// sender s_src[e]).
template <int LMAX, int KIND, int DIRS>
__device__ __forceinline__ void tp_bwd_chunk(const ConvDesc& D, int ne, const int* s_dst, const int* s_src,
                                             float* s_w, const float* s_G, float* s_gY,
                                             const float* __restrict__ x, const float* __restrict__ gm,
                                             unsigned long long* __restrict__ gx) {
    const int t = chunk_tid(), lane = t & 31, warp = t >> 5;
    for (int e = warp; e < ne; e += CONV_WARPS) {
        int recv[DIRS], send[DIRS];
        recv[0] = s_dst[e];
        send[0] = s_src[e];
        if constexpr (DIRS == 2) {
            recv[1] = send[0];
            send[1] = recv[0];
        }
        constexpr int NYS = LMAX >= 3 ? 16 : 9;
        float gY[NYS];
#pragma unroll
        for (int i = 0; i < NYS; ++i) gY[i] = 0.0f;
        static_for<LMAX + 1>([&](auto Lc) {
            constexpr int L1 = decltype(Lc)::value;
            if constexpr (BlockPaths<L1, LMAX, KIND>::list.n > 0) {
                int ub = 0;
                if constexpr (L1 == 0 && LMAX <= 2) {    // short paths: two channels a lane
#pragma unroll 1
                    for (; ub + 64 <= D.mul_in[L1]; ub += 64)
                        tp_bwd_block<L1, LMAX, KIND, DIRS, 2>(D, ub + lane, e, recv, send, gY, s_w, s_G, x, gm, gx);
                }
#pragma unroll 1
                for (; ub < D.mul_in[L1]; ub += 32)
                    tp_bwd_block<L1, LMAX, KIND, DIRS, 1>(D, ub + lane, e, recv, send, gY, s_w, s_G, x, gm, gx);
            }
        });
        constexpr int NY = (LMAX + 1) * (LMAX + 1);
#pragma unroll
        for (int i = 1; i < NY; ++i) gY[i] = warp_sum(gY[i]);
        if (lane < NYS) {
            float val = 0.0f;
#pragma unroll
            for (int i = 1; i < NY; ++i) if (lane == i) val = gY[i];
            s_gY[e * y_stride<LMAX>() + lane] = val;
        }
    }
}

// PAIR = false: one unit per edge, records (dst, src, geom) indexed by edge.
// PAIR = true: one unit per unordered pair, records in pair order and eidx[]
// the pair's edge, which receives the pair's whole dE/dd (its reverse keeps 0:
// forces and virials use dE/dd_e - dE/dd_rev(e) only).  *count is the number of
// units (read on the device).
template <int H, bool BF, int LMAX, bool PAIR>
__global__ void __launch_bounds__(CONV_THREADS, conv_ctas_per_sm(LMAX))
conv_bwd_kernel(const ConvDesc D, const float* __restrict__ W1, const __nv_bfloat16* __restrict__ W3T_h, const __nv_bfloat16* __restrict__ W3_h,
                const __nv_bfloat16* __restrict__ W2T_h, const __nv_bfloat16* __restrict__ W2_h,
                int tile_units, const int* __restrict__ count, const int* __restrict__ dst,
                const int* __restrict__ src, const float4* __restrict__ geom, const int* __restrict__ eidx,
                const float* __restrict__ x, const float* __restrict__ gm,
                unsigned long long* __restrict__ gx, float* __restrict__ gd) {
    extern __shared__ float4 smem4[];
    float* smem = reinterpret_cast<float*>(smem4);
    const ConvSmem L = conv_smem_layout(D.Wpad, D.WpadB, H, D.nG, D.ys, true, BF);
    // One tile of tile_units units (edges or pairs) per CTA, CTA k taking tile k:
    // every output is per unit (dE/dd) or an order-independent sum (dE/dx), so
    // tiles need not follow receiver boundaries.  CTAs start in index order as earlier ones
    // finish, so the resident CTAs sweep one narrow window of receivers at a
    // time, and the senders of that window (atoms near it in the cell-list
    // order), their x rows and dE/dx sums, stay in L2.
    __shared__ int s_range[2];
    if (threadIdx.x == 0) {
        const long long n_e = *count, lo = (long long)blockIdx.x * tile_units;
        s_range[0] = (int)min(lo, n_e);
        s_range[1] = (int)min(lo + tile_units, n_e);
    }
    __syncthreads();
    const int E0 = s_range[0], E1 = s_range[1];
    if (E0 >= E1) return;                        // beyond the device-side unit count
    const int* s_src = reinterpret_cast<const int*>(smem + L.src);
    const int* s_dst = reinterpret_cast<const int*>(smem + L.dst);
    float* s_w = smem + L.w;
    float* s_gY = smem + L.gY;
    load_W1<H>(D, L, smem, W1);
    float* s_gdp = smem + L.gdp;
    float* s_gB = smem + L.stage;                // [NB][EC] (phase B keeps H1 there)
    // The next chunk's edge records are copied to shared memory asynchronously
    // (thread e < EC copies edge e), so no registers hold them across a chunk.
    __shared__ float4 s_ngeo[EC], s_pgeo[EC];
    __shared__ int s_nsrc[EC], s_ndst[EC], s_ne[PAIR ? EC : 1], s_ecur[PAIR ? EC : 1], s_pe[PAIR ? EC : 1];
    auto stage = [&](int c) {
        const int t = chunk_tid();
        if (t < EC && c + t < E1) {
            cp_async4(reinterpret_cast<float*>(s_nsrc + t), reinterpret_cast<const float*>(src + c + t));
            cp_async4(reinterpret_cast<float*>(s_ndst + t), reinterpret_cast<const float*>(dst + c + t));
            cp_async16(s_ngeo + t, geom + c + t);
            if constexpr (PAIR) cp_async4(reinterpret_cast<float*>(s_ne + t), reinterpret_cast<const float*>(eidx + c + t));
        }
    };
    // Phase A of the chunk at c, by 16 threads (i = 0..15), from the staged records
    auto features = [&](int c, int i) {
        const int n = min(EC, E1 - c);
        EdgePrefetch pf;
        if (i < n) {
            pf.src = s_nsrc[i];
            pf.dst = s_ndst[i];
            pf.geom = s_ngeo[i];
            if constexpr (PAIR) s_ecur[i] = s_ne[i];
        }
        chunk_features<LMAX>(D, L, smem, i, c, n, pf);
    };
    // G: dE/dd = (dE/dr) u + (I - u u^T) dE/du / r, thread t < EC the unit c + t
    auto finish = [&](int c, int t, const float4* geo, const int* pe) {
        const float4 g = geo[t];
        const float r = g.w, inv = 1.0f / r;
        const float ux = g.x * inv, uy = g.y * inv, uz = g.z * inv;
        float env, denv;
        envelope(D, r / D.r_cut, env, denv);
        denv /= D.r_cut;
        const float th = 3.14159265358979f * r / D.r_cut;
        const float dth = 3.14159265358979f / D.r_cut;
        float s1, c1;
        sincosf(th, &s1, &c1);
        float sm = 0.0f, sn = s1, cm = 1.0f, cn = c1;
        const float k2 = 2.0f / D.r_cut;
        float dEdr = 0.0f;
        for (int n = 0; n < D.n_basis; ++n) {
            const float nn = (float)(n + 1);
            const float f = k2 * sn * inv;
            const float df = k2 * (nn * dth * cn * inv - sn * inv * inv);
            dEdr = fmaf(s_gB[n * EC + t], df * env + f * denv, dEdr);
            const float ns = 2.0f * c1 * sn - sm;
            const float nc = 2.0f * c1 * cn - cm;
            sm = sn; sn = ns; cm = cn; cn = nc;
        }
        const float* gy = s_gY + t * y_stride<LMAX>();
        const float s3 = 1.7320508075688772f, s15 = 3.872983346207417f, s5 = 2.23606797749979f;
        float gux = s3 * gy[3], guy = s3 * gy[1], guz = s3 * gy[2];
        if (D.lmax >= 2) {
            gux += s15 * (uy * gy[4] + uz * gy[7] + ux * gy[8]);
            guy += s15 * (ux * gy[4] + uz * gy[5] - uy * gy[8]);
            guz += s15 * (uy * gy[5] + ux * gy[7]) + 3.0f * s5 * uz * gy[6];
        }
        if constexpr (LMAX >= 3) {   // gradients of the degree-3 polynomials (projected below)
            const float a3 = 2.0916500663351889f, b3 = 10.246950765959598f;
            const float c3 = 1.6201851746019651f, d3 = 1.3228756555322954f;
            const float zz5 = 5.0f * uz * uz - 1.0f;
            gux += gy[9] * 6.0f * a3 * ux * uy + gy[10] * b3 * uy * uz + gy[13] * c3 * zz5 +
                   gy[14] * b3 * ux * uz + gy[15] * 3.0f * a3 * (ux * ux - uy * uy);
            guy += gy[9] * 3.0f * a3 * (ux * ux - uy * uy) + gy[10] * b3 * ux * uz + gy[11] * c3 * zz5 -
                   gy[14] * b3 * uy * uz - gy[15] * 6.0f * a3 * ux * uy;
            guz += gy[10] * b3 * ux * uy + gy[11] * 10.0f * c3 * uy * uz +
                   gy[12] * d3 * (15.0f * uz * uz - 3.0f) + gy[13] * 10.0f * c3 * ux * uz +
                   gy[14] * 0.5f * b3 * (ux * ux - uy * uy);
        }
        const float dot = gux * ux + guy * uy + guz * uz;
        float* o = gd + (size_t)(PAIR ? pe[t] : c + t) * 3;
        o[0] = s_gdp[3 * t] + dEdr * ux + (gux - dot * ux) * inv;
        o[1] = s_gdp[3 * t + 1] + dEdr * uy + (guy - dot * uy) * inv;
        o[2] = s_gdp[3 * t + 2] + dEdr * uz + (guz - dot * uz) * inv;
    };
    stage(E0);
    cp_async_commit();
    cp_async_wait_all();
    // Phases A and G are serial chains of 16 threads, some 2,500 cycles each.  BF16: the
    // first warp runs G of the previous chunk while the second runs A of this one
    // (24,000 atoms, adjoints of 5 layers 12.25 -> 11.9 ms).  FP32, where the other CTA's
    // W3 products fill the SM meanwhile: one after the other (3,000 atoms: 3.55 ms an
    // evaluation, 3.59 ms overlapped).  Results are the same bits either way.
    constexpr bool OVERLAP = BF;
    for (int c0 = E0;; c0 += EC) {
        const int t = chunk_tid(), warp = t >> 5;
        __syncthreads();       // the previous chunk's dE/dbasis and dE/dY; this chunk's records
        if constexpr (OVERLAP) {
            if (c0 > E0 && t < EC && c0 - EC + t < E1) finish(c0 - EC, t, s_pgeo, s_pe);
        }
        if (c0 >= E1) break;
        if (const int i = OVERLAP ? t - 32 : t; i >= 0 && i < EC) features(c0, i);
        const int ne = min(EC, E1 - c0);
        __syncthreads();       // phase A of this chunk
        stage(c0 + EC);        // lands by the wait before phase G
        // dE/dd of the blocks done so far, copied to shared memory for phase G
        if (t < 3 * ne) {
            if constexpr (PAIR) cp_async4(s_gdp + t, gd + (size_t)s_ecur[t / 3] * 3 + t % 3);
            else cp_async4(s_gdp + t, gd + (size_t)c0 * 3 + t);
        }
        cp_async_commit();
        chunk_hidden<H, BF, LMAX>(D, L, smem, W2T_h);
        chunk_w_gemm<H, BF ? 1 : 3, false>(D, L, smem, W3T_h);
        // E: adjoint of the tensor product (path lists fixed per block kind)
        constexpr int DIRS = PAIR ? 2 : 1;
        switch (D.kind) {
            case 0: tp_bwd_chunk<LMAX, 0, DIRS>(D, ne, s_dst, s_src, s_w, smem + L.G, s_gY, x, gm, gx); break;
            case 1: tp_bwd_chunk<LMAX, 1, DIRS>(D, ne, s_dst, s_src, s_w, smem + L.G, s_gY, x, gm, gx); break;
            case 2: tp_bwd_chunk<LMAX, 2, DIRS>(D, ne, s_dst, s_src, s_w, smem + L.G, s_gY, x, gm, gx); break;
            default: tp_bwd_chunk<LMAX, 3, DIRS>(D, ne, s_dst, s_src, s_w, smem + L.G, s_gY, x, gm, gx); break;
        }
        // F: gA2 = (dE/dw @ W3^T) * silu'(A2), then gH1 = gA2 @ W2^T; gA1 = gH1 * silu'(A1); gB = gA1 @ W1^T
        chunk_gw_gemm<H, BF ? (PAIR ? 2 : 1) : 3, BF ? 1 : 3>(D, L, smem, W3_h);
        float* s_gH = smem + L.gH;
        float* s_A1 = smem + L.A1;
        float* s_A2 = smem + L.A2;
        {   // gA1 = (gA2 @ W2^T) * silu'(A1), stored over A2
            constexpr int AT = BF ? (PAIR ? 2 : 1) : 3, BT = BF ? 2 : 3;
            const int lane = t & 31, g = lane >> 2, tq = lane & 3;
            float c[4];
            const int nt = warp;
            if (nt < H / 8) {
                HiddenB<H, BT> hb;
                hidden_load<H, BT>(W2_h, nt, hb);
                hidden_mma<H, AT, BT>(s_gH, hb, c);
                const int k = nt * 8 + 2 * tq;
                const int o[4] = {hk<H>(k, g), hk<H>(k + 1, g), hk<H>(k, g + 8), hk<H>(k + 1, g + 8)};
#pragma unroll
                for (int q = 0; q < 4; ++q) s_A2[o[q]] = c[q] * dsiluf_(s_A1[o[q]]);
            }
        }
        __syncthreads();
        for (int i = t; i < D.n_basis * EC; i += CONV_THREADS) {
            const int n = i / EC, e = i % EC;
            float a = 0.0f;
#pragma unroll 8
            for (int k = 0; k < H; ++k) a = fmaf(s_A2[hk<H>(k, e)], smem[L.W1 + n * H + k], a);
            s_gB[i] = a;
        }
        if constexpr (OVERLAP) {
            if (t < EC) {          // for phase G (read by the same thread)
                s_pgeo[t] = reinterpret_cast<const float4*>(smem + L.geo)[t];
                if constexpr (PAIR) s_pe[t] = s_ecur[t];
            }
        }
        cp_async_wait_all();
        if constexpr (!OVERLAP) {
            __syncthreads();
            if (t < ne) finish(c0, t, reinterpret_cast<const float4*>(smem + L.geo), s_ecur);
        }
    }
}

// ------------------------------------------------------------- host side
template <bool PAIR>
sevennet_status conv_configure_bwd_mode(int H, size_t need) {
    static size_t granted[2][2] = {{0, 0}, {0, 0}};
    const int hi = H == 64 ? 1 : 0;
    if (H == 64) {
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, false, 1, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, true, 1, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, false, 2, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, true, 2, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, false, 3, PAIR>, need, &granted[hi][1]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<64, true, 3, PAIR>, need, &granted[hi][1]));
    } else if (H == 32) {
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<32, false, 1, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<32, true, 1, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<32, false, 2, PAIR>, need, &granted[hi][0]));
        SN_TRY(conv_set_smem((const void*)conv_bwd_kernel<32, true, 2, PAIR>, need, &granted[hi][0]));
    } else {
        set_error("radial MLP hidden width must be 32 or 64");
        return SEVENNET_EINVAL;
    }
    return SEVENNET_OK;
}

// bound: an upper bound on the number of units (the count itself is *count, on
// the device; in an evaluation about half of it).  Tiles of 1..4 chunks (24,000
// atoms: 4 measured fastest, 3 and 6 1 % slower).  FP32: at least 16 waves of tiles by
// the bound, so that the last wave is a small part (8 waves: 1,500 atoms degree 3
// 2.23 against 2.11 ms, 3,000 atoms 3.54 against 3.52).  BF16: 8, because its chunks
// overlap inside a tile (16 waves: 2,777 atoms, one convolution, 0.821 against 0.806 ms).
template <bool PAIR>
void conv_bwd_dispatch(const LayerDev& L, int H, bool bf, int64_t bound, const int* count, const int* dst,
                       const int* src, const float4* geom, const int* eidx, const float* x, const float* gm,
                       unsigned long long* gxq, float* gd, cudaStream_t st) {
    const int lm = L.conv.lmax;
    bound = std::max<int64_t>(bound, 0);
    const int64_t wave = (int64_t)conv_grid(INT64_MAX, conv_ctas_per_sm(lm));
    const int tile = EC * (int)std::min<int64_t>(4, std::max<int64_t>(1, bound / (EC * (bf ? 8 : 16) * wave)));
    const int grid = (int)std::max<int64_t>(1, (bound + tile - 1) / tile);
    const size_t sm = smem_bytes(L.conv, H, true, bf);
#define SN_LB(HH, BB, LL) conv_bwd_kernel<HH, BB, LL, PAIR><<<grid, CONV_THREADS, sm, st>>>(           \
        L.conv, L.mlp0, L.mlp2h, L.mlp2Th, L.mlp1Th, L.mlp1h,       \
        tile, count, dst, src, geom, eidx, x, gm, gxq, gd)
    if (H == 64) {
        if (bf) { if (lm == 3) SN_LB(64, true, 3); else if (lm == 2) SN_LB(64, true, 2); else SN_LB(64, true, 1); }
        else    { if (lm == 3) SN_LB(64, false, 3); else if (lm == 2) SN_LB(64, false, 2); else SN_LB(64, false, 1); }
    } else {
        if (bf) { if (lm == 2) SN_LB(32, true, 2); else SN_LB(32, true, 1); }
        else    { if (lm == 2) SN_LB(32, false, 2); else SN_LB(32, false, 1); }
    }
#undef SN_LB
}

}  // namespace sn
