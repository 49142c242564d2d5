// Hidden layers of the radial MLP (Sec. 5.1), once per unordered pair of edges:
// H2 = silu(silu(B(r) W1) W2), which depends on the distance only, so an edge and
// its reverse share it.
//
// A warp takes 16 pairs (one m tile): the input layer on FP32 lanes, directly in
// the A-fragment layout, the hidden layer on mma.sync with operands split into
// BF16 terms: two each (three products, 16 mantissa bits) in the BF16 path, whose
// result is rounded to BF16; three each (six products, smallest first, 24 bits) in
// the FP32 path.  Output columns are dealt to the n tiles so that a lane's 16
// results are contiguous.  Bound by instruction issue, mostly the 128 SiLUs of a
// pair (one thread a pair with broadcast weights was bound by the shared-memory
// broadcasts: 178 us for 407,000 pairs).
#include "conv_common.cuh"
#include "packed_fma.cuh"

namespace sn {

constexpr int RAD_WARPS = 4, RAD_TILES = 2;              // m tiles of 16 pairs per warp
constexpr int RAD_PAIRS = RAD_WARPS * RAD_TILES * 16;

// W2 as B fragments [term][n tile][k step][lane], three BF16 terms.  Column c of n
// tile t is output (c / 2) * 16 + 2 t + c % 2.
__global__ void radial_pack_kernel(const float* __restrict__ W2T, uint2* __restrict__ out) {
    constexpr int H = 64;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 8 * 4 * 32) return;
    const int ln = i & 31, ks = (i >> 5) & 3, nt = i >> 7, col = ln >> 2;
    const float* w = W2T + ((col >> 1) * 16 + nt * 2 + (col & 1)) * H + ks * 16 + 2 * (ln & 3);
    float v[4] = {w[0], w[1], w[8], w[9]};
    for (int z = 0; z < 3; ++z) {
        const uint2 q = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
        out[z * 1024 + i] = q;
        const float4 t = unpack_bf16x4(q.x, q.y);
        v[0] -= t.x;
        v[1] -= t.y;
        v[2] -= t.z;
        v[3] -= t.w;
    }
}

sevennet_status radial_pack(sevennet_model* M, LayerDev& L, const float* W2T) {
    if (M->H != 64) return SEVENNET_OK;
    void* p = nullptr;
    if (cudaMalloc(&p, 3 * 1024 * sizeof(uint2)) != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc of the radial weights failed");
        return SEVENNET_ENOMEM;
    }
    M->allocations.push_back(p);
    L.mlp1F = static_cast<uint2*>(p);
    radial_pack_kernel<<<8, 128>>>(W2T, L.mlp1F);
    SN_CUDA(cudaGetLastError());
    return SEVENNET_OK;
}

template <bool BF>
__global__ void __launch_bounds__(RAD_WARPS * 32)
radial_kernel(const ConvDesc D, int64_t cap, const int* __restrict__ count, const float4* __restrict__ geom,
              const float* __restrict__ W1, const uint2* __restrict__ W2F, void* __restrict__ out) {
    constexpr int H = 64, SPL = BF ? 2 : 3;
    __shared__ __align__(16) float s_w1[MAX_NB * H];
    __shared__ uint2 s_b[SPL][8][4][32];                 // B fragments [term][n tile][k step][lane]
    const int64_t n = min((int64_t)*count, cap);
    if ((int64_t)blockIdx.x * RAD_PAIRS >= n) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    for (int i = threadIdx.x; i < D.n_basis * H; i += RAD_WARPS * 32) s_w1[i] = W1[i];
    for (int i = threadIdx.x; i < SPL * 8 * 4 * 32; i += RAD_WARPS * 32) (&s_b[0][0][0][0])[i] = __ldg(W2F + i);
    __syncthreads();
#pragma unroll 1
    for (int mt = 0; mt < RAD_TILES; ++mt) {
        const int64_t p0 = (int64_t)blockIdx.x * RAD_PAIRS + (warp * RAD_TILES + mt) * 16;
        if (p0 >= n) return;
        // hidden units ks * 16 + {2 tq, 2 tq + 1, 2 tq + 8, 2 tq + 9} of pairs g and g + 8, packed by two
        f32x2 h[2][8];
        float pref[2], c1[2], sm[2], sn[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float r = geom[min(p0 + g + 8 * q, n - 1)].w;
            float u, du, s1;
            envelope(D, r / D.r_cut, u, du);
            sincosf(3.14159265358979f * r / D.r_cut, &s1, &c1[q]);
            pref[q] = 2.0f / D.r_cut * (1.0f / r) * u;
            sm[q] = 0.0f;                                // sin((n-1) th), sin(n th)
            sn[q] = s1;
#pragma unroll
            for (int k = 0; k < 8; ++k) h[q][k] = 0ull;
        }
        for (int b = 0; b < D.n_basis; ++b) {
            f32x2 v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                v[q] = pack2(pref[q] * sn[q], pref[q] * sn[q]);
                const float nx = 2.0f * c1[q] * sn[q] - sm[q];
                sm[q] = sn[q];
                sn[q] = nx;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const f32x2 w = *reinterpret_cast<const f32x2*>(s_w1 + b * H + (k >> 1) * 16 + (k & 1) * 8 + 2 * tq);
                h[0][k] = fma2(v[0], w, h[0][k]);
                h[1][k] = fma2(v[1], w, h[1][k]);
            }
        }
        uint32_t a[SPL][4][4];                           // A fragments [term][k step]
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float x, y;
                unpack2(h[q][k], x, y);
                x = siluf_(x);
                y = siluf_(y);
#pragma unroll
                for (int z = 0; z < SPL; ++z) {
                    const uint32_t t = pack_bf16(x, y);
                    a[z][k >> 1][2 * (k & 1) + q] = t;
                    x -= __uint_as_float(t << 16);
                    y -= __uint_as_float(t & 0xffff0000u);
                }
            }
        float c[8][4] = {};
        // products of terms i + j = o < SPL; the n tiles are independent chains.  FP32: the
        // leading products of a k step are added by FADD (see conv_common.cuh)
#pragma unroll
        for (int o = SPL - 1; o > 0; --o)
#pragma unroll
            for (int z = 0; z <= o; ++z)
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                    for (int nt = 0; nt < 8; ++nt) {
                        const uint2 b = s_b[o - z][nt][ks][lane];
                        const uint32_t bb[2] = {b.x, b.y};
                        mma_bf16(c[nt], a[z][ks], bb);
                    }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            float t[4][4] = {};
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const uint2 b = s_b[0][nt][ks][lane];
                const uint32_t bb[2] = {b.x, b.y};
                mma_bf16(BF ? c[nt] : t[ks], a[0][ks], bb);
            }
            if constexpr (!BF) {
#pragma unroll
                for (int q = 0; q < 4; ++q) c[nt][q] += (t[0][q] + t[1][q]) + (t[2][q] + t[3][q]);
            }
        }
        float o[2][16];                                  // pairs g, g + 8: outputs tq * 16 + [0, 16)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q >> 1][2 * nt + (q & 1)] = siluf_(c[nt][q]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int64_t p = p0 + g + 8 * q;
            if (p >= n) continue;
            if constexpr (BF) {
                uint4* to = reinterpret_cast<uint4*>(out) + p * 8 + tq * 2;
                to[0] = make_uint4(pack_bf16(o[q][0], o[q][1]), pack_bf16(o[q][2], o[q][3]), pack_bf16(o[q][4], o[q][5]),
                                   pack_bf16(o[q][6], o[q][7]));
                to[1] = make_uint4(pack_bf16(o[q][8], o[q][9]), pack_bf16(o[q][10], o[q][11]),
                                   pack_bf16(o[q][12], o[q][13]), pack_bf16(o[q][14], o[q][15]));
            } else {
                float4* to = reinterpret_cast<float4*>(out) + p * 16 + tq * 4;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    to[k] = make_float4(o[q][4 * k], o[q][4 * k + 1], o[q][4 * k + 2], o[q][4 * k + 3]);
            }
        }
    }
}

void launch_radial(const LayerDev& L, sevennet_precision prec, int64_t cap_pairs, const int* n_pairs,
                   const float4* p_geom, void* h2, cudaStream_t st) {
    if (cap_pairs <= 0) return;
    const unsigned grid = (unsigned)((cap_pairs + RAD_PAIRS - 1) / RAD_PAIRS);
    if (prec == SEVENNET_BF16)
        radial_kernel<true><<<grid, RAD_WARPS * 32, 0, st>>>(L.conv, cap_pairs, n_pairs, p_geom, L.mlp0, L.mlp1F, h2);
    else
        radial_kernel<false><<<grid, RAD_WARPS * 32, 0, st>>>(L.conv, cap_pairs, n_pairs, p_geom, L.mlp0, L.mlp1F, h2);
}

}  // namespace sn
