// Forward tensor-product convolution of one interaction block (Eq. 3, Figure 2b)
// for the evaluation path: radial weights on tcgen05 tensor cores into TMEM, the
// tensor product on FP32 lanes, the segmented sum in registers.
//
// For a path p = (l1, l2, l3) and channel u the message is
//   m_v[m3, u] = sum_{m1,m2} C[m1,m2,m3] T_v[m1,m2,u],
//   T_v[m1,m2,u] = sum_{e into v} w_e[p,u] x_src(e)[m1,u] Y_e[m2],
// so an edge costs N1 (1 + N2) multiply-adds a channel, needs its harmonics (8
// values for degree 2) instead of coupling matrices, and the coupling is applied
// once per receiver.
//
// Work is split by CTA type: up to four units, a unit being a set of paths of one
// l1 over 32 channels.  The W3 rows of a type's units stay in TMEM as the MMA's A
// operand (lane 32 r + lane of tile i = path i of unit r; from shared memory each
// MMA took 42 cycles to read its 4 KB of A), so w^T [channel][edge] of a 32-slot
// chunk lands in TMEM with a lane per channel, where warps 4 q + r read it.  Each CTA streams a contiguous range of receivers
// (balanced by edges); the NQ warp quads take receivers in turn (v mod NQ).  Helper
// warps run ahead: x rows of the senders, harmonics, the pairs' hidden activations
// H2 (into the swizzled B tile) and the MMAs.  Two rings: x rows and harmonics (shared memory), weights (TMEM).  FP32: W3 and H2 enter as three BF16 terms each (24
// mantissa bits), six products, smallest first.
//
// The edges of a receiver are laid out in groups of four (quads_kernel); the last
// group's empty slots carry a zero x row beside its last edge's weights and harmonics.  The inner loop takes a
// group at a time as two packed FP32 pairs.  Each part has one copy of its code
// (the units of a CTA type run different code; with the loop unrolled over two
// groups and three copies of the epilogue the instruction cache missed and the
// l1 = 2 type ran twice as long).
//
// Measured on the middle block of 128x0e+64x1e+32x2e, 24,000 atoms, BF16: 0.70 ms and
// 0.09 ms of radial.cu, against 2.01 ms of the chunked kernel (conv_fwd_tc.cu); FP32,
// 3,000 atoms, whole evaluation 8.26 -> 5.7 ms.  Bound by the consumers' FP32 lanes
// and, for units of l1 = 0 (the fewest multiply-adds per byte of a row), by the row copies.
#include "conv_common.cuh"
#include "packed_fma.cuh"
#include "tmem.cuh"

#include <algorithm>

namespace sn {

constexpr int ST_E = 32;            // edges per chunk (N of the MMA)
constexpr int ST_NQ = 3;            // warp quads
constexpr int ST_NH = 4;            // helper warps (as many work as there are stages of x, if fewer)
constexpr int ST_THREADS = (4 * ST_NQ + ST_NH) * 32;
constexpr int ST_MAX_STAGES = 8;    // x rows and harmonics
constexpr int ST_MAX_W = 7;         // weight buffers
constexpr int ST_SMEM_MAX = 232448;
constexpr int ST_TILE_BYTES = 128 * 128;     // one A tile: 128 rows of 64 BF16
constexpr int ST_A_COLS = 32;                // TMEM columns of an A tile
constexpr int ST_B_BYTES = ST_E * 128;       // one B tile

struct StSmem {
    int b, x, y, dst, bar, misc, total, x_stage;
};
// weight buffers that fit TMEM's 512 columns beside the A tiles
__host__ __device__ inline int st_w_bufs(int tiles, bool bf) {
    const int n = (512 - (bf ? 1 : 3) * tiles * ST_A_COLS) / (tiles * ST_E);
    return n < ST_MAX_W ? n : ST_MAX_W;
}
__host__ __device__ inline StSmem st_smem(int tiles, int row_floats, int lmax, int stages, bool bf) {
    StSmem s;
    const int splits = bf ? 1 : 3, ny = (lmax + 1) * (lmax + 1) - 1;
    int o = 0;
    s.b = o;    o += (stages < ST_NH ? stages : ST_NH) * splits * ST_B_BYTES;
    s.x_stage = ST_E * row_floats * 4;
    s.x = o;    o += stages * s.x_stage;
    s.y = o;    o += stages * ny * ST_E * 4;
    s.dst = o;  o += stages * ST_E;
    s.bar = o;  o += 8 * 2 * (ST_MAX_STAGES + ST_MAX_W + ST_NH);
    s.misc = o; o += 32;
    s.total = o + 1024;              // the base is rounded up to 1,024 bytes
    return s;
}

struct StArgs {                      // launch-wide pointers
    int n_atoms, x_dim, m_dim;
    int64_t cap_pairs;
    const int *row_ptr, *quad_ptr, *src, *pair_of;
    const int2* quads;
    const float4* geom;
    const void* h2;
    const float* x;
    float* m;
    int* flags;
    unsigned wait_limit;             // clock cycles
};

struct StCtx {                       // one CTA's stream
    unsigned char* sm;
    StSmem L;
    int stages, w_bufs, helpers, Q0, Q1;      // Q: groups of four edges of the CTA's receivers
    unsigned tmem, tmem_w;           // A tiles, weight buffers
    uint64_t *full, *empty, *wfull, *wempty, *turn, *bdone;
    volatile int* abort;
    int* issued;                     // per helper: twice its chunks whose MMAs are issued, plus one for row copies ahead of them
};

// A group of up to four consecutive edges of one receiver: x = first edge,
// y = receiver | (edges - 1) << 29 (atoms are fewer than 2^29).
__device__ __forceinline__ int quad_atom(int2 q) { return q.y & 0x1fffffff; }
__device__ __forceinline__ int quad_last(int2 q) { return q.y >> 29; }

// ------------------------------------------------------------- consumers
template <int LMAX, int KIND, int L1, int J>
struct StUnitPaths {
    static constexpr StSets S = st_sets(L1, LMAX, KIND);
    static constexpr PathList P = path_list(L1, LMAX, KIND);
    static constexpr int NP = S.cnt[J];
    __host__ __device__ static constexpr int l2(int i) { return P.l2[S.path[J][i]]; }
    __host__ __device__ static constexpr int l3(int i) { return P.l3[S.path[J][i]]; }
    __host__ __device__ static constexpr int off(int i) {      // sums before path i
        int o = 0;
        for (int k = 0; k < i; ++k) o += st_path_acc(L1, l2(k), l3(k));
        return o;
    }
    __host__ __device__ static constexpr bool uses(int l) {    // harmonics of degree l are read
        for (int k = 0; k < NP; ++k)
            if (l > 0 && l2(k) == l) return true;
        return false;
    }
};

template <int LMAX, int KIND, int L1, int J>
__device__ __forceinline__ void st_unit(const StType& T, const StUnit& U, const StArgs& A, const StCtx& C, int quad,
                                        int r) {
    using UP = StUnitPaths<LMAX, KIND, L1, J>;
    constexpr int N1 = 2 * L1 + 1, NP = UP::NP, NACC = UP::off(NP);
    constexpr int NY = (LMAX + 1) * (LMAX + 1) - 1;
    const int lane = threadIdx.x & 31;
    f32x2 acc[NACC];
#pragma unroll
    for (int i = 0; i < NACC; ++i) acc[i] = 0ull;
    // kept in registers: reloaded from the parameter bank they cost the epilogue
    // about 1,500 cycles a receiver
    int xstep = U.xstep, row = T.row_floats, m_off[NP], m_mul[NP];
    float* const m_lane = A.m + lane;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        m_off[i] = U.m_off[i];
        m_mul[i] = U.m_mul[i];
        asm volatile("" : "+r"(m_off[i]), "+r"(m_mul[i]));
    }
    asm volatile("" : "+r"(xstep), "+r"(row));
    auto finalize = [&](int v) {
        float* mr = m_lane + (size_t)v * A.m_dim;
        static_for<NP>([&](auto Ic) {
            constexpr int i = decltype(Ic)::value;
            constexpr int l2 = UP::l2(i), l3 = UP::l3(i), N2 = 2 * l2 + 1, N3 = 2 * l3 + 1, o = UP::off(i);
            constexpr int na = st_path_acc(L1, l2, l3);
            float Tm[N1 * N2], out[N3];
#pragma unroll
            for (int k = 0; k < N1 * N2; ++k) Tm[k] = 0.0f;
#pragma unroll
            for (int k = 0; k < na; ++k) {
                float lo, hi;
                unpack2(acc[o + k], lo, hi);
                Tm[k] = lo + hi;
                acc[o + k] = 0ull;
            }
            // a scalar product (l3 = 0) kept its one sum in Tm[0]: its coupling is
            // diagonal with equal entries
            CG<L1, l2, l3>::M(Tm, out);
            float* mp = mr + m_off[i];
#pragma unroll
            for (int c = 0; c < N3; ++c) mp[c * m_mul[i]] = out[c];
        });
    };
    auto wait = [&](uint64_t* bar, unsigned phase) { return pipe_wait(bar, phase, C.abort, A.wait_limit); };
    const unsigned tm0 = C.tmem_w + ((unsigned)(32 * r) << 16);
    int cur = -1, s = -1, d = -1, c0 = C.Q0 - ST_E / 4, vq = -1;
    unsigned parity = 0, wparity = 0, mine = 0, tm = 0;
    const float *s_y = nullptr, *s_x = nullptr;
    while (true) {
        bool end = false;
        while (!mine) {                                // done with this chunk: release it, take the next one
            if (s >= 0) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(C.wempty + d);
                    mbar_arrive(C.empty + s);
                }
            }
            c0 += ST_E / 4;
            if (++s == C.stages) { s = 0; parity ^= 1u; }
            if (++d == C.w_bufs) { d = 0; wparity ^= 1u; }
            end = c0 >= C.Q1 || !wait(C.full + s, parity) || !wait(C.wfull + d, wparity);
            if (end) break;
            tc_fence_after();
            s_y = reinterpret_cast<const float*>(C.sm + C.L.y) + s * NY * ST_E;
            s_x = reinterpret_cast<const float*>(C.sm + C.L.x + s * C.L.x_stage) + U.xoff + lane;
            tm = tm0 + d * T.tiles * ST_E;
            // receiver of each group (-1: none)
            vq = lane < ST_E / 4 ? reinterpret_cast<const int*>(C.sm + C.L.dst)[s * (ST_E / 4) + lane] : -1;
            mine = __ballot_sync(0xffffffffu, vq >= 0 && vq % ST_NQ == quad);
        }
        const int q = end ? 0 : __ffs(mine) - 1;
        const int v = end ? -1 : __shfl_sync(0xffffffffu, vq, q);
        if (v != cur) {
            if (cur >= 0) finalize(cur);
            cur = v;
        }
        if (end) break;
        mine &= mine - 1;
        float w[NP][4], x[4][N1];
#pragma unroll
        for (int i = 0; i < NP; ++i) tmem_ld4(tm + i * ST_E + 4 * q, w[i]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int a = 0; a < N1; ++a) x[k][a] = s_x[(4 * q + k) * row + a * xstep];
        f32x2 x2[2][N1];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int a = 0; a < N1; ++a) x2[h][a] = pack2(x[2 * h][a], x[2 * h + 1][a]);
        tmem_wait();
#pragma unroll
        for (int i = 0; i < NP; ++i) tmem_tie(w[i]);
        static_for<LMAX + 1>([&](auto Lc) {
            constexpr int l2 = decltype(Lc)::value, N2 = 2 * l2 + 1;
            ulonglong2 y2[N2] = {};
            if constexpr (UP::uses(l2)) {
#pragma unroll
                for (int b = 0; b < N2; ++b)
                    y2[b] = *reinterpret_cast<const ulonglong2*>(s_y + (l2 * l2 - 1 + b) * ST_E + 4 * q);
            }
            static_for<2 * NP>([&](auto Ic) {
                constexpr int i = decltype(Ic)::value / 2, h = decltype(Ic)::value % 2;
                if constexpr (UP::l2(i) == l2) {
                    constexpr int l3 = UP::l3(i), o = UP::off(i);
                    const f32x2 w2 = pack2(w[i][2 * h], w[i][2 * h + 1]);
                    auto y = [&](int b) { return h ? y2[b].y : y2[b].x; };
                    if constexpr (l2 == 0) {
#pragma unroll
                        for (int a = 0; a < N1; ++a) acc[o + a] = fma2(w2, x2[h][a], acc[o + a]);
                    } else if constexpr (L1 == 0) {
                        const f32x2 p = mul2(w2, x2[h][0]);
#pragma unroll
                        for (int b = 0; b < N2; ++b) acc[o + b] = fma2(p, y(b), acc[o + b]);
                    } else if constexpr (l3 == 0) {
                        f32x2 p = mul2(x2[h][0], y(0));
#pragma unroll
                        for (int a = 1; a < N1; ++a) p = fma2(x2[h][a], y(a), p);
                        acc[o] = fma2(w2, p, acc[o]);
                    } else {
#pragma unroll
                        for (int a = 0; a < N1; ++a) {
                            const f32x2 p = mul2(w2, x2[h][a]);
#pragma unroll
                            for (int b = 0; b < N2; ++b)
                                acc[o + a * N2 + b] = fma2(p, y(b), acc[o + a * N2 + b]);
                        }
                    }
                }
            });
        });
    }
}

// ------------------------------------------------------------- helpers
// Helper warp w of nh prepares every nh-th chunk from start to end: edge
// records, x rows, harmonics, H2 into its B tile, MMAs.  The latencies of its
// dependent loads overlap with the other helpers' chunks (one producer warp with
// prefetched registers took 3,800 cycles a chunk, two load latencies among them).
// MMAs are issued in chunk order (the turn barriers): a parity wait tells apart
// only neighbouring phases, and in order chunk j finds chunk j - 1 - w_bufs
// released; the same holds for the stages of x, of which there are at least nh.
template <int LMAX, bool BF>
__device__ __forceinline__ void st_helper(const StType& T, const StArgs& A, const StCtx& C, int wh) {
    constexpr int SPL = BF ? 1 : 3, NY = (LMAX + 1) * (LMAX + 1) - 1, NH2 = BF ? 1 : 2;
    const int lane = threadIdx.x & 31;
    auto wait = [&](uint64_t* bar, unsigned phase) { return pipe_wait(bar, phase, C.abort, A.wait_limit); };
    const unsigned idesc = umma_idesc(128, ST_E);
    const int n_chunks = (C.Q1 - C.Q0 + ST_E / 4 - 1) / (ST_E / 4);
    const int nh = C.helpers;
    if (wh >= n_chunks || wh >= nh) return;
    // lane = slot; an empty slot of a group takes the group's last edge with a zero
    // x row, a missing group the last one
    auto fetch_quad = [&](int c) { return __ldg(A.quads + min(C.Q0 + c * (ST_E / 4) + (lane >> 2), C.Q1 - 1)); };
    int2 quad = fetch_quad(wh);
    int s = wh % C.stages, d = wh % C.w_bufs;
    unsigned round = 0;
    int ahead = 0;                             // 1: row copies of a chunk whose MMAs are not issued
    unsigned par = 1u ^ ((wh / C.stages) & 1u), wpar = 1u ^ ((wh / C.w_bufs) & 1u);   // empty: the first round passes
    for (int j = wh; j < n_chunks; j += nh) {
        const int e = quad.x + min(lane & 3, quad_last(quad));
        const unsigned valid = __ballot_sync(0xffffffffu, (lane & 3) <= quad_last(quad));
        const int v = C.Q0 + j * (ST_E / 4) + (lane >> 2) < C.Q1 ? quad_atom(quad) : -1;
        const int pair = __ldg(A.pair_of + e), src = __ldg(A.src + e);
        const float4 geom = __ldg(A.geom + e);
        float4 hv[8][NH2];                         // H2: lane = (row mod 4, eighth of the row)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int p = __shfl_sync(0xffffffffu, pair, 4 * q + (lane >> 3));
            const int64_t pc = max((int64_t)0, min((int64_t)p, A.cap_pairs - 1));
            const float4* g = reinterpret_cast<const float4*>(A.h2) + (pc * 8 + (lane & 7)) * NH2;
#pragma unroll
            for (int k = 0; k < NH2; ++k) hv[q][k] = __ldg(g + k);
        }
        if (!wait(C.empty + s, par)) break;
        ahead = 1;
        // x rows by bulk copies, a lane a row; zeros in the empty slots
        const int row_bytes = T.row_floats * 4;
        unsigned char* xs = C.sm + C.L.x + s * C.L.x_stage;
        if (lane == 0) mbar_add_tx(C.full + s, (unsigned)(__popc(valid) * row_bytes));
        __syncwarp();
        if ((valid >> lane) & 1u) {
            const float* xr = A.x + (size_t)src * A.x_dim;
            for (int g = 0; g < T.n_seg; ++g)
                for (int k = 0; k < T.seg_n[g]; ++k)
                    bulk_copy(xs + lane * row_bytes + 4 * (T.seg_dst[g] + k * T.seg_floats[g]),
                              xr + T.seg_src[g] + k * T.seg_step[g], (unsigned)(4 * T.seg_floats[g]), C.full + s);
        }
        for (unsigned none = ~valid; none; none &= none - 1)
            for (int i = lane * 16; i < row_bytes; i += 512)
                *reinterpret_cast<float4*>(xs + (__ffs(none) - 1) * row_bytes + i) = make_float4(0.f, 0.f, 0.f, 0.f);
        quad = fetch_quad(j + nh);
        float Y[NY];
        const float inv = 1.0f / geom.w;
        edge_harmonics<LMAX>(geom.x * inv, geom.y * inv, geom.z * inv, Y);
        float* s_y = reinterpret_cast<float*>(C.sm + C.L.y) + s * NY * ST_E;
#pragma unroll
        for (int b = 0; b < NY; ++b) s_y[b * ST_E + lane] = Y[b];
        if ((lane & 3) == 0) reinterpret_cast<int*>(C.sm + C.L.dst)[s * (ST_E / 4) + (lane >> 2)] = v;
        __syncwarp();
        if (lane == 0) mbar_arrive(C.full + s);
        if (round > 0 && !wait(C.bdone + wh, (round - 1) & 1u)) break;    // this helper's B tile is free
        unsigned char* bt = C.sm + C.L.b + wh * SPL * ST_B_BYTES;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int rowi = 4 * q + (lane >> 3), ch = lane & 7;
            unsigned char* to = bt + rowi * 128 + ((ch ^ (rowi & 7)) << 4);
            if constexpr (BF) {
                *reinterpret_cast<float4*>(to) = hv[q][0];
            } else {
                const float vv[8] = {hv[q][0].x, hv[q][0].y, hv[q][0].z, hv[q][0].w,
                                     hv[q][1].x, hv[q][1].y, hv[q][1].z, hv[q][1].w};
                uint32_t t[3][4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {      // v = t0 + t1 + t2, each the BF16 nearest to what is left
                    float a = vv[2 * k], b = vv[2 * k + 1];
#pragma unroll
                    for (int z = 0; z < 3; ++z) {
                        t[z][k] = pack_bf16(a, b);
                        a -= __uint_as_float(t[z][k] << 16);
                        b -= __uint_as_float(t[z][k] & 0xffff0000u);
                    }
                }
#pragma unroll
                for (int z = 0; z < 3; ++z)
                    *reinterpret_cast<uint4*>(to + z * ST_B_BYTES) = make_uint4(t[z][0], t[z][1], t[z][2], t[z][3]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        if (j > 0 && !wait(C.turn + wh, (wh == 0 ? round - 1 : round) & 1u)) break;
        if (!wait(C.wempty + d, wpar)) break;
        tc_fence_after();
        __syncwarp();
        if (elect_one()) {
            const unsigned b0 = smem_u32(bt);
            for (int i = 0; i < T.tiles; ++i) {
                const unsigned to = C.tmem_w + (d * T.tiles + i) * ST_E;
                // FP32: (A term, B term) = (0,2) (2,0) (1,1) (0,1) (1,0) (0,0), one chain of 24 MMAs.
                // Smallest first, so that only the last four truncate at the size of the sum.
                // Messages against 64 bits, 19 blocks of five models of degree 2 and 3: 3.8e-7 to
                // 8.7e-7, 0.95 to 1.00 of the FFMA sums' error on the same edges and within 3 % of
                // the chunked kernels, which add the leading products by FADD.
                constexpr int NPR = BF ? 1 : 6;
                constexpr int pa[6] = {0, 2, 1, 0, 1, 0}, pb[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
                for (int q = 0; q < NPR; ++q) {
                    const int sa = BF ? 0 : pa[q], sb = BF ? 0 : pb[q];
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_bf16_ts(to, C.tmem + (sa * T.tiles + i) * ST_A_COLS + ks * 8,
                                     umma_desc(b0 + sb * ST_B_BYTES + ks * 32), idesc, q + ks > 0);
                }
            }
            umma_commit(C.wfull + d);
            umma_commit(C.bdone + wh);
            mbar_arrive(C.turn + (wh + 1 == nh ? 0 : wh + 1));
        }
        __syncwarp();
        ++round;
        ahead = 0;
        for (s += nh; s >= C.stages; s -= C.stages) par ^= 1u;
        for (d += nh; d >= C.w_bufs; d -= C.w_bufs) wpar ^= 1u;
    }
    if (lane == 0) C.issued[wh] = 2 * (int)round + ahead;
    // no MMA in flight when TMEM is freed, whether or not a wait ran out
    if (round > 0 && !wait(C.bdone + wh, (round - 1) & 1u)) mbar_wait(C.bdone + wh, (round - 1) & 1u, BULK_WAIT_LIMIT);
}

// After a wait ran out, one thread: waits until the last chunk that went through each of
// the n barriers is complete (ahead 0: its MMAs, 1: its row copies).  Chunk j belongs to
// helper j mod nh and uses phase j / n of barrier j mod n; a barrier's chunks are issued in order.
__device__ __noinline__ void st_drain(uint64_t* bars, int n, int nh, const int* issued, int ahead) {
    int top = -1;
    for (int w = 0; w < nh; ++w) {
        const int done = (issued[w] + ahead) / 2;
        if (done > 0) top = max(top, w + (done - 1) * nh);
    }
    for (int b = 0; b < n; ++b)
        for (int j = top; j >= 0; --j)
            if (j % n == b && j / nh < (issued[j % nh] + ahead) / 2) {
                mbar_wait(bars + b, (j / n) & 1, BULK_WAIT_LIMIT / 8);
                break;
            }
}

// First v in [0, n] with row_ptr[v] >= key; one whole warp.
__device__ __forceinline__ int warp_lower_bound(const int* __restrict__ row_ptr, int n, long long key) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;
    while (hi - lo > 32) {
        const int p = lo + (int)((long long)(hi - lo) * (lane + 1) / 33);
        const unsigned below = __ballot_sync(0xffffffffu, (long long)row_ptr[p] < key);
        const int c = __popc(below);
        const int p_lo = __shfl_sync(0xffffffffu, p, c > 0 ? c - 1 : 0), p_hi = __shfl_sync(0xffffffffu, p, c < 32 ? c : 31);
        if (c > 0) lo = p_lo + 1;
        if (c < 32) hi = p_hi;
    }
    const int p = lo + lane;
    return lo + __popc(__ballot_sync(0xffffffffu, p < hi && (long long)row_ptr[p] < key));
}

template <int LMAX, int KIND, bool BF>
__global__ void __launch_bounds__(ST_THREADS, 1)
conv_fwd_stream_kernel(const __grid_constant__ StPlan P, const StArgs A) {
    extern __shared__ unsigned char st_smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ty = 0;
    while (ty + 1 < P.n_types && (int)blockIdx.x >= P.t[ty + 1].cta0) ++ty;
    const StType& T = P.t[ty];
    StCtx C;
    C.sm = st_smem_raw + ((1024u - (smem_u32(st_smem_raw) & 1023u)) & 1023u);
    C.stages = P.stages;
    C.L = st_smem(T.tiles, T.row_floats, LMAX, P.stages, BF);
    C.w_bufs = st_w_bufs(T.tiles, BF);
    C.helpers = min(ST_NH, C.stages);
    C.full = reinterpret_cast<uint64_t*>(C.sm + C.L.bar);
    C.empty = C.full + ST_MAX_STAGES;
    C.wfull = C.empty + ST_MAX_STAGES;
    C.wempty = C.wfull + ST_MAX_W;
    C.turn = C.wempty + ST_MAX_W;
    C.bdone = C.turn + ST_NH;
    int* misc = reinterpret_cast<int*>(C.sm + C.L.misc);       // [0] abort, [1] tmem, [2..3] receiver range, [4..7] issued
    C.abort = misc;
    C.issued = misc + 4;
    const int nb = T.n_cta, b = (int)blockIdx.x - T.cta0;
    if (warp == 0) {
        const long long n_e = A.quad_ptr[A.n_atoms];
        const int v = b == 0 ? 0 : warp_lower_bound(A.quad_ptr, A.n_atoms, n_e * b / nb);
        if (lane == 0) misc[2] = v;
    } else if (warp == 1) {
        const long long n_e = A.quad_ptr[A.n_atoms];
        const int v = b == nb - 1 ? A.n_atoms : warp_lower_bound(A.quad_ptr, A.n_atoms, n_e * (b + 1) / nb);
        if (lane == 0) misc[3] = v;
    } else if (warp == 2) {
        if (lane == 0) {
            misc[0] = 0;
            for (int s = 0; s < P.stages; ++s) {
                mbar_init(C.full + s, 1);
                mbar_init(C.empty + s, T.n_units * ST_NQ);
            }
            for (int d = 0; d < C.w_bufs; ++d) {
                mbar_init(C.wfull + d, 1);
                mbar_init(C.wempty + d, T.n_units * ST_NQ);
            }
            for (int w = 0; w < ST_NH; ++w) {
                C.issued[w] = 0;
                mbar_init(C.turn + w, 1);
                mbar_init(C.bdone + w, 1);
            }
        }
    } else if (warp == 3) {
        tmem_alloc(reinterpret_cast<unsigned*>(misc + 1), 512);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    C.tmem = (unsigned)misc[1];
    C.tmem_w = C.tmem + (BF ? 1 : 3) * T.tiles * ST_A_COLS;
    if (warp < 4) {                              // the A tiles: lane's row of every tile
        const uint4* src = reinterpret_cast<const uint4*>(T.w3) + (size_t)(32 * warp + lane) * 8;
        for (int i = 0; i < (BF ? 1 : 3) * T.tiles; ++i) {
            uint32_t a[32];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint4 q = __ldg(src + (size_t)i * 128 * 8 + k);
                a[4 * k] = q.x;
                a[4 * k + 1] = q.y;
                a[4 * k + 2] = q.z;
                a[4 * k + 3] = q.w;
            }
            tmem_st32(C.tmem + ((unsigned)(32 * warp) << 16) + i * ST_A_COLS, a);
        }
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int v0 = misc[2], v1 = misc[3];
    C.Q0 = A.quad_ptr[v0];
    C.Q1 = A.quad_ptr[v1];
    if (warp >= 4 * ST_NQ) {
        st_helper<LMAX, BF>(T, A, C, warp - 4 * ST_NQ);
    } else {
        const int r = warp & 3, quad = warp >> 2;
        if (r < T.n_units) {
            const StUnit& U = T.u[r];
            for (int base = v0 + 32 * quad; base < v1; base += 32 * ST_NQ) {    // receivers without edges
                const int v = base + lane;
                unsigned none = __ballot_sync(0xffffffffu, v < v1 && A.row_ptr[v] == A.row_ptr[v + 1]);
                for (; none; none &= none - 1) {
                    float* mr = A.m + (size_t)(base + __ffs(none) - 1) * A.m_dim + lane;
                    for (int i = 0; i < U.n_paths; ++i)
                        for (int c = 0; c < U.n3[i]; ++c) mr[U.m_off[i] + c * U.m_mul[i]] = 0.0f;
                }
            }
            static_for<LMAX + 1>([&](auto Lc) {
                constexpr int L1 = decltype(Lc)::value;
                static_for<ST_MAX_SETS>([&](auto Jc) {
                    constexpr int J = decltype(Jc)::value;
                    if constexpr (J < st_sets(L1, LMAX, KIND).n) {
                        if (U.l1 == L1 && U.set == J) st_unit<LMAX, KIND, L1, J>(T, U, A, C, quad, r);
                    }
                });
            });
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (misc[0]) {             // a wait ran out: what is in flight ends, the CTA's messages are NaN, and the call reports it
        if (threadIdx.x == 0) {
            st_drain(C.wfull, C.w_bufs, C.helpers, C.issued, 0);
            st_drain(C.full, C.stages, C.helpers, C.issued, 1);
            if (A.flags) atomicOr(A.flags + FLAG_COPY_TIMEOUT, 1);
        }
        for (int v = v0 + warp; v < v1; v += ST_THREADS / 32)
            for (int r = 0; r < T.n_units; ++r)
                for (int i = 0; i < T.u[r].n_paths; ++i)
                    for (int c = 0; c < T.u[r].n3[i]; ++c)
                        A.m[(size_t)v * A.m_dim + T.u[r].m_off[i] + c * T.u[r].m_mul[i] + lane] = __int_as_float(0x7fc00000);
    }
    __syncthreads();
    if (warp == 3) tmem_dealloc(C.tmem, 512);
}

// ------------------------------------------------------------- host side
#define SN_ST_KERNELS(X, LL)                                                              \
    X(LL, 0, false) X(LL, 1, false) X(LL, 2, false) X(LL, 3, false)                       \
    X(LL, 0, true) X(LL, 1, true) X(LL, 2, true) X(LL, 3, true)

sevennet_status st_configure(int lmax) {
#define SN_ST_CFG(LL, KK, BB)                                                                               \
    SN_CUDA(cudaFuncSetAttribute((const void*)conv_fwd_stream_kernel<LL, KK, BB>,                          \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM_MAX));
    if (lmax == 1) { SN_ST_KERNELS(SN_ST_CFG, 1) }
    else if (lmax == 2) { SN_ST_KERNELS(SN_ST_CFG, 2) }
    else { SN_ST_KERNELS(SN_ST_CFG, 3) }
#undef SN_ST_CFG
    return SEVENNET_OK;
}

// The W3 columns of the A operand's rows (-1: none) and their three BF16 terms.
struct StRows { int col[128 * ST_TILES]; };

__global__ void st_pack_kernel(const StRows R, int tiles, const float* __restrict__ W3T, __nv_bfloat16* __restrict__ out) {
    const int i = blockIdx.x * 256 + threadIdx.x, row = i >> 6, k = i & 63;
    const int col = R.col[row];
    float v = col >= 0 ? W3T[(size_t)col * 64 + k] : 0.0f;
    for (int z = 0; z < 3; ++z) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        out[((size_t)z * tiles * 128 + row) * 64 + k] = h;
        v -= __bfloat162float(h);
    }
}

// Units of the block in order of falling l1, four to a CTA type; CTAs shared out
// by the multiply-adds of a type's largest unit plus 34 for the loads and the loop
// around them (a 32-slot chunk measured about 900 + 26 cycles per multiply-add), or
// by its helpers' copies (about 110 cycles of issue each, four helpers) if those
// take longer.  ok = 0 where a type does not fit shared memory: the block then
// keeps the chunked kernels.
struct StU { int l1, set, g; };

static void st_plan_types(const ConvDesc& D, const std::vector<StU>& units, int sms, StPlan (&plan)[2]) {
    using U = StU;
    const int n_types = ((int)units.size() + 3) / 4;
    for (int bf = 0; bf < 2; ++bf) {
        StPlan& P = plan[bf];
        P = StPlan{};
        P.n_types = n_types;
        std::vector<int> cost(n_types, 0);
        int max_fixed = 0;
        bool fits = false;
        for (int t = 0; t < n_types; ++t) {
            StType& T = P.t[t];
            T.n_units = (int16_t)std::min<int>(4, (int)units.size() - 4 * t);
            int row = 0;
            for (int q = 0; q < T.n_units; ++q) {              // pieces of an x row: one run of groups per l1
                const U& u = units[4 * t + q];
                int k = -1;
                for (int g = 0; g < T.n_seg; ++g)
                    if (T.seg_src[g] >= D.x_off[u.l1] && T.seg_src[g] < D.x_off[u.l1] + (2 * u.l1 + 1) * D.mul_in[u.l1]) k = g;
                if (k < 0) {
                    k = T.n_seg++;
                    T.seg_src[k] = D.x_off[u.l1] + 32 * u.g;
                    T.seg_n[k] = 2 * u.l1 + 1;
                    T.seg_step[k] = D.mul_in[u.l1];
                    T.seg_floats[k] = 32;
                }
                const int g0 = (T.seg_src[k] - D.x_off[u.l1]) / 32;
                if (u.g < g0) {
                    T.seg_src[k] -= 32 * (g0 - u.g);
                    T.seg_floats[k] += 32 * (g0 - u.g);
                }
                T.seg_floats[k] = std::max(T.seg_floats[k], 32 * (u.g - std::min(g0, u.g) + 1));
            }
            for (int k = 0; k < T.n_seg; ++k) { T.seg_dst[k] = row; row += T.seg_n[k] * T.seg_floats[k]; }
            T.row_floats = row;
            for (int q = 0; q < T.n_units; ++q) {
                const U& u = units[4 * t + q];
                const StSets S = st_sets(u.l1, D.lmax, D.kind);
                StUnit& V = T.u[q];
                V.l1 = (int16_t)u.l1;
                V.set = (int16_t)u.set;
                V.n_paths = (int16_t)S.cnt[u.set];
                T.tiles = std::max(T.tiles, V.n_paths);
                for (int k = 0; k < T.n_seg; ++k)
                    if (T.seg_src[k] >= D.x_off[u.l1] && T.seg_src[k] < D.x_off[u.l1] + (2 * u.l1 + 1) * D.mul_in[u.l1]) {
                        V.xoff = T.seg_dst[k] + 32 * u.g - (T.seg_src[k] - D.x_off[u.l1]);
                        V.xstep = T.seg_floats[k];
                    }
                for (int i = 0; i < V.n_paths; ++i) {
                    const PathDesc& Q = D.paths[D.pbeg[u.l1] + S.path[u.set][i]];
                    V.m_off[i] = Q.m_off + Q.m_ch0 + 32 * u.g;
                    V.m_mul[i] = Q.m_mul;
                    V.n3[i] = (int16_t)(2 * Q.l3 + 1);
                }
                cost[t] = std::max(cost[t], 34 + st_set_cost(u.l1, D.lmax, D.kind, u.set));
            }
            int copies = 0;
            for (int k = 0; k < T.n_seg; ++k) {                // whole irrep blocks are one copy
                if (T.seg_floats[k] == T.seg_step[k]) {
                    T.seg_floats[k] *= T.seg_n[k];
                    T.seg_n[k] = 1;
                }
                copies += T.seg_n[k];
            }
            cost[t] = std::max(cost[t], 12 + 33 * copies);
            max_fixed = std::max(max_fixed, (int)T.tiles);
        }
        for (int st = ST_MAX_STAGES; st >= 2 && !fits; --st) {
            int need = 0;
            for (int t = 0; t < n_types; ++t) need = std::max(need, st_smem(P.t[t].tiles, P.t[t].row_floats, D.lmax, st, bf).total);
            if (need <= ST_SMEM_MAX && st_w_bufs(max_fixed, bf) >= 2) { fits = true; P.stages = st; P.smem = need; }
        }
        if (!fits) { P.ok = 0; continue; }
        int total = 0, used = 0;
        for (int c : cost) total += c;
        for (int t = 0; t < n_types; ++t) {                    // at least one CTA a type; the rest by cost
            P.t[t].n_cta = std::max(1, (int)((int64_t)sms * cost[t] / total));
            used += P.t[t].n_cta;
        }
        while (used != sms) {
            int best = -1;
            for (int t = 0; t < n_types; ++t) {
                if (used > sms && P.t[t].n_cta <= 1) continue;
                const double c = (double)cost[t] / P.t[t].n_cta;
                if (best < 0 || (used < sms ? c > (double)cost[best] / P.t[best].n_cta : c < (double)cost[best] / P.t[best].n_cta)) best = t;
            }
            P.t[best].n_cta += used < sms ? 1 : -1;
            used += used < sms ? 1 : -1;
        }
        int at = 0;
        for (int t = 0; t < n_types; ++t) { P.t[t].cta0 = at; at += P.t[t].n_cta; }
        P.n_cta = at;
        P.ok = 1;
    }
}

sevennet_status st_plan_build(sevennet_model* M, LayerDev& L, const float* W3T) {
    using U = StU;
    const ConvDesc& D = L.conv;
    L.st[0].ok = L.st[1].ok = 0;
    if (D.H != 64) return SEVENNET_OK;
    const int sms = num_sms(M->device);
    std::vector<StU> units;
    // a type's four units: first the channel groups of a set, so that a type reads
    // whole irrep blocks (one copy a row; a part of a block takes one per component);
    // where such rows are too wide, first the sets of a group
    for (int by_group = 0; by_group < 2 && !(L.st[0].ok && L.st[1].ok); ++by_group) {
        units.clear();
        for (int l1 = D.lmax; l1 >= 0; --l1) {
            const int ns = st_sets(l1, D.lmax, D.kind).n, ng = D.mul_in[l1] / 32;
            if (ns > ST_MAX_SETS) return SEVENNET_OK;
            for (int k = 0; k < ns * ng; ++k)
                units.push_back(by_group ? StU{l1, k % ns, k / ns} : StU{l1, k / ng, k % ng});
        }
        const int n_types = ((int)units.size() + 3) / 4;
        if (n_types < 1 || n_types > ST_MAX_TYPES || sms < n_types) return SEVENNET_OK;
        st_plan_types(D, units, sms, L.st);
    }
    if (!L.st[0].ok && !L.st[1].ok) return SEVENNET_OK;
    const int n_types = L.st[0].n_types;
    // W3 as the A operand: row 32 r + lane of tile i = path i of unit r; three BF16
    // terms, of which the BF16 path reads the first
    for (int t = 0; t < n_types; ++t) {
        const int tiles = L.st[0].t[t].tiles;
        StRows rows;
        for (int& c : rows.col) c = -1;
        for (int q = 0; q < L.st[0].t[t].n_units; ++q) {
            const U& u = units[4 * t + q];
            const StSets S = st_sets(u.l1, D.lmax, D.kind);
            for (int i = 0; i < S.cnt[u.set]; ++i)
                for (int lane = 0; lane < 32; ++lane)
                    rows.col[128 * i + 32 * q + lane] = D.paths[D.pbeg[u.l1] + S.path[u.set][i]].col0 + 32 * u.g + lane;
        }
        void* p = nullptr;
        if (cudaMalloc(&p, (size_t)3 * tiles * ST_TILE_BYTES) != cudaSuccess) {
            cudaGetLastError();
            set_error("cudaMalloc of %d bytes failed", 3 * tiles * ST_TILE_BYTES);
            return SEVENNET_ENOMEM;
        }
        M->allocations.push_back(p);
        st_pack_kernel<<<tiles * 32, 256>>>(rows, tiles, W3T, static_cast<__nv_bfloat16*>(p));
        L.st[0].t[t].w3 = L.st[1].t[t].w3 = p;
    }
    SN_CUDA(cudaGetLastError());
    return SEVENNET_OK;
}

// Bytes of hidden activations reserved per pair (they share memory with the
// gradients, which are dead during the forward): 256 where both precisions of
// every block can stream, 128 where BF16 can, 0 otherwise.  The lines keep the
// workspace from growing much at 64 edges an atom, 32 pairs: BF16 takes 4,096
// bytes an atom, so none from there on; FP32 takes 8,192, and from rows of 7,000
// a workspace grows by 4 % at most (32x0e+32x1e+32x2e, rows of 7,168, 5 blocks: 3 %).
// They are lines of memory, not of time.  FP32, 6,000 atoms, chunked and streaming:
// 32x0e+32x1e+32x2e 3.93 and 3.23 ms; below the line 64x0e+64x1e (8 % more memory)
// 3.07 and 2.25 ms, 96x0e+32x1e 3.09 and 2.24 ms; BF16 below its line 32x0e+32x1e
// 2.04 and 1.61 ms.  At 48 atoms streaming is up to 9 % slower, at 600 even or faster.
int st_h2_bytes(const sevennet_model* M) {
    const int64_t row = st_grad_bytes(M);
    bool ok[2] = {row >= 7000, row >= 4096};
    for (const LayerDev& L : M->layers)
        for (int b = 0; b < 2; ++b) ok[b] = ok[b] && L.st[b].ok;
    return ok[0] && ok[1] ? 256 : (ok[1] ? 128 : 0);
}
int64_t st_grad_bytes(const sevennet_model* M) {
    return (int64_t)M->x_max * 12 + (int64_t)M->y_max * 4 + (int64_t)M->h_max * 8;
}

void launch_conv_fwd_stream(const LayerDev& Ld, sevennet_precision prec, int64_t n_atoms, int64_t cap_pairs,
                            const int* row_ptr, const int* quad_ptr, const int2* quads, const int* src,
                            const float4* geom, const int* pair_of, const void* h2, const float* x, float* m, int* flags,
                            unsigned wait_limit, cudaStream_t st) {
    const bool bf = prec == SEVENNET_BF16;
    const StPlan& P = Ld.st[bf ? 1 : 0];
    if (n_atoms <= 0) return;
    const StArgs A{(int)n_atoms, Ld.conv.x_dim, Ld.conv.m_dim, cap_pairs, row_ptr, quad_ptr, src, pair_of, quads, geom, h2, x, m, flags, wait_limit};
#define SN_ST_RUN(LL, KK, BB)                                                             \
    if (Ld.conv.lmax == LL && Ld.conv.kind == KK && bf == BB) {                           \
        conv_fwd_stream_kernel<LL, KK, BB><<<P.n_cta, ST_THREADS, P.smem, st>>>(P, A);    \
        return;                                                                           \
    }
    SN_ST_KERNELS(SN_ST_RUN, 1)
    SN_ST_KERNELS(SN_ST_RUN, 2)
    SN_ST_KERNELS(SN_ST_RUN, 3)
#undef SN_ST_RUN
}

// Groups of up to four consecutive edges of a receiver, in order.
__global__ void quads_kernel(int64_t n, const int* __restrict__ row_ptr, const int* __restrict__ quad_ptr,
                             int2* __restrict__ quads) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t v = i >> 3;                              // eight lanes a receiver
    if (v >= n) return;
    const int e0 = row_ptr[v], e1 = row_ptr[v + 1], q0 = quad_ptr[v];
    for (int q = (int)(i & 7); e0 + 4 * q < e1; q += 8)
        quads[q0 + q] = make_int2(e0 + 4 * q, (int)v | ((min(4, e1 - e0 - 4 * q) - 1) << 29));
}

void launch_quads(int64_t n_atoms, const int* row_ptr, const int* quad_ptr, int2* quads, cudaStream_t st) {
    if (n_atoms > 0)
        quads_kernel<<<(unsigned)((n_atoms * 8 + 255) / 256), 256, 0, st>>>(n_atoms, row_ptr, quad_ptr, quads);
}

// The pair of every edge: its own where it stands for the pair, else its reverse's.
__global__ void pair_of_kernel(int64_t n_atoms, const int* __restrict__ row_ptr, const int* __restrict__ rev,
                               const int* __restrict__ pair_ptr, const int* __restrict__ p_e,
                               int* __restrict__ pair_of) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= pair_ptr[n_atoms]) return;
    const int e = p_e[p];
    pair_of[e] = (int)p;
    pair_of[rev[e]] = (int)p;
}

void launch_pair_of(int64_t cap_pairs, int64_t n_atoms, const int* row_ptr, const int* rev, const int* pair_ptr,
                    const int* p_e, int* pair_of, cudaStream_t st) {
    if (cap_pairs > 0)
        pair_of_kernel<<<(unsigned)((cap_pairs + 255) / 256), 256, 0, st>>>(n_atoms, row_ptr, rev, pair_ptr, p_e, pair_of);
}

}  // namespace sn
