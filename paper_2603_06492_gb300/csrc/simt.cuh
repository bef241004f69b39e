// CUDA-core (SIMT) kernels: exact fp32 FMA, no tensor cores.
//
// These carry the fp32 validation mode end to end and every piece of the bf16
// path that has no tensor-core kernel yet.  Reductions over tokens run in a fixed
// order: dbias, dM and the frequency and phase gradients in fixed chunks whose
// partial results are summed in chunk order, dW, dW_up and dW_down as products
// whose K ranges depend on the shape only.
#pragma once

#include "activations.cuh"
#include "cluster.cuh"

namespace noble {
namespace simt {

// One operand of a product: element (row, k) lives at p[row * ld + k], or at
// p[k * ld + row] when mn is set.  Every contiguous extent and every pitch is
// a multiple of 8 elements and every pointer 16-byte aligned (checked at the
// entry points, or workspace slots), so groups of four consecutive elements
// are read with one 16-byte (fp32) or 8-byte (bf16) load.
struct Operand {
    const void *p;
    int64_t ld;
    int mn;
    int bf;  // elements are bf16 (else fp32)
};
struct Seg {
    Operand A, B;
    int64_t K;
};

// One job of a grouped launch.
//   kGemm       C[m][n] = sum_seg sum_k A(m,k) B(n,k) (+ bias[n]), fp32 FMA; with
//               kchunk < K (one segment) C[z][m][n], pitch ldc = N, of every
//               chunk z of kchunk columns of k
//   kColsum     C[c][o] = sum of X[t][o] over the rows t of 128-row chunk c
//               (X = seg[0].A, M rows, N columns; C fp32, pitch ldc)
//   kTranspose  C[j][i] = A(i,j), a square fp32 matrix of M rows
constexpr int kGemm = 0, kColsum = 1, kTranspose = 2;
constexpr int kColsumRows = 128;
struct Job {
    int kind;
    int64_t M, N;
    Seg seg[2];  // seg[1].K = 0: one segment
    const float *bias;
    void *C;
    int64_t ldc;
    int c_bf;             // C is bf16
    int64_t kchunk;       // kGemm: columns of k per output, seg[0].K if not chunked
    int64_t tiles;        // kGemm: tiles of one output
    int64_t tiles_n;      // kGemm: tiles along N; else column blocks
    int64_t units;        // kGemm: tiles of all chunks, one cluster each; else blocks, one CTA each
    int64_t begin;        // first cluster of the job
};
constexpr int kMaxJobs = 7;
struct Jobs {
    Job j[kMaxJobs];
    int n;
};

// Packed pair of fp32 FMAs (each rounded as fmaf): one issue slot for two, so
// that the shared-memory loads fit beside them.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}

// Loads here are ordinary ones: these kernels are resident, as programmatic
// dependents, while the kernel before them writes what they read after
// griddepcontrol.wait, and the read-only path is defined only for data that stays
// constant as long as the kernel runs.

// Four consecutive elements at byte address p.
__device__ __forceinline__ float4 load4(const char *p, int bf)
{
    if (bf) {
        const uint2 u = *reinterpret_cast<const uint2 *>(p);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return *reinterpret_cast<const float4 *>(p);
}

// An operand tile of ROWS x BK in shared memory, [k][row], rows permuted
// within a k by an XOR with a multiple of four that spreads the four-element
// groups of a K-contiguous operand (one lane per row and group) over the
// banks: neither the transposing stores nor the 16-byte reads conflict.
template <int BK>
__device__ __forceinline__ int tile_row(int k, int row) { return row ^ (k / 4 % (BK / 4) * (128 / BK)); }

// A thread's share of an operand tile: GR groups of four elements along the
// contiguous dimension, global -> registers -> shared.
template <int ROWS, int BK, int THREADS>
struct TileLoad {
    static constexpr int GR = ROWS * BK / 4 / THREADS;
    static constexpr int kRowStep = THREADS / (BK / 4);  // K-contiguous: rows between a thread's groups
    static constexpr int kKStep = THREADS / (ROWS / 4);  // row-contiguous: k between a thread's groups
    static_assert(GR >= 1 && kKStep >= 1, "tile");
    const char *p;         // group 0 of the current k-tile
    int64_t gstep, kstep;  // bytes between groups, and between k-tiles
    int row, k, mn, bf;
    int rows_left;         // rows of the operand from the tile's first one on

    __device__ __forceinline__ void init(const Operand &o, int64_t r0, int64_t rows, int64_t k0, int tid)
    {
        mn = o.mn, bf = o.bf;
        const int es = bf ? 2 : 4;
        rows_left = (int)(rows - r0 < ROWS ? rows - r0 : ROWS);
        if (mn) {
            row = (tid % (ROWS / 4)) * 4, k = tid / (ROWS / 4);
            p = reinterpret_cast<const char *>(o.p) + ((k0 + k) * o.ld + r0 + row) * es;
            gstep = (int64_t)kKStep * o.ld * es, kstep = (int64_t)BK * o.ld * es;
        } else {
            row = tid / (BK / 4), k = (tid % (BK / 4)) * 4;
            p = reinterpret_cast<const char *>(o.p) + ((r0 + row) * o.ld + k0 + k) * es;
            gstep = (int64_t)kRowStep * o.ld * es, kstep = BK * es;
        }
    }
    // the next k-tile, of which kleft >= 1 columns of k exist; zeros elsewhere
    __device__ __forceinline__ void load(float4 (&v)[GR], int kleft)
    {
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            const bool in = mn ? (row < rows_left && k + g * kKStep < kleft) : (row + g * kRowStep < rows_left && k < kleft);
            v[g] = in ? load4(p + g * gstep, bf) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        p += kstep;
    }
    __device__ __forceinline__ void store(float *s, const float4 (&v)[GR]) const
    {
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            if (mn) {
                const int kk = k + g * kKStep;
                *reinterpret_cast<float4 *>(s + kk * ROWS + tile_row<BK>(kk, row)) = v[g];
            } else {
                float *d = s + k * ROWS + tile_row<BK>(k, row + g * kRowStep);
                d[0] = v[g].x, d[ROWS] = v[g].y, d[2 * ROWS] = v[g].z, d[3 * ROWS] = v[g].w;
            }
        }
    }
};

__device__ __forceinline__ void store4(const Job &J, int64_t m, int64_t n, float4 v)
{
    if (J.bias) {
        const float4 b = *reinterpret_cast<const float4 *>(J.bias + n);
        v.x += b.x, v.y += b.y, v.z += b.z, v.w += b.w;
    }
    if (J.c_bf) {
        __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        uint2 q;
        q.x = *reinterpret_cast<uint32_t *>(&lo), q.y = *reinterpret_cast<uint32_t *>(&hi);
        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(J.C) + m * J.ldc + n) = q;
    } else {
        *reinterpret_cast<float4 *>(static_cast<float *>(J.C) + m * J.ldc + n) = v;
    }
}

// Column sums of one 128-row chunk over 64 columns: 16 column quads by
// THREADS / 16 row groups, each group's rows in ascending order, the groups
// added in order.
template <int THREADS>
__device__ __forceinline__ void colsum_block(const Job &J, int64_t unit, float *sm)
{
    constexpr int GROUPS = THREADS / 16;
    const int tid = threadIdx.x, quad = tid % 16, grp = tid / 16;
    const int64_t chunk = unit / J.tiles_n, o = (unit % J.tiles_n) * 64 + quad * 4;
    const int64_t t0 = chunk * kColsumRows;
    const int rows = (int)(J.M - t0 < kColsumRows ? J.M - t0 : kColsumRows);
    const Operand &X = J.seg[0].A;
    const int64_t es = X.bf ? 2 : 4;
    const char *p = reinterpret_cast<const char *>(X.p) + (t0 * X.ld + o) * es;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (o < J.N) {
#pragma unroll 8
        for (int t = grp; t < rows; t += GROUPS) {
            const float4 v = load4(p + t * X.ld * es, X.bf);
            s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
        }
    }
    reinterpret_cast<float4 *>(sm)[tid] = s;
    __syncthreads();
    if (grp == 0 && o < J.N) {
        for (int g = 1; g < GROUPS; ++g) {
            const float4 v = reinterpret_cast<float4 *>(sm)[g * 16 + quad];
            s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
        }
        *reinterpret_cast<float4 *>(static_cast<float *>(J.C) + chunk * J.ldc + o) = s;
    }
}

// A 32 x 32 block of a square fp32 transpose.
template <int THREADS>
__device__ __forceinline__ void transpose_block(const Job &J, int64_t unit, float *sm)
{
    const float *A = static_cast<const float *>(J.seg[0].A.p);
    float *C = static_cast<float *>(J.C);
    const int n = (int)J.M, i0 = (int)(unit / J.tiles_n) * 32, j0 = (int)(unit % J.tiles_n) * 32;
    const int c = threadIdx.x % 32;
    for (int i = threadIdx.x / 32; i < 32; i += THREADS / 32)
        if (i0 + i < n && j0 + c < n) sm[i * 33 + c] = A[(int64_t)(i0 + i) * n + j0 + c];
    __syncthreads();
    for (int j = threadIdx.x / 32; j < 32; j += THREADS / 32)
        if (j0 + j < n && i0 + c < n) C[(int64_t)(j0 + j) * n + i0 + c] = sm[c * 33 + j];
}

// Grouped fp32 GEMM: one 64 x 64 tile per cluster of S CTAs, each of which
// sums one K range (rank S - 1 also the second segment); the partial tiles
// meet through distributed shared memory, rank q adding rows
// [64 q / S, 64 (q + 1) / S) over the ranks in order, so the result does not
// depend on timing.
//
// A thread owns 8 x 4 outputs as 16 packed FMAs per k, its operands for the
// next k read one step ahead.  What bounds it is the FMA rate (128 per clock
// and SM, 77 TFLOP/s measured) and the shared-memory reads beside it.
// Measured on 8192 x 4096 x 1024: 55 TFLOP/s, with plain FMAs 45, with 8 x 8
// outputs and a 128 x 128 tile 55-58 (but 19 against 37 on 1024 x 1024 x 1024,
// whose 64 such tiles leave most of the chip idle), with 8 x 16 outputs 50;
// one 64 x 64 tile kernel of 4 x 4 outputs before it, 17-20.
constexpr int kBM = 64, kBN = 64, kBK = 32, kThreads = 128, kTN = 4;
constexpr int kBlocksPerSm = 4;

__global__ void __launch_bounds__(kThreads, kBlocksPerSm) sgemm_group(const __grid_constant__ Jobs jobs)
{
    constexpr int kTileFloats = kBK * (kBM + kBN);
    static_assert(kBM * kBN <= 2 * kTileFloats, "the partial tile reuses the operand buffers");
    __shared__ __align__(16) float sm[2 * kTileFloats];
    ptx::griddep_wait();
    ptx::griddep_launch();
    const uint32_t rank = cluster::ctarank(), S = cluster::nctarank();
    const int64_t cl = blockIdx.x / S;
    int ji = 0;
    while (ji + 1 < jobs.n && cl >= jobs.j[ji + 1].begin) ++ji;
    const Job &J = jobs.j[ji];
    if (J.kind != kGemm) {
        const int64_t unit = (cl - J.begin) * S + rank;
        if (unit < J.units) {
            if (J.kind == kColsum)
                colsum_block<kThreads>(J, unit, sm);
            else
                transpose_block<kThreads>(J, unit, sm);
        }
        return;  // uniform over the cluster: no other CTA of it waits
    }
    // 32 bits hold every index of a launch: a division takes a quarter of the time
    const uint32_t unit = (uint32_t)(cl - J.begin), tiles = (uint32_t)J.tiles, tiles_n = (uint32_t)J.tiles_n;
    const uint32_t z = unit / tiles, tile = unit % tiles;
    const int m0 = (int)(tile / tiles_n) * kBM, n0 = (int)(tile % tiles_n) * kBN;
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    // warp tile 32 x 32; a thread's rows lr + {0..3, 16..19}, columns lc + {0..3}
    const int lr = (warp % 2) * 32 + (lane / 8) * 4, lc = (warp / 2) * 32 + (lane % 8) * 4;

    uint64_t acc[8][kTN / 2];  // row i of the thread's eight, column pair j
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < kTN / 2; ++j) acc[i][j] = 0ull;

    // k in [kb, ke) of one segment, two tiles deep
    auto segment = [&](const Seg &sg, int64_t kb, int64_t ke) {
        TileLoad<kBM, kBK, kThreads> la;
        TileLoad<kBN, kBK, kThreads> lb;
        float4 va[la.GR], vb[lb.GR];
        int kleft = (int)(ke - kb);
        la.init(sg.A, m0, J.M, kb, tid);
        lb.init(sg.B, n0, J.N, kb, tid);
        la.load(va, kleft);
        lb.load(vb, kleft);
        la.store(sm, va);
        lb.store(sm + kBK * kBM, vb);
        __syncthreads();
        int cur = 0;
#pragma unroll 1
        while (true) {
            const float *sA = sm + cur, *sB = sA + kBK * kBM;
            kleft -= kBK;
            const bool more = kleft > 0;
            if (more) {
                la.load(va, kleft);
                lb.load(vb, kleft);
            }
            float4 fa[2][2], fb[2];
            auto frag = [&](int k, int s) {
                const int pr = tile_row<kBK>(k, lr), pc = tile_row<kBK>(k, lc);
                fa[s][0] = *reinterpret_cast<const float4 *>(sA + k * kBM + pr);
                fa[s][1] = *reinterpret_cast<const float4 *>(sA + k * kBM + (pr ^ 16));
                fb[s] = *reinterpret_cast<const float4 *>(sB + k * kBN + pc);
            };
            frag(0, 0);
#pragma unroll
            for (int k = 0; k < kBK; ++k) {
                const int s = k & 1;
                if (k + 1 < kBK) frag(k + 1, s ^ 1);
                const float av[8] = {fa[s][0].x, fa[s][0].y, fa[s][0].z, fa[s][0].w,
                                     fa[s][1].x, fa[s][1].y, fa[s][1].z, fa[s][1].w};
                const uint64_t b0 = pack2(fb[s].x, fb[s].y), b1 = pack2(fb[s].z, fb[s].w);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint64_t a = pack2(av[i], av[i]);
                    acc[i][0] = fma2(a, b0, acc[i][0]);
                    acc[i][1] = fma2(a, b1, acc[i][1]);
                }
            }
            if (!more) break;
            cur = kTileFloats - cur;
            la.store(sm + cur, va);
            lb.store(sm + cur + kBK * kBM, vb);
            __syncthreads();
        }
        __syncthreads();  // the buffers are free again
    };
    // this rank's K range: whole k-tiles of segment 0 (its chunk z), segment 1 on the last rank
    const int64_t per = (int64_t)(((uint32_t)((J.kchunk + kBK - 1) / kBK) + S - 1) / S) * kBK;
    const int64_t kr = (int64_t)rank * per, kb = z * J.kchunk + kr;
    const int64_t ke = min(kb + min(per, J.kchunk - kr), J.seg[0].K);
    if (kb < ke) segment(J.seg[0], kb, ke);
    if (rank == S - 1 && J.seg[1].K > 0) segment(J.seg[1], 0, J.seg[1].K);

    if (S == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = lr + (i & 3) + (i >> 2) * 16;
            const float2 u = unpack2(acc[i][0]), w = unpack2(acc[i][1]);
            if (m0 + r < J.M && n0 + lc < J.N) store4(J, z * J.M + m0 + r, n0 + lc, make_float4(u.x, u.y, w.x, w.y));
        }
        return;
    }
    // partial tile into this CTA's shared memory, then the sums over the ranks
#pragma unroll
    for (int i = 0; i < 8; ++i)
        *reinterpret_cast<ulonglong2 *>(sm + (lr + (i & 3) + (i >> 2) * 16) * kBN + lc) =
            make_ulonglong2(acc[i][0], acc[i][1]);
    cluster::sync();
    const int rows = kBM / (int)S;
    const uint32_t base = ptx::smem_u32(sm);
    for (int e = tid; e < rows * (kBN / 4); e += kThreads) {
        const int r = (int)rank * rows + e / (kBN / 4), c = e % (kBN / 4) * 4;
        const uint32_t off = base + (uint32_t)(r * kBN + c) * 4u;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t q = 0; q < S; ++q) {
            const float4 v = cluster::ld4(cluster::map_to_rank(off, q));
            s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
        }
        if (m0 + r < J.M && n0 + c < J.N) store4(J, z * J.M + m0 + r, n0 + c, s);
    }
    // no CTA leaves while another still reads its shared memory
    cluster::sync();
}

// Row kernels of the bottleneck.  A thread of the 256 handles one column
// j = tid % r of NT tokens, tid / r + (256 / r) u, so that one load of the mixing
// matrix serves NT tokens; a block covers rows_per_block(r, NT) tokens.  They
// are bound by latency (a chain of r loads and FMAs per output): NT is the
// largest of 1, 2, 4, 8 that leaves two blocks per SM.
constexpr int kRowThreads = 256;
__host__ __device__ constexpr int rows_per_block(int64_t r, int nt) { return (int)(kRowThreads / r) * nt; }

// s[u] = sum_k v[(u G + g) r + k] Mx[k r + j], k ascending, for the thread's NT tokens.
template <int NT>
__device__ __forceinline__ void rows_times_matrix(const float *v, const float *Mx, int r, int j, int g, float (&s)[NT])
{
    const int G = kRowThreads / r;
#pragma unroll
    for (int u = 0; u < NT; ++u) s[u] = 0.f;
#pragma unroll 2
    for (int k = 0; k < r; k += 8) {
        float m[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) m[q] = Mx[(k + q) * r + j];
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float4 *p = reinterpret_cast<const float4 *>(v + (u * G + g) * r + k);
            const float4 x = p[0], y = p[1];
            s[u] = fmaf(x.x, m[0], s[u]), s[u] = fmaf(x.y, m[1], s[u]);
            s[u] = fmaf(x.z, m[2], s[u]), s[u] = fmaf(x.w, m[3], s[u]);
            s[u] = fmaf(y.x, m[4], s[u]), s[u] = fmaf(y.y, m[5], s[u]);
            s[u] = fmaf(y.z, m[6], s[u]), s[u] = fmaf(y.w, m[7], s[u]);
        }
    }
}

// CosNet forward on rows (Eq. 2): from h [T][r] (fp32) computes
//   a = cos(omega1 h + phi1), b = a M, c = cos(omega2 b + phi2)
// and writes b (fp32) and c (TOut), each [T][r].
// With act != act::kCos the two-layer variant of the ablation (Section 4.4):
// a = f(h), b = a M, c = f(b) (activations.cuh).
template <typename TOut, int NT>
__global__ void __launch_bounds__(kRowThreads)
cosnet_fwd_rows(int64_t T, int r, int act, const float *h, const float *om1, const float *ph1, const float *M,
                const float *om2, const float *ph2, float *b_out, TOut *c_out)
{
    __shared__ __align__(16) float a_s[kRowThreads * NT];  // [tokens][r]
    ptx::griddep_wait();
    ptx::griddep_launch();
    const int j = threadIdx.x % r, g = threadIdx.x / r, G = kRowThreads / r;
    const int64_t t0 = (int64_t)blockIdx.x * G * NT + g;
    const bool cosine = act == act::kCos;
    const float w1 = cosine ? om1[j] : 0.f, p1 = cosine ? ph1[j] : 0.f;
    const float w2 = cosine ? om2[j] : 0.f, p2 = cosine ? ph2[j] : 0.f;
    float hv[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) hv[u] = t0 + u * G < T ? h[(t0 + u * G) * r + j] : 0.f;
#pragma unroll
    for (int u = 0; u < NT; ++u)
        a_s[(u * G + g) * r + j] = cosine ? cosf(fmaf(w1, hv[u], p1)) : act::f(act, hv[u]);
    __syncthreads();
    float s[NT];
    rows_times_matrix<NT>(a_s, M, r, j, g, s);
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        const int64_t t = t0 + u * G;
        if (t >= T) continue;
        b_out[t * r + j] = s[u];
        Elem<TOut>::store(c_out + t * r + j, cosine ? cosf(fmaf(w2, s[u], p2)) : act::f(act, s[u]));
    }
}

// One-layer bottleneck on rows, the variants of the ablation (Section 4.4):
// c = cos(omega1 h + phi1) (act::kCos) or c = f(h) (identity, tanh,
// LeakyReLU, GELU; activations.cuh), elementwise over h [T][r] (n = T r).
template <typename TOut>
__global__ void __launch_bounds__(256)
sigma_fwd_rows(int64_t n, int r, int act, const float *h, const float *om1, const float *ph1, TOut *c_out)
{
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(idx % r);
        const float v = h[idx];
        Elem<TOut>::store(c_out + idx, act == act::kCos ? cosf(fmaf(om1[i], v, ph1[i])) : act::f(act, v));
    }
}

// Bottleneck backward on rows (chain rule through Eq. 2).  From saved h, b
// (fp32), dc = dy W_up (fp32) and Mt = M^T computes per token
//   du2 = -sin(u2) dc, db = omega2 du2, da = db M^T, du1 = -sin(u1) da,
//   dh = omega1 du1, a = cos(u1)
// writing dh (TOut), a and db (fp32) [T][r].  With act != act::kCos (two-layer
// variant f(f(h) M)): db = f'(b) dc, du1 = f'(h) da, dh = du1, a = f(h), and
// the sums are zero.  One-layer variants (two == 0): da = dc, no a and db.
// The block's column sums (sum du1*h, sum du1, sum du2*b, sum du2; [4][r])
// overwrite the first four of its own dc rows, which it has read by then: the
// buffer is four rows longer than T, and a block covers at least four tokens.
template <typename TOut, int NT>
__global__ void __launch_bounds__(kRowThreads)
cosnet_bwd_rows(int64_t T, int r, int act, int two, const float *h, const float *b, float *dc, const float *om1,
                const float *ph1, const float *Mt, const float *om2, const float *ph2, TOut *dh_out, float *a_out,
                float *db_out)
{
    __shared__ __align__(16) float db_s[kRowThreads * NT];  // [tokens][r]
    __shared__ float red[4][kRowThreads];
    ptx::griddep_wait();
    ptx::griddep_launch();
    const int j = threadIdx.x % r, g = threadIdx.x / r, G = kRowThreads / r;
    const int64_t t0 = (int64_t)blockIdx.x * G * NT + g;
    const bool cosine = act == act::kCos;
    const float w1 = cosine ? om1[j] : 0.f, p1 = cosine ? ph1[j] : 0.f;
    const float w2 = cosine && two ? om2[j] : 0.f, p2 = cosine && two ? ph2[j] : 0.f;
    float hv[NT], da[NT];
    float so1 = 0.f, sp1 = 0.f, so2 = 0.f, sp2 = 0.f;
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        const int64_t t = t0 + u * G;
        hv[u] = t < T ? h[t * r + j] : 0.f;
        da[u] = t < T ? dc[t * r + j] : 0.f;
    }
    if (two) {
        float bv[NT];
#pragma unroll
        for (int u = 0; u < NT; ++u) bv[u] = t0 + u * G < T ? b[(t0 + u * G) * r + j] : 0.f;
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const int64_t t = t0 + u * G;
            const float du2 = (cosine ? -sinf(fmaf(w2, bv[u], p2)) : act::df(act, bv[u])) * da[u];
            const float dbv = cosine ? w2 * du2 : du2;
            db_s[(u * G + g) * r + j] = dbv;
            if (t < T) db_out[t * r + j] = dbv;
            if (cosine) {
                so2 += du2 * bv[u];
                sp2 += du2;
            }
        }
        __syncthreads();
        rows_times_matrix<NT>(db_s, Mt, r, j, g, da);
    }
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        const int64_t t = t0 + u * G;
        if (t >= T) continue;
        if (cosine) {
            float s1, c1;
            sincosf(fmaf(w1, hv[u], p1), &s1, &c1);
            const float du1 = -s1 * da[u];
            if (two) a_out[t * r + j] = c1;
            Elem<TOut>::store(dh_out + t * r + j, w1 * du1);
            so1 += du1 * hv[u];
            sp1 += du1;
        } else {
            if (two) a_out[t * r + j] = act::f(act, hv[u]);
            Elem<TOut>::store(dh_out + t * r + j, act::df(act, hv[u]) * da[u]);
        }
    }
    red[0][threadIdx.x] = so1, red[1][threadIdx.x] = sp1, red[2][threadIdx.x] = so2, red[3][threadIdx.x] = sp2;
    __syncthreads();
    float *part = dc + (int64_t)blockIdx.x * G * NT * r;
    for (int k = threadIdx.x; k < 4 * r; k += kRowThreads) {
        float s = 0.f;
        for (int q = 0; q < G; ++q) s += red[k / r][q * r + k % r];
        part[k] = s;
    }
}

// Three-layer cosine (the deepest row of the ablation, Section 4.4, Table 5)
// on rows: from h [T][r] (fp32)
//   a = cos(omega1 h + phi1), b = a M, a2 = cos(omega2 b + phi2), b2 = a2 M2,
//   c = cos(omega3 b2 + phi3)
// writing b, b2 (fp32) and c (TOut), each [T][r].  Block: tokens_per_block
// rows; shared memory 2 tokens_per_block r floats.
template <typename TOut>
__global__ void __launch_bounds__(256)
cosnet3_fwd_rows(int64_t T, int r, int tokens_per_block, const float *h, const float *om1, const float *ph1,
                 const float *M, const float *om2, const float *ph2, const float *M2, const float *om3,
                 const float *ph3, float *b_out, float *b2_out, TOut *c_out)
{
    extern __shared__ float sm3[];
    const int n = tokens_per_block * r;
    float *a_s = sm3, *a2_s = sm3 + n;
    const int64_t t0 = (int64_t)blockIdx.x * tokens_per_block;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, i = idx % r;
        const int64_t t = t0 + tt;
        a_s[idx] = t < T ? cosf(fmaf(om1[i], h[t * r + i], ph1[i])) : 0.f;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, j = idx % r;
        const int64_t t = t0 + tt;
        float s = 0.f;
        for (int i = 0; i < r; ++i) s = fmaf(a_s[tt * r + i], M[i * r + j], s);
        a2_s[idx] = cosf(fmaf(om2[j], s, ph2[j]));
        if (t < T) b_out[t * r + j] = s;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, j = idx % r;
        const int64_t t = t0 + tt;
        if (t >= T) continue;
        float s = 0.f;
        for (int i = 0; i < r; ++i) s = fmaf(a2_s[tt * r + i], M2[i * r + j], s);
        b2_out[t * r + j] = s;
        Elem<TOut>::store(c_out + t * r + j, cosf(fmaf(om3[j], s, ph3[j])));
    }
}

// Backward of cosnet3_fwd_rows (chain rule through the three layers): from
// saved h, b, b2 (fp32) and dc = dy W_up (fp32)
//   du3 = -sin(u3) dc, db2 = omega3 du3, da2 = db2 M2^T,
//   du2 = -sin(u2) da2, db = omega2 du2, da = db M^T,
//   du1 = -sin(u1) da, dh = omega1 du1,  a = cos(u1), a2 = cos(u2)
// writing dh (TDh), a, db, a2, db2 (TAct), each [T][r], and per-block column
// sums over the block's tokens in ascending order, part[blk][q][r] with
// q = 0 sum du1*h, 1 sum du1, 2 sum du2*b, 3 sum du2, 4 sum du3*b2, 5 sum du3.
// Shared memory 8 tokens_per_block r floats.
template <typename TDh, typename TAct>
__global__ void __launch_bounds__(256)
cosnet3_bwd_rows(int64_t T, int r, int tokens_per_block, const float *h, const float *b, const float *b2,
                 const float *dc, const float *om1, const float *ph1, const float *M, const float *om2,
                 const float *ph2, const float *M2, const float *om3, const float *ph3, TDh *dh_out,
                 TAct *a_out, TAct *db_out, TAct *a2_out, TAct *db2_out, float *part)
{
    extern __shared__ float sm3[];
    const int n = tokens_per_block * r;
    float *db2_s = sm3, *db_s = sm3 + n;
    float *q_s = sm3 + 2 * n;  // six [tokens_per_block][r] arrays, in the order of part
    const int64_t t0 = (int64_t)blockIdx.x * tokens_per_block;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, j = idx % r;
        const int64_t t = t0 + tt;
        float du3 = 0.f, bv = 0.f;
        if (t < T) {
            bv = b2[t * r + j];
            du3 = -sinf(fmaf(om3[j], bv, ph3[j])) * dc[t * r + j];
        }
        db2_s[idx] = om3[j] * du3;
        q_s[4 * n + idx] = du3 * bv;
        q_s[5 * n + idx] = du3;
        if (t < T) Elem<TAct>::store(db2_out + t * r + j, om3[j] * du3);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, i = idx % r;
        const int64_t t = t0 + tt;
        float du2 = 0.f, bv = 0.f;
        if (t < T) {
            float da2 = 0.f;
            for (int j = 0; j < r; ++j) da2 = fmaf(db2_s[tt * r + j], M2[i * r + j], da2);
            bv = b[t * r + i];
            float s2, c2;
            sincosf(fmaf(om2[i], bv, ph2[i]), &s2, &c2);
            du2 = -s2 * da2;
            Elem<TAct>::store(a2_out + t * r + i, c2);
            Elem<TAct>::store(db_out + t * r + i, om2[i] * du2);
        }
        db_s[idx] = om2[i] * du2;
        q_s[2 * n + idx] = du2 * bv;
        q_s[3 * n + idx] = du2;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int tt = idx / r, i = idx % r;
        const int64_t t = t0 + tt;
        float du1 = 0.f, hv = 0.f;
        if (t < T) {
            float da = 0.f;
            for (int j = 0; j < r; ++j) da = fmaf(db_s[tt * r + j], M[i * r + j], da);
            hv = h[t * r + i];
            float s1, c1;
            sincosf(fmaf(om1[i], hv, ph1[i]), &s1, &c1);
            du1 = -s1 * da;
            Elem<TAct>::store(a_out + t * r + i, c1);
            Elem<TDh>::store(dh_out + t * r + i, om1[i] * du1);
        }
        q_s[idx] = du1 * hv;
        q_s[n + idx] = du1;
    }
    __syncthreads();
    float *pb = part + (int64_t)blockIdx.x * 6 * r;
    for (int k = threadIdx.x; k < 6 * r; k += blockDim.x) {
        const int q = k / r, j = k % r;
        float s = 0.f;
        for (int tt = 0; tt < tokens_per_block; ++tt) s += q_s[q * n + tt * r + j];
        pb[k] = s;
    }
}

// out[k / seg_len][k % seg_len] = sum_p part[p * n + k].
// Block = 8 warps over 32 columns; warp w sums parts [w*P/8, (w+1)*P/8) in
// ascending order, then the 8 warp sums are added in warp order, so the
// result does not depend on scheduling.
struct Outs4 {
    float *p[8];  // up to eight outputs of seg_len elements each
};
__global__ void __launch_bounds__(256) reduce_partials(int64_t nparts, int64_t n, int64_t seg_len,
                                                       const float *part, Outs4 outs)
{
    __shared__ float sm[8][33];
    const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
    const int64_t k = (int64_t)blockIdx.x * 32 + lane;
    const int64_t per = (nparts + 7) / 8;
    const int64_t pb = w * per, pe = min(nparts, pb + per);
    float s = 0.f;
    if (k < n) {
        // eight loads in flight, then added in ascending p
        int64_t p = pb;
        for (; p + 8 <= pe; p += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = part[(p + u) * n + k];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; p < pe; ++p) s += part[p * n + k];
    }
    sm[w][lane] = s;
    __syncthreads();
    if (w == 0 && k < n) {
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) t += sm[i][lane];
        float *dst = outs.p[k / seg_len];
        if (dst) dst[k % seg_len] = t;
    }
}

}  // namespace simt
}  // namespace noble
