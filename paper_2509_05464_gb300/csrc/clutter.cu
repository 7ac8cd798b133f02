// clutter.cu -- a6 Casorati Gram, a7 Hermitian eigen-decomposition and
// energy cutoff, a8 clutter projection and power Doppler (Sec. 2.4.2).
//
// The SVD of the Casorati matrix S (pixels x frames) is obtained from the
// eigen-decomposition of its frames x frames Gram matrix G = S^H S
// (eigenvalues sigma^2, eigenvectors = right singular vectors).  Removing
// the k largest components is S_f = S - (S V_k) V_k^H and the power Doppler
// is the mean of |S_f|^2 over frames.  With k << F this is O(P F k) and
// bound by the single read of S.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>

#include <cuda.h>  // driver types only: the two driver calls are fetched at run time

#include "batch.cuh"
#include "fq_internal.cuh"

namespace {

// ------------------------------------------------------------ workspace --
struct ClutterLayout {
    size_t status, G, part, V, Vt, lam, k, hv, tau, big, ii, tc, total;
    int n_chunks;
    int64_t chunk_len;
};

constexpr int kMaxF = 512;      // frames
constexpr int kGramThreads = 256;
constexpr int kGramWideF = 272; // the most frames with panels of 16 pixels, beyond it 8
constexpr int kGramCtas = 3;    // CTAs of the Gram kernel per SM
constexpr int kGramRound = 32;  // pixel chunks are multiples of this

// 4 x 4 complex blocks of the upper triangle (block rows bi <= bj)
__host__ __device__ inline int gram_cols(int F) { return (F + 3) / 4; }
__host__ __device__ inline int gram_blocks(int F) { return gram_cols(F) * (gram_cols(F) + 1) / 2; }
__host__ __device__ inline int gram_parts(int F) { return (gram_blocks(F) + kGramThreads - 1) / kGramThreads; }
__host__ __device__ inline int gram_px(int F) { return F <= kGramWideF ? 16 : 8; }  // pixels per shared-memory panel
// 16-byte units from plane to plane of a panel: half of the banks on, so that the
// copies of a row, which alternate between the planes, meet no other's bank
__host__ __device__ inline int gram_plane(int F) { return (gram_cols(F) + 3) / 8 * 8 + 4; }
size_t gram_smem(int F) { return 2 * (size_t)gram_px(F) * 2 * gram_plane(F) * sizeof(float4); }
size_t gram_smem_upto(int F) { return std::max(gram_smem(F), gram_smem(std::min(F, kGramWideF))); }
// Dynamic shared memory the kernels are opted in to: the most of any call, not
// the call's own, which another thread's smaller call could take back between
// this thread's opt-in and its launch.
constexpr size_t kEigSmemMax = 190 * 1024;
constexpr int kFastMaxK = 48;  // top-k eigenvectors by inverse iteration up to this k

inline size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

int gram_chunks(int64_t P, int F)
{
    // the CTAs that fit (gram_partial_kernel), all in one wave
    int want = kGramCtas * 152 / gram_parts(F);
    int64_t max_chunks = (P + kGramRound - 1) / kGramRound;
    if (want > max_chunks) want = (int)max_chunks;
    if (want < 1) want = 1;
    return want;
}

__host__ __device__ inline bool eig_in_smem(int F) { return (size_t)F * (F + 1) / 2 * sizeof(float2) <= kEigSmemMax; }

// Operand bytes of the tensor-core Gram modes (0 = CUDA-core FP32 Gram).
int tc_esz(int gram_mode) { return gram_mode == FQ_GRAM_BF16 ? 2 : (gram_mode == FQ_GRAM_TF32 ? 4 : 0); }

ClutterLayout layout(int64_t P, int F, int gram_mode = FQ_GRAM_F32, bool force_big = false, int max_chunks = INT_MAX)
{
    ClutterLayout L;
    size_t o = 0;
    const int esz = tc_esz(gram_mode);
    L.status = o; o += 256;
    L.G = o; o += al256(sizeof(float2) * F * F);
    L.n_chunks = std::min(gram_chunks(P, F), max_chunks);
    int64_t per = (P + L.n_chunks - 1) / L.n_chunks;
    L.chunk_len = (per + kGramRound - 1) / kGramRound * kGramRound;
    L.part = o; o += esz ? 0 : al256(sizeof(float2) * (size_t)L.n_chunks * F * F);
    L.tc = o; o += esz ? fqi::gram_tc_workspace_bytes(P, F, esz) : 0;
    L.V = o; o += al256(sizeof(float2) * F * F);
    L.Vt = o; o += al256(sizeof(float2) * F * F);
    L.lam = o; o += al256(sizeof(double) * F);
    L.k = o; o += 256;
    L.hv = o; o += al256(sizeof(float2) * F * F);
    L.tau = o; o += al256(sizeof(float) * F);
    L.big = o; o += (eig_in_smem(F) && !force_big) ? 0 : al256(sizeof(float2) * (size_t)F * (F + 1) / 2);
    L.ii = o; o += al256(sizeof(float) * 6 * (size_t)kFastMaxK * F);
    L.total = o;
    return L;
}

size_t eig_only_bytes(int F)
{
    // status, hv, tau, Vt, k, big
    size_t o = 256 + al256(sizeof(float2) * F * F) + al256(sizeof(float) * F) + al256(sizeof(float2) * F * F) + 256;
    if (!eig_in_smem(F)) o += al256(sizeof(float2) * (size_t)F * (F + 1) / 2);
    return o;
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// ----------------------------------------------------------------- Gram --
// FP32 on the CUDA cores.  A CTA takes a pixel chunk and up to 256 of the
// upper triangle's 4 x 4 complex blocks, one per thread (16 complex sums in
// registers, 64 FMAs per pixel against four 16-byte shared-memory loads).
// It walks the chunk in panels of 16 pixels x F frames, double-buffered with
// cp.async: S is read once per part (2 parts at 100 frames, 5 at 200), and
// only blocks of the triangle are computed (F = 100: 5200 of 5050 products;
// 32 x 32 tiles with 2 x 2 outputs per thread computed 10240 and read two
// 8-byte operands per complex product).  2^21 pixels x 100 frames: 6.9 -> 2.8
// ms; 65536 x 200: 0.60 -> 0.29 ms, with three CTAs per SM (two 3.1; FMA pipe
// 48% busy, the rest issue: four loads, the panels' copies and barriers).  A
// panel row is two planes, columns (4b, 4b + 1) and (4b + 2, 4b + 3), so that the
// 16-byte loads of 32 consecutive blocks are contiguous.
//
// Panels of more than 272 frames hold 8 pixels, so that three CTAs fit as well
// (16 pixels: two, and one from 448 frames on).  There a copy comes with every 64
// FMAs, and its instructions count: a row of the next panel is copied with each
// pixel's sums, one unit a thread from a running address.  65536 x 512: 3.57 ->
// 2.48 ms, x 300: 0.79 -> 0.75 (the same in narrower panels, where few threads
// have a unit of a row, 2^21 x 100: 2.8 -> 3.1).
// BF16 input has to be widened: a thread holds its part of the next panel (at
// most 18 values) in registers while it computes, and writes it out after;
// waiting for the loads first left the SMs idle: 65536 x 220 0.49 -> 0.37 ms, x
// 512 13.6 -> 2.18.
constexpr int kGramHold = 18;
static_assert(16 * kGramWideF <= kGramThreads * kGramHold && 8 * kMaxF <= kGramThreads * kGramHold, "panel values per thread");
static_assert(kMaxF <= 2 * kGramThreads, "two columns of a row per thread");

template <int PX, typename T>
struct GramStage;

// The walk of a thread over the units (two columns, one 16-byte store) of a
// panel by steps of 256, by shared-memory address.
struct GramWalk {
    int U, du, u;
    unsigned row, drow, rowb, plane;  // shared-memory byte addresses
    __device__ __forceinline__ GramWalk(int units, int ps, const float4 *buf) : U(units)
    {
        const int dp = kGramThreads / U, px = threadIdx.x / U;
        du = kGramThreads - dp * U;
        u = threadIdx.x - px * U;
        rowb = 32u * ps;
        plane = 16u * ps - 8u;
        drow = dp * rowb;
        row = (unsigned)__cvta_generic_to_shared(buf) + px * rowb;
    }
    __device__ __forceinline__ unsigned at() const { return row + 8u * u + (u & 1) * plane; }
    __device__ __forceinline__ void next()
    {
        row += drow;
        u += du;
        if (u >= U) {
            u -= U;
            row += rowb;
        }
    }
};

template <int PX>
struct GramStage<PX, float> {
    // wide panels: a row of the next with each pixel's sums; else all copies at once
    static constexpr bool kRows = PX == 8;
    const float *S;
    int F, ps;  // frames, plane stride
    bool wide;  // rows of whole 16-byte units
    const float *src;
    unsigned dst;
    __device__ __forceinline__ GramStage(const float *s, int f, int p) : S(s), F(f), ps(p)
    {
        wide = (F & 1) == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    }
    // start the copy of pixels p0 .. p0 + n - 1 into buf (kRows: by the calls of row() that follow)
    __device__ __forceinline__ void fetch(int64_t p0, int n, float4 *buf)
    {
        const int t = threadIdx.x;
        src = S + (p0 * F + (wide ? 2 * t : t)) * 2;
        const unsigned b = (unsigned)__cvta_generic_to_shared(buf);
        if constexpr (kRows) {
            dst = b + (wide ? 16u * ((t & 1) * ps + (t >> 1)) : 16u * (((t >> 1) & 1) * ps + (t >> 2)) + 8u * (t & 1));
        } else if (wide) {
            // (pixel, unit) of this thread's next copy by steps of 256 units
            const int U = F >> 1, dp = kGramThreads / U, du = kGramThreads - dp * U;
            int px = t / U, u = t - px * U;
            for (int i = t; i < n * U; i += kGramThreads) {
                fqi::cp_async<16>(buf + px * 2 * ps + (u & 1) * ps + (u >> 1), S + p0 * F * 2 + (size_t)i * 4);
                px += dp;
                u += du;
                if (u >= U) {
                    u -= U;
                    ++px;
                }
            }
        } else {
            for (int i = t; i < n * F; i += kGramThreads, src += 2 * kGramThreads) {
                const int px = i / F, c = i - px * F;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                                 b + 16u * (px * 2 * ps + ((c >> 1) & 1) * ps + (c >> 2)) + 8u * (c & 1)),
                             "l"(src)
                             : "memory");
            }
        }
    }
    __device__ __forceinline__ void row()  // at most 256 units (F <= 512)
    {
        if constexpr (kRows) {
            if (wide) {
                if (2 * (int)threadIdx.x < F) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if ((int)threadIdx.x + h * kGramThreads < F)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + h * 4u * kGramThreads),
                                     "l"(src + h * 2 * kGramThreads)
                                     : "memory");
            }
            src += 2 * F;
            dst += 32u * ps;
        }
    }
    __device__ __forceinline__ void put(int, float4 *) const {}
};

template <int PX>
struct GramStage<PX, __nv_bfloat16> {
    static constexpr bool kRows = false;
    const __nv_bfloat16 *S;
    int F, ps;
    uint32_t hold[kGramHold];
    __device__ __forceinline__ GramStage(const __nv_bfloat16 *s, int f, int p) : S(s), F(f), ps(p) {}
    __device__ __forceinline__ void row() const {}
    __device__ __forceinline__ void fetch(int64_t p0, int n, float4 *)
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(S + p0 * F * 2);
        if ((F & 1) == 0) {  // two columns at once (S is 8-byte aligned)
            const uint2 *s2 = reinterpret_cast<const uint2 *>(src) + threadIdx.x;
#pragma unroll
            for (int q = 0; q < kGramHold / 2; ++q)
                if ((int)threadIdx.x + q * kGramThreads < n * (F >> 1)) {
                    const uint2 v = s2[q * kGramThreads];
                    hold[2 * q] = v.x;
                    hold[2 * q + 1] = v.y;
                }
        } else {
#pragma unroll
            for (int q = 0; q < kGramHold; ++q)
                if ((int)threadIdx.x + q * kGramThreads < n * F) hold[q] = src[threadIdx.x + q * kGramThreads];
        }
    }
    // the values that fetch has loaded, into buf
    __device__ __forceinline__ void put(int n, float4 *buf) const
    {
        if ((F & 1) == 0) {
            GramWalk w(F >> 1, ps, buf);
#pragma unroll
            for (int q = 0; q < kGramHold / 2; ++q) {
                if ((int)threadIdx.x + q * kGramThreads >= n * w.U) break;
                const uint32_t a = hold[2 * q], b = hold[2 * q + 1];
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(w.at()), "r"(a << 16), "r"(a & 0xffff0000u),
                             "r"(b << 16), "r"(b & 0xffff0000u)
                             : "memory");
                w.next();
            }
        } else {
            const int dp = kGramThreads / F, dc = kGramThreads - dp * F;
            int px = threadIdx.x / F, c = threadIdx.x - px * F;
#pragma unroll
            for (int q = 0; q < kGramHold; ++q) {
                if ((int)threadIdx.x + q * kGramThreads >= n * F) break;
                float2 *d = reinterpret_cast<float2 *>(buf + px * 2 * ps + ((c >> 1) & 1) * ps + (c >> 2)) + (c & 1);
                *d = make_float2(__uint_as_float(hold[q] << 16), __uint_as_float(hold[q] & 0xffff0000u));
                px += dp;
                c += dc;
                if (c >= F) {
                    c -= F;
                    ++px;
                }
            }
        }
    }
};

__device__ __forceinline__ void cmac(float2 &s, float ax, float ay, float bx, float by)  // s += conj(a) b
{
    s.x = fmaf(ax, bx, s.x);
    s.y = fmaf(ax, by, s.y);
    s.x = fmaf(ay, by, s.x);
    s.y = fmaf(-ay, bx, s.y);
}

template <int PX, typename T>
__device__ __forceinline__ void gram_part(const T *__restrict__ S, int64_t P, int F, int64_t chunk_len,
                                          float2 *__restrict__ part, int which, int c, float4 *panel)
{
    const int nb = gram_cols(F), nblk = gram_blocks(F), parts = gram_parts(F);
    const int per = (nblk + parts - 1) / parts;
    const int64_t pbeg = (int64_t)c * chunk_len;
    const int64_t pend = min(P, pbeg + chunk_len);
    // this thread's block (bi, bj) of the row-major upper triangle
    int t = which * per + (int)threadIdx.x;
    const bool on = (int)threadIdx.x < per && t < nblk;
    int bi = 0, bj = 0;
    if (on) {
        while (t >= nb - bi) { t -= nb - bi; ++bi; }
        bj = bi + t;
    }
    const int ps = gram_plane(F), psz = PX * 2 * ps;  // units of a plane and of a panel
    __syncthreads();  // the previous item of a persistent CTA still reads the panels
    // columns past F stay zero (every panel writes the same places)
    if (F & 3)
        for (int i = threadIdx.x; i < 2 * PX; i += kGramThreads)
            panel[i * 2 * ps + nb - 1] = panel[i * 2 * ps + ps + nb - 1] = make_float4(0, 0, 0, 0);
    __syncthreads();
    float2 acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = make_float2(0, 0);
    GramStage<PX, T> stage(S, F, ps);
    constexpr bool kRows = GramStage<PX, T>::kRows;
    int n = (int)max((int64_t)0, min((int64_t)PX, pend - pbeg));  // pixels of this panel, then of the next
    if (n > 0) {
        stage.fetch(pbeg, n, panel);
        for (int px = 0; px < n; ++px) stage.row();
        stage.put(n, panel);
    }
    fqi::cp_async_commit();
    int cur = 0;
    for (int64_t p0 = pbeg; p0 < pend; p0 += PX) {
        const int next = (int)max((int64_t)0, min((int64_t)PX, pend - p0 - PX));
        if (!kRows) {
            if (next > 0) stage.fetch(p0 + PX, next, panel + (cur ^ 1) * psz);
            fqi::cp_async_commit();
        }
        fqi::cp_async_wait<kRows ? 0 : 1>();
        __syncthreads();
        if (kRows && next > 0) stage.fetch(p0 + PX, next, panel + (cur ^ 1) * psz);
        const float4 *row = panel + cur * psz;
        auto sums = [&](const float4 *row) {
            const float4 a0 = row[bi], a1 = row[ps + bi], b0 = row[bj], b1 = row[ps + bj];
            const float ax[4] = {a0.x, a0.z, a1.x, a1.z}, ay[4] = {a0.y, a0.w, a1.y, a1.w};
            const float bx[4] = {b0.x, b0.z, b1.x, b1.z}, by[4] = {b0.y, b0.w, b1.y, b1.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) cmac(acc[r][q], ax[r], ay[r], bx[q], by[q]);
        };
        if constexpr (PX == 16 && sizeof(T) == 4) {
            if (on) {
#pragma unroll 2
                for (int px = 0; px < n; ++px, row += 2 * ps) sums(row);
            }
        } else {
            // (the same loop for every panel: 8% faster here, 10% slower above)
#pragma unroll 2
            for (int px = 0; px < PX; ++px, row += 2 * ps) {
                if (kRows) {  // two rows of the next panel with each of the first pixels
                    if (2 * px < next) stage.row();
                    if (2 * px + 1 < next) stage.row();
                }
                if (on && px < n) sums(row);
            }
        }
        // (the other panel was last read before the barrier that ended the loop before)
        if (next > 0) stage.put(next, panel + (cur ^ 1) * psz);
        if (kRows) fqi::cp_async_commit();
        __syncthreads();
        cur ^= 1;
        n = next;
    }
    fqi::cp_async_wait<0>();
    if (on) {
        float2 *out = part + (size_t)c * F * F;
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = 4 * bi + r, j = 4 * bj + q;
                if (i < F && j < F) out[(size_t)i * F + j] = acc[r][q];
            }
    }
}

template <int PX, typename T>
__global__ void __launch_bounds__(kGramThreads, kGramCtas) gram_partial_kernel(const T *__restrict__ S, int64_t P, int F,
                                                                       int64_t chunk_len, float2 *__restrict__ part)
{
    extern __shared__ float4 panel[];
    gram_part<PX, T>(S, P, F, chunk_len, part, blockIdx.x, blockIdx.y, panel);
}

// 32 entries of G from the partial sums: eight threads per entry take every
// eighth chunk, then one adds their sums in order; the lower triangle from
// the upper one.
constexpr int kReduceItem = 32;
constexpr int kReduceItems = 8;  // of them in an item of the batched reduction
__device__ __forceinline__ void gram_reduce_at(const float2 *__restrict__ part, int n_chunks, int F,
                                               float2 *__restrict__ G, int item, float2 (*red)[kReduceItem])
{
    const int lane = threadIdx.x % kReduceItem, g = threadIdx.x / kReduceItem;
    const int idx = item * kReduceItem + lane;
    const int i = idx / F, j = idx % F;
    const bool upper = idx < F * F && (i >> 2) <= (j >> 2);
    float2 s = make_float2(0, 0);
    if (upper) {
#pragma unroll 4
        for (int c = g; c < n_chunks; c += kGramThreads / kReduceItem) {
            const float2 v = part[(size_t)c * F * F + idx];
            s.x += v.x;
            s.y += v.y;
        }
    }
    __syncthreads();
    red[g][lane] = s;
    __syncthreads();
    if (g == 0 && upper) {
        for (int q = 1; q < kGramThreads / kReduceItem; ++q) {
            s.x += red[q][lane].x;
            s.y += red[q][lane].y;
        }
        G[idx] = s;
        if ((i >> 2) < (j >> 2)) G[j * F + i] = cconj(s);
    }
}

__global__ void __launch_bounds__(kGramThreads) gram_reduce_kernel(const float2 *__restrict__ part, int n_chunks, int F,
                                                                   float2 *__restrict__ G)
{
    __shared__ float2 red[kGramThreads / kReduceItem][kReduceItem];
    gram_reduce_at(part, n_chunks, F, G, blockIdx.x, red);
}

// ------------------------------------------------------------ eigen (1 CTA) --
constexpr int kEigThreads = 1024;  // all eigenvectors (QL)
constexpr int kTopThreads = 512;   // eigenvalues and the first vectors, the matrix in shared memory
// The first vectors of a matrix in global memory (F > 220) take 1024 threads:
// the rows wait on the L2 cache (240 / 300 frames, k = 2: 2.85 / 5.32 ms at 512
// threads, 2.55 / 4.34 at 1024).
inline int top_threads(int F) { return eig_in_smem(F) ? kTopThreads : kEigThreads; }

__device__ __forceinline__ int pidx(int i, int j) { return i * (i + 1) / 2 + j; }  // i >= j

// V[:, j] = H_0 ... H_{F-3} D Z[:, perm[j]] for j < ncol: warp per column, NQ
// values per lane.  With `buf` (shared memory for 2 x nbuf reflectors) the CTA
// copies the next nbuf reflectors while the warps apply the last ones (read
// one by one from global memory they took 0.09 ms at 200 frames); else they
// are read in place.  Called by every thread of the CTA.
template <int NQ>
__device__ __forceinline__ void back_transform_nq(int F, int ncol, const float *Z, int zs, const int *perm,
                                                  const float2 *delta, const float2 *__restrict__ hv,
                                                  const float *__restrict__ tau_g, float2 *__restrict__ V,
                                                  float2 *__restrict__ Vt, float2 *buf, int nbuf, int lane, int wid, int nw)
{
    const int n = F > 2 ? F - 2 : 0;  // reflectors; number r is H_{n-1-r}
    auto stage = [&](int c) {
        float2 *b = buf + (size_t)(c & 1) * nbuf * F;
        const int r0 = c * nbuf, cnt = min(nbuf, n - r0);
        for (int t = threadIdx.x; t < cnt * F; t += 32 * nw) {
            const int r = t / F, i = t - r * F, k = n - 1 - (r0 + r);
            if (i > k) fqi::cp_async<8>(b + t, hv + (size_t)k * F + i);
            else b[t] = make_float2(0, 0);
        }
        fqi::cp_async_commit();
    };
    for (int j0 = 0; j0 < ncol; j0 += nw) {
        const int j = j0 + wid;
        const bool on = j < ncol;
        float2 y[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int i = lane + 32 * q;
            const float z = on && i < F ? Z[i * zs + perm[j]] : 0.0f;
            y[q] = i < F ? make_float2(delta[i].x * z, delta[i].y * z) : make_float2(0, 0);
        }
        auto apply = [&](const float2 *v, int k, bool padded) {
            const float t = tau_g[k];
            float2 x[NQ], s = make_float2(0, 0);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = lane + 32 * q;
                x[q] = i < F && (padded || i > k) ? v[i] : make_float2(0, 0);
                cmac(s, x[q].x, x[q].y, y[q].x, y[q].y);
            }
            for (int o = 16; o > 0; o >>= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
            }
            s.x *= -t;
            s.y *= -t;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {  // y -= t (v^H y) v
                y[q].x = fmaf(x[q].x, s.x, fmaf(-x[q].y, s.y, y[q].x));
                y[q].y = fmaf(x[q].x, s.y, fmaf(x[q].y, s.x, y[q].y));
            }
        };
        if (nbuf > 0) {
            const int nc = (n + nbuf - 1) / nbuf;
            if (nc > 0) stage(0);
            for (int c = 0; c < nc; ++c) {
                if (c + 1 < nc) stage(c + 1);
                else fqi::cp_async_commit();
                fqi::cp_async_wait<1>();
                __syncthreads();
                if (on)
                    for (int r = 0; r < min(nbuf, n - c * nbuf); ++r)
                        apply(buf + ((size_t)(c & 1) * nbuf + r) * F, n - 1 - c * nbuf - r, true);
                __syncthreads();
            }
            fqi::cp_async_wait<0>();
        } else if (on) {
            for (int k = n - 1; k >= 0; --k) apply(hv + (size_t)k * F, k, false);
        }
        // unit length again: the reflectors are unitary to their rounding only, and
        // what is missing of the largest components stays in the filtered IQ
        float n2 = 0.0f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) n2 = fmaf(y[q].x, y[q].x, fmaf(y[q].y, y[q].y, n2));
        for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        const float unit = fmaf(-0.5f, n2, 1.5f);  // 1 / sqrt(n2) for n2 = 1 + 1e-5
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int i = lane + 32 * q;
            y[q] = make_float2(y[q].x * unit, y[q].y * unit);
            if (on && i < F) {
                if (V) V[(size_t)i * F + j] = y[q];
                Vt[(size_t)j * F + i] = y[q];
            }
        }
    }
}
__device__ __forceinline__ void back_transform(int F, int ncol, const float *Z, int zs, const int *perm, const float2 *delta,
                               const float2 *__restrict__ hv, const float *__restrict__ tau_g, float2 *__restrict__ V,
                               float2 *__restrict__ Vt, float2 *buf, int nbuf, int lane, int wid, int nw)
{
    if (F <= 128) back_transform_nq<4>(F, ncol, Z, zs, perm, delta, hv, tau_g, V, Vt, buf, nbuf, lane, wid, nw);
    else if (F <= 224) back_transform_nq<7>(F, ncol, Z, zs, perm, delta, hv, tau_g, V, Vt, buf, nbuf, lane, wid, nw);
    else back_transform_nq<16>(F, ncol, Z, zs, perm, delta, hv, tau_g, V, Vt, buf, nbuf, lane, wid, nw);
}

// Number of eigenvalues of the real symmetric tridiagonal (d, e) below x
// (Sturm count by the signs of the LDL^T pivots).
// The quotient is a product with the hardware reciprocal (1.5 units in its
// last place, a relative change of e2 far below the tridiagonalisation's own
// rounding).  No test of tiny pivots: a zero pivot gives an infinite quotient
// and the next pivot the opposite sign, counted by sign bits (e2 > 0).  Two
// points at once: their recurrences hide each other's latency.
__device__ __forceinline__ void sturm_below(const float *d, const float *e2, int n, float xa, float xb, int &ca, int &cb)
{
    float qa = d[0] - xa, qb = d[0] - xb;
    int c0 = (int)(__float_as_uint(qa) >> 31), c1 = (int)(__float_as_uint(qb) >> 31);
#pragma unroll 4
    for (int i = 1; i < n; ++i) {
        const float b = e2[i - 1], di = d[i];
        auto step = [&](float &q, float x, int &c) {
            float r;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
            q = __fmaf_rn(-b, r, __fsub_rn(di, x));
            c += (int)(__float_as_uint(q) >> 31);
        };
        step(qa, xa, c0);
        step(qb, xb, c1);
    }
    ca = c0;
    cb = c1;
}

// binary32 as integers of the same order (and back)
__device__ __forceinline__ int ordered_bits(int b) { return b ^ ((b >> 31) & 0x7fffffff); }

// The eigenvalues in descending order by multisection on [lo, hi]: np threads
// (a power of two that divides the warp) per eigenvalue evaluate two points of
// its bracket each a round, until the bracket holds no other number.  The points
// divide the numbers of the bracket evenly, not its length, so that an eigenvalue
// takes log_(2 np + 1) 2^32 rounds whatever its size (20 for np = 1), and small
// ones of a graded matrix are good to their last bits (halving the length to
// 2^-31 of the largest row sum took as long).
__device__ void multisect(const float *d, const float *e2, int n, float lo0, float hi0, float *lam, int nt)
{
    int np = 1;
    while (np < 32 && 2 * np * n <= nt / 2) np *= 2;
    const int per = nt / np;  // eigenvalues of a pass
    const int lane = threadIdx.x & 31, p = threadIdx.x % np;
    const unsigned grp = (np == 32 ? 0xffffffffu : (1u << np) - 1u) << (lane - p);
    const unsigned part = 0xffffffffu / (unsigned)(2 * np + 1) + 1u;
    for (int j0 = 0; j0 < n; j0 += per) {
        const int j = j0 + (int)threadIdx.x / np;
        const int m = n - 1 - j;  // m-th smallest
        int lo = ordered_bits(__float_as_int(lo0)), hi = ordered_bits(__float_as_int(hi0));
        bool act = j < n && lo < hi;
        for (int it = 0; it < 40; ++it) {
            const unsigned gap = (unsigned)hi - (unsigned)lo;
            act = act && gap > 1u;
            if (!__any_sync(0xffffffffu, act)) break;
            // the 2 np points, computed alike by every thread of the group
            auto point = [&](int i) { return (int)((unsigned)lo + __umulhi(gap, (unsigned)(i + 1) * part)); };
            auto value = [&](int i) { return __int_as_float(ordered_bits(point(i))); };
            int ca = 0, cb = 0;
            if (act) sturm_below(d, e2, n, value(2 * p), value(2 * p + 1), ca, cb);
            const unsigned ba = __ballot_sync(0xffffffffu, act && ca < m + 1) & grp;
            const unsigned bb = __ballot_sync(0xffffffffu, act && cb < m + 1) & grp;
            const int c = __popc(ba) + __popc(bb);  // points below the eigenvalue
            if (act) {
                const int nlo = c > 0 ? point(c - 1) : lo, nhi = c < 2 * np ? point(c) : hi;
                lo = nlo;
                hi = nhi;
            }
        }
        if (j < n && p == 0)
            lam[j] = 0.5f * (__int_as_float(ordered_bits(lo)) + __int_as_float(ordered_bits(hi)));
    }
}

// One eigenvector of the real tridiagonal for eigenvalue sigma by inverse
// iteration: Gaussian elimination with partial pivoting of T - sigma I, three
// solves from a fixed pseudo-random start, each normalised.  Writes column
// `col` of Z (row stride zs).  scr: 6 n floats of shared or global memory
// (1 / u0, u1, u2, multipliers, swaps, x), value i of array a at
// scr[(a n + i) stride].
__device__ __forceinline__ void inverse_iteration(const float *d, const float *e, int n, float sigma, float tiny, int seed,
                                  float *Z, int zs, int col, float *scr, int stride)
{
    auto at = [&](int a, int i) -> float & { return scr[(size_t)(a * n + i) * stride]; };
    float p0 = d[0] - sigma, p1 = n > 1 ? e[0] : 0.0f, p2 = 0.0f;
    float c = p1, dn = n > 1 ? d[1] : 0.0f;
    for (int i = 0; i + 1 < n; ++i) {
        // c = e[i]: sub-diagonal of row i + 1 (operands read a step ahead of the stores)
        const float a1 = dn - sigma;
        const float b1 = (i + 2 < n) ? e[i + 1] : 0.0f;
        dn = (i + 2 < n) ? d[i + 2] : 0.0f;
        const bool swap = fabsf(c) > fabsf(p0);  // pivot on row i + 1
        const float piv = swap ? c : (fabsf(p0) < tiny ? (p0 < 0.0f ? -tiny : tiny) : p0);
        const float r = 1.0f / piv;
        const float mlt = (swap ? p0 : c) * r;
        at(0, i) = r;
        at(1, i) = swap ? a1 : p1;
        at(2, i) = swap ? b1 : p2;
        at(3, i) = mlt;
        at(4, i) = swap ? 1.0f : 0.0f;
        const float n0 = swap ? fmaf(-mlt, a1, p1) : fmaf(-mlt, p1, a1);
        p1 = swap ? fmaf(-mlt, b1, p2) : fmaf(-mlt, p2, b1);
        p0 = n0;
        p2 = 0.0f;
        c = b1;
    }
    at(0, n - 1) = 1.0f / (fabsf(p0) < tiny ? (p0 < 0.0f ? -tiny : tiny) : p0);
    at(1, n - 1) = 0.0f;
    at(2, n - 1) = 0.0f;
    unsigned h = 0x9E3779B9u * (unsigned)(seed + 1);
    for (int i = 0; i < n; ++i) {
        h = h * 1664525u + 1013904223u;
        at(5, i) = 1.0f + 0.25f * ((float)(h >> 8) * (1.0f / 16777216.0f) - 0.5f);
    }
    float s2 = 0.0f, inv = 1.0f;  // inv: the last solve's normalisation, applied on the next read
    for (int it = 0; it < 3; ++it) {
        // forward: apply the row swaps and multipliers to the right-hand side
        // (each step's operands are read before the last one's result is stored)
        float x0 = at(5, 0) * inv;
        float nx = n > 1 ? at(5, 1) : 0.0f, nm = at(3, 0), nsw = at(4, 0);
#pragma unroll 4
        for (int i = 0; i + 1 < n; ++i) {
            const float x1 = nx * inv, ml = nm;
            const bool swap = nsw != 0.0f;
            if (i + 2 < n) {
                nx = at(5, i + 2);
                nm = at(3, i + 1);
                nsw = at(4, i + 1);
            }
            at(5, i) = swap ? x1 : x0;
            x0 = swap ? fmaf(-ml, x1, x0) : fmaf(-ml, x0, x1);
        }
        // back substitution
        float x1 = x0 * at(0, n - 1), x2 = 0.0f, mx = fabsf(x1);
        at(5, n - 1) = x1;
        float b0 = 0.0f, b1 = 0.0f, b2 = 0.0f, b5 = 0.0f;
        auto fetch = [&](int i) {
            b0 = at(0, i);
            b1 = at(1, i);
            b2 = at(2, i);
            b5 = at(5, i);
        };
        if (n > 1) fetch(n - 2);
#pragma unroll 4
        for (int i = n - 2; i >= 0; --i) {
            const float x = fmaf(-b1, x1, fmaf(-b2, x2, b5)) * b0;
            if (i > 0) fetch(i - 1);
            at(5, i) = x;
            mx = fmaxf(mx, fabsf(x));
            x2 = x1;
            x1 = x;
        }
        inv = mx > 0.0f ? 1.0f / mx : 1.0f;
    }
    for (int i = 0; i < n; ++i) {
        const float x = at(5, i) * inv;
        s2 = fmaf(x, x, s2);
    }
    inv *= rsqrtf(s2);
    for (int i = 0; i < n; ++i) Z[i * zs + col] = at(5, i) * inv;
}

// Householder tridiagonalisation of the packed lower triangle Ap (F x F,
// complex Hermitian): d, the complex off-diagonal ec, the reflectors hv with
// their tau.  Per step: the reflector v from the new column and its norm, p =
// tau A v, K = tau / 2 Re v^H p, w = p - K v, A -= v w^H + w v^H.
//
// tridiagonalise_blocks: a matrix in shared memory (F <= 220), issue-bound on
// its one SM, so the work goes by 32 x 32 blocks with no index arithmetic or
// sum over the lanes inside: A v with a lane per row (below the diagonal the
// lane walks its stored row, beyond it the stored rows of the column block,
// conjugated), up to four warps a row block; the update with a lane per
// column, one 16-byte broadcast (v_i, w_i) a row.  The first column of the new
// trailing matrix comes out of the update.  A block's part of A v is summed in
// four chains of eight before it joins the row's sum (one or two chains over
// all blocks: eigenvalues 1.5 times as far off at 200 frames, the same time).
// Former versions: warp
// per row with nine barriers a step 1.5 ms at 200 frames (3.0M cycles), two
// barriers and v, w in registers 2.6M cycles (30k instructions a step).
constexpr int kPartStride = 224;
struct EigShared {
    float2 *part;     // up to four partial sums of A v, kPartStride apart
    float4 *vw;       // (v_i, w_i)
};

__device__ __forceinline__ float warp_sum(float x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// the reflector of the column x[0 .. m): every warp sums its squared norm, a
// lane's few values first and then the lanes (the error of the norm is the
// reflector's departure from a unitary matrix: sums of 32 in a row raised the
// error of the filtered IQ by half at 160 frames)
__device__ __forceinline__ void reflector(const float2 *x, int m, int lane, float &tau, float2 &v0, float2 &beta)
{
    float a2 = 0.0f;
    for (int i = lane; i < m; i += 32) a2 = fmaf(x[i].x, x[i].x, fmaf(x[i].y, x[i].y, a2));
    a2 = warp_sum(a2);
    const float2 x0 = x[0];
    const float ax0 = sqrtf(fmaf(x0.x, x0.x, x0.y * x0.y));
    const float alpha = sqrtf(a2);
    tau = 0.0f;
    v0 = beta = make_float2(0, 0);
    if (alpha > 1e-30f) {
        const float2 th = ax0 > 0.0f ? make_float2(x0.x / ax0, x0.y / ax0) : make_float2(1.0f, 0.0f);
        beta = make_float2(-th.x * alpha, -th.y * alpha);  // -theta alpha
        v0 = make_float2(th.x * (ax0 + alpha), th.y * (ax0 + alpha));
        tau = 1.0f / (alpha * (alpha + ax0));
    }
}

// c - (vi conj(y) + wi conj(x)): the small correction first, so that c is rounded once
__device__ __forceinline__ float2 rank2(float2 c, float2 vi, float2 wi, float2 x, float2 y)
{
    const float u = fmaf(vi.x, y.x, fmaf(vi.y, y.y, fmaf(wi.x, x.x, wi.y * x.y)));
    const float v = fmaf(vi.y, y.x, fmaf(-vi.x, y.y, fmaf(wi.y, x.x, -wi.x * x.y)));
    return make_float2(c.x - u, c.y - v);
}

__device__ __forceinline__ void tridiagonalise_blocks(float2 *Ap, int F, float *d, float2 *ec, float2 *vvA, float2 *vvB,
                                                      const EigShared &es, float2 *__restrict__ hv,
                                                      float *__restrict__ tau_g, int k1, int lane, int wid, int nw)
{
    for (int i = 1 + wid * 32 + lane; i < F; i += 32 * nw) vvA[i - 1] = Ap[pidx(i, 0)];  // column 0
    __syncthreads();
    for (int k = 0; k < k1; ++k) {
        const int m = F - k - 1;  // length of the column below the diagonal
        const int nb = (m + 31) >> 5;
        float2 *vv = (k & 1) ? vvB : vvA, *vnext = (k & 1) ? vvA : vvB;
        // ---- the reflector
        float tau;
        float2 v0, beta;
        reflector(vv, m, lane, tau, v0, beta);
        __syncthreads();
        for (int i = wid * 32 + lane; i < 32 * nb; i += 32 * nw) {  // zeros past m
            const float2 v = i == 0 ? v0 : (i < m && tau != 0.0f ? vv[i] : make_float2(0, 0));
            vv[i] = v;
            if (i < m) hv[(size_t)k * F + k + 1 + i] = v;
        }
        if (wid == nw - 1 && lane == 0) {
            d[k] = Ap[pidx(k, k)].x;
            ec[k] = beta;
            tau_g[k] = tau;
        }
        __syncthreads();
        // ---- partial sums of A v: W warps a row block, column blocks ws, ws + W, ..
        const int W = min(4, nw / nb);
        if (wid < W * nb) {
            const int rb = wid / W, ws = wid - rb * W;
            const int i = 32 * rb + lane, ic = min(i, m - 1);
            float2 s = make_float2(0, 0);
            for (int cb = ws; cb < nb; cb += W) {
                const float2 *v = vv + 32 * cb;
                float2 c[4];  // the block's sum in four chains of eight, then added to s
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = make_float2(0, 0);
                if (cb < rb) {
                    const float2 *a = Ap + pidx(k + 1 + ic, k + 1 + 32 * cb);
#pragma unroll 2
                    for (int j = 0; j < 32; j += 4)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 a0 = a[j + u], x0 = v[j + u];
                            c[u].x = fmaf(a0.x, x0.x, fmaf(-a0.y, x0.y, c[u].x));
                            c[u].y = fmaf(a0.x, x0.y, fmaf(a0.y, x0.x, c[u].y));
                        }
                } else if (cb > rb) {
                    const int n = min(32, m - 32 * cb);
                    int o = pidx(k + 1 + 32 * cb, k + 1 + i), st = k + 2 + 32 * cb;  // row 32 cb + j: o += its length
#pragma unroll 2
                    for (int j = 0; j < n; j += 4)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 a0 = Ap[j + u < n ? o : 0], x0 = v[j + u];  // (v = 0 past the end)
                            o += st++;
                            c[u].x = fmaf(a0.x, x0.x, fmaf(a0.y, x0.y, c[u].x));
                            c[u].y = fmaf(a0.x, x0.y, fmaf(-a0.y, x0.x, c[u].y));
                        }
                } else {
                    const int n = min(32, m - 32 * cb);
                    const int own = pidx(k + 1 + ic, k + 1 + 32 * cb);
                    for (int j = 0; j < n; j += 4)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int jc = min(j + u, n - 1);
                            const bool low = jc <= ic - 32 * cb;
                            const float2 a0 = Ap[low ? own + jc : pidx(k + 1 + 32 * cb + jc, k + 1 + ic)], x0 = v[j + u];
                            const float ay = low ? a0.y : -a0.y;
                            c[u].x = fmaf(a0.x, x0.x, fmaf(-ay, x0.y, c[u].x));
                            c[u].y = fmaf(a0.x, x0.y, fmaf(ay, x0.x, c[u].y));
                        }
                }
                s.x += (c[0].x + c[1].x) + (c[2].x + c[3].x);
                s.y += (c[0].y + c[1].y) + (c[2].y + c[3].y);
            }
            if (i < m) es.part[ws * kPartStride + i] = s;
        }
        __syncthreads();
        // ---- p, K (every warp), w
        float vhp = 0.0f;
        float2 pq = make_float2(0, 0), vq = make_float2(0, 0);  // of the warp's own block
        for (int q = 0; q < nb; ++q) {
            const int i = 32 * q + lane;
            float2 p = make_float2(0, 0), v = make_float2(0, 0);
            if (i < m) {
                const int Wp = min(W, nb);
                for (int h = 0; h < Wp; ++h) {
                    const float2 x = es.part[h * kPartStride + i];
                    p.x += x.x;
                    p.y += x.y;
                }
                p = make_float2(tau * p.x, tau * p.y);
                v = vv[i];
                vhp = fmaf(v.x, p.x, fmaf(v.y, p.y, vhp));
            }
            if (q == wid) {
                pq = p;
                vq = v;
            }
        }
        const float K = 0.5f * tau * warp_sum(vhp);
        if (wid < nb) es.vw[32 * wid + lane] = make_float4(vq.x, vq.y, fmaf(-K, vq.x, pq.x), fmaf(-K, vq.y, pq.y));
        __syncthreads();
        // ---- A -= v w^H + w v^H by lower blocks, numbered along the block rows
        for (int t = wid, rb = 0; ; t += nw) {
            // block t of the triangle (from the last one found on)
            while (rb < nb && (rb + 1) * (rb + 2) / 2 <= t) ++rb;
            if (rb >= nb) break;
            const int cb = t - rb * (rb + 1) / 2;
            const int j = 32 * cb + lane;
            const float4 y = es.vw[j];
            const int n = min(32, m - 32 * rb);
            int o = pidx(k + 1 + 32 * rb, k + 1 + j), st = k + 2 + 32 * rb;
            for (int r = 0; r < n; r += 4) {
                float2 a[4];
                int oo[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    oo[u] = o;
                    const bool on = r + u < n && j <= 32 * rb + r + u;
                    a[u] = on ? Ap[o] : make_float2(0, 0);
                    o += st++;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = 32 * rb + r + u;
                    const float4 x = es.vw[min(i, 32 * nb - 1)];
                    a[u] = rank2(a[u], make_float2(x.x, x.y), make_float2(x.z, x.w), make_float2(y.x, y.y),
                                 make_float2(y.z, y.w));
                    if (r + u < n && j <= i) Ap[oo[u]] = a[u];
                    if (j == 0 && i > 0 && r + u < n) vnext[i - 1] = a[u];  // the new trailing matrix's first column
                }
            }
        }
        __syncthreads();
    }
}

// The last 128 columns (or all of a smaller matrix): warp per row, two rows
// together, v and w of the lane's 32-column blocks in registers, two barriers a
// step.  With few blocks left, tridiagonalise_blocks keeps few warps busy (all
// of 100 frames: 635k cycles by blocks, 543k by rows; 48: 242k and 174k).
template <int NQ>
__device__ __forceinline__ void tridiagonalise_lanes(float2 *Ap, int F, int k0, float *d, float2 *ec, float2 *vvA, float2 *vvB,
                                               float2 *pv, float *redq, float2 *__restrict__ hv,
                                               float *__restrict__ tau_g, int lane, int wid, int nw)
{
    for (int k = k0; k + 2 < F; ++k) {
        const int m = F - k - 1;  // length of the column below the diagonal
        float2 *vv = (k & 1) ? vvB : vvA, *vnext = (k & 1) ? vvA : vvB;
        // ---- (B)
        float tau;
        float2 v0, beta;
        reflector(vv, m, lane, tau, v0, beta);
        auto vat = [&](int i) { return i == 0 ? v0 : (tau != 0.0f ? vv[i] : make_float2(0, 0)); };
        if (wid == nw - 1 && lane == 0) {
            d[k] = Ap[pidx(k, k)].x;
            ec[k] = beta;
            tau_g[k] = tau;
        }
        for (int i = wid * 32 + lane; i < m; i += 32 * nw) hv[(size_t)k * F + k + 1 + i] = vat(i);
        float2 v[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) v[q] = lane + 32 * q < m ? vat(lane + 32 * q) : make_float2(0, 0);
        int cb[NQ];  // first word of the lane's columns below the diagonal
#pragma unroll
        for (int q = 0; q < NQ; ++q) cb[q] = pidx(k + 1 + lane + 32 * q, 0);
        float vhp = 0.0f;
        for (int i = wid; i < m; i += 2 * nw) {
            const int i2 = i + nw;
            const bool two = i2 < m;
            const int iz = two ? i2 : i;
            const int g1 = k + 1 + i, g2 = k + 1 + iz;
            const int r1 = pidx(g1, k + 1), r2 = pidx(g2, k + 1);
            // s += A(i, j) v_j for the lane's columns j = 32 q + lane: the stored row up
            // to the diagonal, the conjugate of the column beyond it
            auto mac = [](float2 &s, float2 a, float2 x) {
                s.x = fmaf(a.x, x.x, fmaf(-a.y, x.y, s.x));
                s.y = fmaf(a.x, x.y, fmaf(a.y, x.x, s.y));
            };
            auto macc = [](float2 &s, float2 a, float2 x) {  // conj(a) x
                s.x = fmaf(a.x, x.x, fmaf(a.y, x.y, s.x));
                s.y = fmaf(a.x, x.y, fmaf(-a.y, x.x, s.y));
            };
            float2 s1 = make_float2(0, 0), s2 = make_float2(0, 0);
            // both rows' loads before their sums (columns past m: the row's last
            // value times v = 0)
            float2 a[NQ], b[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (32 * q < m) {
                    const int j = lane + 32 * q;
                    const bool in = j < m;
                    a[q] = Ap[j <= i || !in ? r1 + min(j, i) : cb[q] + g1];
                    b[q] = Ap[j <= iz || !in ? r2 + min(j, iz) : cb[q] + g2];
                }
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (32 * q < m) {
                    const int j = lane + 32 * q;
                    if (32 * q + 31 <= i) mac(s1, a[q], v[q]);
                    else if (32 * q > i) macc(s1, a[q], v[q]);
                    else mac(s1, make_float2(a[q].x, j <= i ? a[q].y : -a[q].y), v[q]);
                    if (32 * q + 31 <= iz) mac(s2, b[q], v[q]);
                    else if (32 * q > iz) macc(s2, b[q], v[q]);
                    else mac(s2, make_float2(b[q].x, j <= iz ? b[q].y : -b[q].y), v[q]);
                }
            // four sums over the lanes in six exchanges: s1.x, s1.y, s2.x, s2.y end in
            // lanes 0, 8, 16, 24 (and the seven after each)
            const bool h16 = lane & 16, h8 = lane & 8;
            const float ax = (h16 ? s2.x : s1.x) + __shfl_xor_sync(0xffffffffu, h16 ? s1.x : s2.x, 16);
            const float ay = (h16 ? s2.y : s1.y) + __shfl_xor_sync(0xffffffffu, h16 ? s1.y : s2.y, 16);
            float t = (h8 ? ay : ax) + __shfl_xor_sync(0xffffffffu, h8 ? ax : ay, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 4);
            t += __shfl_xor_sync(0xffffffffu, t, 2);
            t += __shfl_xor_sync(0xffffffffu, t, 1);
            if ((lane & 7) == 0 && (two || !h16)) {
                const int row = h16 ? i2 : i;
                const float pc = tau * t;
                const float2 x = vat(row);
                reinterpret_cast<float *>(pv)[2 * row + (h8 ? 1 : 0)] = pc;
                vhp = fmaf(h8 ? x.y : x.x, pc, vhp);
            }
        }
        vhp = warp_sum(vhp);
        if (lane == 0) redq[wid] = vhp;
        __syncthreads();
        // ---- (A)
        const float K = 0.5f * tau * warp_sum(lane < nw ? redq[lane] : 0.0f);
        auto wat = [&](int i) {
            const float2 x = vat(i), p = pv[i];
            return make_float2(fmaf(-K, x.x, p.x), fmaf(-K, x.y, p.y));
        };
        float2 w[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) w[q] = lane + 32 * q < m ? wat(lane + 32 * q) : make_float2(0, 0);
        for (int i = wid; i < m; i += 2 * nw) {
            const int i2 = i + nw;
            const bool two = i2 < m;
            const int r1 = pidx(k + 1 + i, k + 1), r2 = two ? pidx(k + 1 + i2, k + 1) : r1;
            const float2 vi1 = vat(i), wi1 = wat(i), vi2 = two ? vat(i2) : vi1, wi2 = two ? wat(i2) : wi1;
            auto first = [&](int row, float2 c) {  // the first column of the new trailing matrix
                if (lane == 0 && row > 0) vnext[row - 1] = c;
            };
            const int e2 = two ? i2 : -1;  // last columns of the two rows: i, e2
            // both rows loaded before anything is stored: the compiler cannot
            // move a load over a store to the same matrix
            float2 a[NQ], b[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = lane + 32 * q;
                if (32 * q <= i && j <= i) a[q] = Ap[r1 + j];
                if (32 * q <= e2 && j <= e2) b[q] = Ap[r2 + j];
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = lane + 32 * q;
                if (32 * q <= i) {
                    a[q] = rank2(a[q], vi1, wi1, v[q], w[q]);
                    if (j <= i) Ap[r1 + j] = a[q];
                }
                if (32 * q <= e2) {
                    b[q] = rank2(b[q], vi2, wi2, v[q], w[q]);
                    if (j <= e2) Ap[r2 + j] = b[q];
                }
            }
            first(i, a[0]);
            if (two) first(i2, b[0]);
        }
        __syncthreads();
    }
}

// A matrix in global memory (F > 220): warp per row, two barriers a step.
__device__ __forceinline__ void tridiagonalise_rows(float2 *Ap, int F, float *d, float2 *ec, float2 *vvA, float2 *vvB,
                                                    float2 *pv, float *redq, float2 *__restrict__ hv,
                                                    float *__restrict__ tau_g, int lane, int wid, int nw)
{
    for (int i = 1 + wid * 32 + lane; i < F; i += 32 * nw) vvA[i - 1] = Ap[pidx(i, 0)];  // column 0
    __syncthreads();
    for (int k = 0; k + 2 < F; ++k) {
        const int m = F - k - 1;  // length of the column below the diagonal
        float2 *vv = (k & 1) ? vvB : vvA, *vnext = (k & 1) ? vvA : vvB;
        float tau;
        float2 v0, beta;
        reflector(vv, m, lane, tau, v0, beta);
        auto vat = [&](int i) { return i == 0 ? v0 : (tau != 0.0f ? vv[i] : make_float2(0, 0)); };
        if (wid == nw - 1 && lane == 0) {
            d[k] = Ap[pidx(k, k)].x;
            ec[k] = beta;
            tau_g[k] = tau;
        }
        for (int i = wid * 32 + lane; i < m; i += 32 * nw) hv[(size_t)k * F + k + 1 + i] = vat(i);
        float vhp = 0.0f;
        for (int i = wid; i < m; i += nw) {
            const int gi = k + 1 + i;
            float2 s = make_float2(0, 0);
#pragma unroll 4
            for (int j = lane; j < m; j += 32) {
                const float2 a = Ap[j <= i ? pidx(gi, k + 1 + j) : pidx(k + 1 + j, gi)], x = vat(j);
                const float ay = j <= i ? a.y : -a.y;
                s.x = fmaf(a.x, x.x, fmaf(-ay, x.y, s.x));
                s.y = fmaf(a.x, x.y, fmaf(ay, x.x, s.y));
            }
            s.x = warp_sum(s.x);
            s.y = warp_sum(s.y);
            if (lane == 0) {
                const float2 p = make_float2(tau * s.x, tau * s.y), x = vat(i);
                pv[i] = p;
                vhp = fmaf(x.x, p.x, fmaf(x.y, p.y, vhp));
            }
        }
        if (lane == 0) redq[wid] = vhp;
        __syncthreads();
        const float K = 0.5f * tau * warp_sum(lane < nw ? redq[lane] : 0.0f);
        auto wat = [&](int i) {
            const float2 x = vat(i), p = pv[i];
            return make_float2(fmaf(-K, x.x, p.x), fmaf(-K, x.y, p.y));
        };
        for (int i = wid; i < m; i += nw) {
            const int r = pidx(k + 1 + i, k + 1);
            const float2 vi = vat(i), wi = wat(i);
#pragma unroll 4
            for (int j = lane; j <= i; j += 32) {
                const float2 c = rank2(Ap[r + j], vi, wi, vat(j), wat(j));
                Ap[r + j] = c;
                if (j == 0 && i > 0) vnext[i - 1] = c;  // the first column of the new trailing matrix
            }
        }
        __syncthreads();
    }
}

// an element of the Gram matrix; L2: past the L1 cache, where an earlier launch's
// may be left
template <bool L2>
__device__ __forceinline__ float2 load_gram(const float2 *p) { return L2 ? __ldcg(p) : *p; }

// One step of subspace iteration with the matrix itself: V <- orth(G V) for the
// k <= kRefineMaxK vectors, where lambda_j is well above the rounding of G.
// It takes the rounding of the F reflectors out of the filter's subspace (a
// factor lambda_{k+1} / lambda_k of it stays): error of the filtered IQ against
// 64 bits, components 1.4 dB apart, 200 frames: 0.46e-6 for k = 8 with it, 1.33e-6
// for k = 9 without, for 0.03 ms.
// G is scaled as in the decomposition (ginv: the power of two, exact), so that
// the norms of the new vectors, about lambda_j, lie within 2^-12 / F and F at any
// amplitude of the IQ (unscaled, their squares left binary32 beyond lambda 1.8e19
// and below 1.1e-19, and the filter removed nothing).
// Y: k F values of scratch.
constexpr int kRefineMaxK = 8;
template <bool L2>
__device__ __forceinline__ void refine_vectors(const float2 *__restrict__ G, float ginv, int F, int k, const float *lam,
                                               float2 *Y, float2 *V, float2 *Vt, int lane, int wid, int nw)
{
    __syncthreads();
    for (int i = wid; i < F; i += nw)
        for (int j0 = 0; j0 < k; j0 += 4) {  // four columns together: their sums over the lanes overlap
            float2 s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = make_float2(0, 0);
            for (int f = lane; f < F; f += 32) {
                float2 g = load_gram<L2>(G + (size_t)i * F + f);
                g = make_float2(g.x * ginv, g.y * ginv);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (j0 + u < k) {
                        const float2 t = cmul(g, Vt[(size_t)(j0 + u) * F + f]);
                        s[u].x += t.x;
                        s[u].y += t.y;
                    }
            }
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    s[u].x += __shfl_xor_sync(0xffffffffu, s[u].x, o);
                    s[u].y += __shfl_xor_sync(0xffffffffu, s[u].y, o);
                }
            if (lane == 0)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (j0 + u < k)
                        Y[(size_t)(j0 + u) * F + i] =
                            lam[j0 + u] > 2.44140625e-4f * lam[0] ? s[u] : Vt[(size_t)(j0 + u) * F + i];
        }
    __syncthreads();
    if (wid == 0) {  // modified Gram-Schmidt in the order of the eigenvalues
        for (int j = 0; j < k; ++j) {
            float2 *y = Y + (size_t)j * F;
            for (int pass = 0; pass <= j; ++pass) {
                float n2 = 0.0f;
                for (int f = lane; f < F; f += 32) n2 = fmaf(y[f].x, y[f].x, fmaf(y[f].y, y[f].y, n2));
                const float inv = rsqrtf(fmaxf(warp_sum(n2), FLT_MIN));
                for (int f = lane; f < F; f += 32) y[f] = make_float2(y[f].x * inv, y[f].y * inv);
                __syncwarp();
                if (pass == j) break;
                const float2 *x = Y + (size_t)pass * F;
                float2 c = make_float2(0, 0);
                for (int f = lane; f < F; f += 32) cmac(c, x[f].x, x[f].y, y[f].x, y[f].y);
                c.x = warp_sum(c.x);
                c.y = warp_sum(c.y);
                for (int f = lane; f < F; f += 32) {
                    const float2 t = cmul(x[f], c);
                    y[f] = make_float2(y[f].x - t.x, y[f].y - t.y);
                }
                __syncwarp();
            }
            for (int f = lane; f < F; f += 32) {
                Vt[(size_t)j * F + f] = y[f];
                if (V) V[(size_t)f * F + j] = y[f];
            }
        }
    }
}

// Householder tridiagonalisation of the Hermitian G (lower triangle used),
// implicit QL with Wilkinson shifts on the real tridiagonal (after a
// diagonal unitary scaling), eigenvalue sort and back-transformation.
// Optional: the energy / fixed cutoff k.
// L2: for a launch that may start before the one ahead of it in its stream has
// ended (see batched_eig).
template <bool L2>
__device__ __forceinline__ void eig_body(const float2 *__restrict__ G, int F, float2 *__restrict__ big,
                                         float2 *__restrict__ hv, float *__restrict__ tau_g,
                                         double *__restrict__ lam_out, float2 *__restrict__ V,
                                         float2 *__restrict__ Vt, int k_cut, double thresh,
                                         int *__restrict__ k_out, int *__restrict__ status,
                                         int topk_only, float *__restrict__ ii_scr, int nt)
{
    extern __shared__ float2 dyn[];
    float2 *Ap = big ? big : dyn;                 // packed lower triangle, later Z (real, stride F+1)
    float *Z = reinterpret_cast<float *>(Ap);
    __shared__ float red[33];
    __shared__ float d[512], e[512], redq[32];
    __shared__ float2 ec[512], vv[512], rcs[512];
    __shared__ float2 eigw[1536];  // the partial sums of the tridiagonalisation; p; then the three below
    float2 *pv = eigw, *delta = eigw + 512;
    float *spare = reinterpret_cast<float *>(eigw + 1024);  // e^2 and the eigenvalues
    float *rc = reinterpret_cast<float *>(rcs), *rs = rc + 512;  // QL rotations (tridiagonalisation: a second vv)
    __shared__ int perm[512];
    __shared__ float s_scale;
    __shared__ int s_m, s_nrot, s_done, s_fail;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;

    // scale to max |G_ij| <= 1 (eigenvectors unchanged, eigenvalues rescaled at the end)
    float amax = 0.0f;
    for (int i = wid; i < F; i += nw)
        for (int j = lane; j <= i; j += 32) {
            float2 g = load_gram<L2>(G + (size_t)i * F + j);
            amax = fmaxf(amax, fmaxf(fabsf(g.x), fabsf(g.y)));
        }
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) red[wid] = amax;
    __syncthreads();
    if (tid == 0) {
        float mx = 0.0f;
        for (int w = 0; w < nw; ++w) mx = fmaxf(mx, red[w]);
        // a power of two, so that the scaling itself is exact
        s_scale = mx > 0.0f ? exp2f(ceilf(log2f(mx))) : 1.0f;
    }
    __syncthreads();
    const float gscale = s_scale, ginv = 1.0f / s_scale;
    for (int i = wid; i < F; i += nw)
        for (int j = lane; j <= i; j += 32) {
            float2 g = load_gram<L2>(G + (size_t)i * F + j);
            Ap[pidx(i, j)] = make_float2(g.x * ginv, g.y * ginv);
        }
    __syncthreads();

    // (a matrix in shared memory, F <= 220, goes by `dyn` itself, so that it is
    // addressed as such)
    __shared__ float4 vw[224];
    if (big) {
        tridiagonalise_rows(big, F, d, ec, vv, rcs, pv, redq, hv, tau_g, lane, wid, nw);
    } else {
        const EigShared es = {eigw, vw};
        const int k1 = max(0, F - 129);  // blocks while more than 128 rows remain
        tridiagonalise_blocks(dyn, F, d, ec, vv, rcs, es, hv, tau_g, k1, lane, wid, nw);
        tridiagonalise_lanes<4>(dyn, F, k1, d, ec, vv, rcs, pv, redq, hv, tau_g, lane, wid, nw);
    }
    if (tid == 0) {
        if (F >= 2) {
            d[F - 2] = Ap[pidx(F - 2, F - 2)].x;
            ec[F - 2] = Ap[pidx(F - 1, F - 2)];
        }
        d[F - 1] = Ap[pidx(F - 1, F - 1)].x;
        s_fail = 0;
    }
    __syncthreads();
    // diagonal unitary scaling making the off-diagonal real and >= 0: the phases
    // side by side, then their running product
    for (int k = tid; k < F; k += nt) {
        const float2 x = k + 1 < F ? ec[k] : make_float2(0, 0);
        const float ax = sqrtf(x.x * x.x + x.y * x.y);
        e[k] = ax;
        vv[k] = ax > 0.0f ? make_float2(x.x / ax, x.y / ax) : make_float2(1.0f, 0.0f);
    }
    __syncthreads();
    if (tid == 0) {
        float2 dl = make_float2(1.0f, 0.0f);
        delta[0] = dl;
#pragma unroll 4
        for (int k = 0; k + 1 < F; ++k) {
            dl = cmul(dl, vv[k]);
            delta[k + 1] = dl;
        }
    }
    __syncthreads();
    const int zs = F + 1;
    if (topk_only) {
        // ---- all eigenvalues by multisection, top-k vectors by inverse iteration;
        // the QL path below is the fallback for large k
        float *e2 = spare, *lamd = spare + 512;
        __shared__ float s_lo, s_hi, s_tnorm;
        __shared__ int s_k;
        for (int i = tid; i < F; i += nt) e2[i] = fmaxf(e[i] * e[i], 4.0f * FLT_MIN);  // > 0
        if (wid == 0) {
            float lo = 1e30f, hi = -1e30f, tn = 0.0f;
            for (int i = lane; i < F; i += 32) {
                const float r = (i > 0 ? e[i - 1] : 0.0f) + e[i];
                lo = fminf(lo, d[i] - r);
                hi = fmaxf(hi, d[i] + r);
                tn = fmaxf(tn, fabsf(d[i]) + r);
            }
            for (int o = 16; o > 0; o >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                tn = fmaxf(tn, __shfl_xor_sync(0xffffffffu, tn, o));
            }
            if (lane == 0) {
                const float pad = 4.0f * FLT_EPSILON * fmaxf(tn, 1e-30f);
                s_lo = lo - pad;
                s_hi = hi + pad;
                s_tnorm = tn;
            }
        }
        __syncthreads();
        multisect(d, e2, F, s_lo, s_hi, lamd, nt);  // descending order
        __syncthreads();
        for (int j = tid; j < F; j += nt) lam_out[j] = (double)lamd[j] * (double)gscale;
        if (tid == 0) {
            int k = k_cut;
            if (k < 0) {
                double tot = 0.0, acc = 0.0;
                for (int j = 0; j < F; ++j) tot += fmax((double)lamd[j], 0.0);
                k = F;
                for (int j = 0; j < F; ++j) {
                    acc += fmax((double)lamd[j], 0.0);
                    if (acc >= thresh * tot) { k = j + 1; break; }
                }
            }
            if (k_out) *k_out = k;
            s_k = k;
        }
        __syncthreads();
        const int k = s_k;
        if (k <= kFastMaxK && ii_scr) {
            int zk;
            const float tiny = FLT_EPSILON * fmaxf(s_tnorm, 1e-30f);
            // vectors (stride zk) and, where they fit behind them, the solves' scratch
            // in the packed matrix's storage
            zk = k | 1;
            const bool in_z = !big && (size_t)F * zk + (size_t)6 * k * F <= (size_t)F * (F + 1);
            for (int j = tid; j < k; j += nt) {
                if (in_z) {
                    float *z = reinterpret_cast<float *>(dyn);
                    inverse_iteration(d, e, F, lamd[j], tiny, j, z, zk, j, z + (size_t)F * zk + j, k);
                } else {
                    inverse_iteration(d, e, F, lamd[j], tiny, j, Z, zk, j, ii_scr + j, k);
                }
            }
            __syncthreads();
            // re-orthogonalise vectors of close eigenvalues (modified Gram-Schmidt, warp 0)
            if (wid == 0) {
                const float gap = 1e-3f * s_tnorm;
                for (int j = 1; j < k; ++j) {
                    bool any = false;
                    for (int i = 0; i < j; ++i) {
                        if (fabsf(lamd[i] - lamd[j]) > gap) continue;
                        any = true;
                        float dot = 0.0f;
                        for (int r = lane; r < F; r += 32) dot += Z[r * zk + i] * Z[r * zk + j];
                        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                        for (int r = lane; r < F; r += 32) Z[r * zk + j] -= dot * Z[r * zk + i];
                        __syncwarp();
                    }
                    if (any) {
                        float n2 = 0.0f;
                        for (int r = lane; r < F; r += 32) n2 += Z[r * zk + j] * Z[r * zk + j];
                        for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                        const float inv = rsqrtf(n2);
                        for (int r = lane; r < F; r += 32) Z[r * zk + j] *= inv;
                        __syncwarp();
                    }
                }
            }
            for (int j = tid; j < F; j += nt) perm[j] = j;
            __syncthreads();
            // reflectors staged behind the k vectors (2 nbuf F complex values)
            const int nbuf = min(16, (F - zk) / 4);
            if (!big && nbuf > 0)
                back_transform(F, k, reinterpret_cast<float *>(dyn), zk, perm, delta, hv, tau_g, V, Vt,
                               dyn + (F * zk + 1) / 2, nbuf, lane, wid, nw);
            else
                back_transform(F, k, Z, zk, perm, delta, hv, tau_g, V, Vt, nullptr, 0, lane, wid, nw);
            if (k <= kRefineMaxK && k < F)
                refine_vectors<L2>(G, ginv, F, k, lamd, big || 2 * k > F + 1 ? reinterpret_cast<float2 *>(ii_scr) : dyn, V, Vt, lane, wid, nw);
            return;
        }
    }
    // Z = identity (stride F+1), reusing the packed-matrix storage
    for (int i = tid; i < F * zs; i += nt) Z[i] = ((i / zs) == (i % zs)) ? 1.0f : 0.0f;
    __syncthreads();

    // ---- implicit QL; thread 0 runs the scalar recurrence, everybody applies the
    // rotations.  An off-diagonal counts as zero below the rounding of its
    // neighbours or a thousandth of that of the whole matrix; where ten sweeps (two or
    // three are usual) have not come to that, the sweeps' own rounding keeps it
    // above, and the rounding of the whole matrix is what can be had (without this
    // 1 of 8 matrices of 100 frames and half of those of 300 did not converge)
    float tnorm = 0.0f;
    if (tid == 0) {
        for (int i = 0; i < F; ++i) tnorm = fmaxf(tnorm, fabsf(d[i]) + fabsf(e[i]));
    }
    for (int l = 0; l < F; ++l) {
        int iter = 0;
        bool stop_all = false;
        while (true) {
            if (tid == 0) {
                int m = l;
                for (; m < F - 1; ++m) {
                    float dd = fabsf(d[m]) + fabsf(d[m + 1]);
                    if (fabsf(e[m]) <= FLT_EPSILON * dd || fabsf(e[m]) <= (iter < 10 ? 1e-3f : 1.0f) * FLT_EPSILON * tnorm) break;
                }
                s_done = (m == l);
                s_nrot = 0;
                if (m != l) {
                    if (++iter > 60) {
                        s_fail = 1;
                        s_done = 1;
                    } else {
                        float g = (d[l + 1] - d[l]) / (2.0f * e[l]);
                        float r = sqrtf(fmaf(g, g, 1.0f));
                        g = d[m] - d[l] + e[l] / (g + copysignf(r, g));
                        float s = 1.0f, c = 1.0f, p = 0.0f;
                        bool early = false;
                        int nrot = 0;
                        for (int i = m - 1; i >= l; --i) {
                            float f = s * e[i], b = c * e[i];
                            // r = |(f, g)| and 1/r from one reciprocal square root plus a
                            // Newton step (the matrix is scaled to max |entry| = 1, so no
                            // overflow is possible)
                            const float q = fmaf(f, f, g * g);
                            if (q == 0.0f) {
                                e[i + 1] = 0.0f;
                                d[i + 1] -= p;
                                e[m] = 0.0f;
                                early = true;
                                break;
                            }
                            float rr = rsqrtf(q);
                            rr = rr * fmaf(-0.5f * q * rr, rr, 1.5f);
                            r = q * rr;
                            e[i + 1] = r;
                            s = f * rr;
                            c = g * rr;
                            g = d[i + 1] - p;
                            r = (d[i] - g) * s + 2.0f * c * b;
                            p = s * r;
                            d[i + 1] = g + p;
                            g = c * r - b;
                            rc[nrot] = c;
                            rs[nrot] = s;
                            ++nrot;
                        }
                        if (!early) {
                            d[l] -= p;
                            e[l] = g;
                            e[m] = 0.0f;
                        }
                        s_nrot = nrot;
                        s_m = m;
                    }
                }
            }
            __syncthreads();
            // every thread reads the sweep description between the two barriers
            const int done = s_done, nrot = s_nrot, mm = s_m, fail = s_fail;
            if (!done) {
                // rotation r acts on columns (i, i+1) with i = m - 1 - r
                for (int row = tid; row < F; row += nt) {
                    float *zr = Z + row * zs;
                    for (int r = 0; r < nrot; ++r) {
                        int i = mm - 1 - r;
                        float c = rc[r], s = rs[r];
                        float t = zr[i + 1];
                        zr[i + 1] = s * zr[i] + c * t;
                        zr[i] = c * zr[i] - s * t;
                    }
                }
            }
            __syncthreads();
            if (done) {
                stop_all = fail != 0;
                break;
            }
        }
        if (stop_all) break;
    }
    __syncthreads();
    // ---- sort descending (rank by value, ties by index)
    for (int i = tid; i < F; i += nt) {
        float di = d[i];
        int rank = 0;
        for (int j = 0; j < F; ++j) {
            float dj = d[j];
            rank += (dj > di) || (dj == di && j < i);
        }
        perm[rank] = i;
    }
    __syncthreads();
    for (int j = tid; j < F; j += nt) lam_out[j] = (double)d[perm[j]] * (double)gscale;
    if (tid == 0) {
        int k = k_cut;
        if (k < 0) {
            double tot = 0.0, acc = 0.0;
            for (int j = 0; j < F; ++j) tot += fmax((double)d[perm[j]], 0.0);
            k = F;
            for (int j = 0; j < F; ++j) {
                acc += fmax((double)d[perm[j]], 0.0);
                if (acc >= thresh * tot) { k = j + 1; break; }
            }
        }
        if (k_out) *k_out = k;
        if (status && s_fail) *status = FQ_ERR_NUMERICAL;
    }
    back_transform(F, F, Z, zs, perm, delta, hv, tau_g, V, Vt, nullptr, 0, lane, wid, nw);
}

template <int NT>
__global__ void __launch_bounds__(NT) eig_kernel(const float2 *__restrict__ G, int F, float2 *__restrict__ big,
                                                          float2 *__restrict__ hv, float *__restrict__ tau_g,
                                                          double *__restrict__ lam_out, float2 *__restrict__ V,
                                                          float2 *__restrict__ Vt, int k_cut, double thresh,
                                                          int *__restrict__ k_out, int *__restrict__ status,
                                                          int topk_only, float *__restrict__ ii_scr)
{
    eig_body<false>(G, F, big, hv, tau_g, lam_out, V, Vt, k_cut, thresh, k_out, status, topk_only, ii_scr, NT);
}

// One CTA per member, each with the threads of its single call, so that its sums
// are the same.
template <int NT>
__global__ void __launch_bounds__(NT) eig_batched_kernel(const fqb::EnsDev *__restrict__ ens,
                                                         const int *__restrict__ members)
{
    if (NT == kEigThreads) asm volatile("griddepcontrol.launch_dependents;");  // (see batched_eig)
    const fqb::EnsDev &e = ens[members[blockIdx.x]];
    char *ws = e.cws;
    double *lam = e.eigvals ? e.eigvals : (double *)(ws + e.cl_lam);
    int *kk = e.k_used ? e.k_used : (int *)(ws + e.cl_k);
    eig_body<NT == kTopThreads>((const float2 *)(ws + e.cl_G), e.F, eig_in_smem(e.F) ? nullptr : (float2 *)(ws + e.cl_big), (float2 *)(ws + e.cl_hv),
             (float *)(ws + e.cl_tau), lam, (float2 *)(ws + e.cl_V), (float2 *)(ws + e.cl_Vt), e.k_cut,
             e.energy_thresh, kk, e.status, 1, (float *)(ws + e.cl_ii), NT);
    if (NT == kTopThreads) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------ projection + power Doppler --
// One warp per pixel: y_j = sum_f S[f] V[f][j] for j < k, then
// S_f = S - sum_j y_j conj(V[:, j]) and pd = mean |S_f|^2.  Lane l holds
// frames l, l + 32, ..: NQ (a power of two, 32 NQ >= F) of them, so that the
// unrolled loops issue no work for frames beyond F (with NQ fixed at 16, the
// loops of a 100-frame ensemble issued four times the instructions they
// needed and the kernel was issue-bound at ~20% of HBM bandwidth).

// the pixel's frames into registers (frames beyond F read as 0)
template <typename T, int NQ>
__device__ __forceinline__ void project_load(const T *__restrict__ S, int64_t p, int F, int lane, float2 (&s)[NQ])
{
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        int f = lane + 32 * q;
        s[q] = f < F ? fqi::load_c(S, p * F + f) : make_float2(0, 0);
    }
}

template <typename T, int NQ>
__device__ __forceinline__ void project_compute(const float2 (&s)[NQ], int64_t p, int F,
                                                const float2 *__restrict__ Vt, int k, T *__restrict__ S_f,
                                                float *__restrict__ pd, float invF, int lane)
{
    float2 sf[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) sf[q] = s[q];
    if (k >= F) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) sf[q] = make_float2(0, 0);
    } else {
        for (int j = 0; j < k; ++j) {
            const float2 *vj = Vt + (size_t)j * F;
            float2 y = make_float2(0, 0);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                int f = lane + 32 * q;
                if (f < F) {
                    float2 t = cmul(s[q], vj[f]);
                    y.x += t.x;
                    y.y += t.y;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                y.x += __shfl_xor_sync(0xffffffffu, y.x, o);
                y.y += __shfl_xor_sync(0xffffffffu, y.y, o);
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                int f = lane + 32 * q;
                if (f < F) {
                    float2 t = cmul(y, cconj(vj[f]));
                    sf[q].x -= t.x;
                    sf[q].y -= t.y;
                }
            }
        }
    }
    float e = 0.0f;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        int f = lane + 32 * q;
        if (f < F) {
            e += sf[q].x * sf[q].x + sf[q].y * sf[q].y;
            if (S_f) fqi::store_c(S_f, p * F + f, sf[q]);
        }
    }
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (pd && lane == 0) pd[p] = e * invF;
}

template <typename T, int NQ = 16>
__device__ __forceinline__ void project_pixel(const T *__restrict__ S, int64_t p, int F, const float2 *__restrict__ Vt,
                                              int k, T *__restrict__ S_f, float *__restrict__ pd, float invF, int lane)
{
    float2 s[NQ];
    project_load<T, NQ>(S, p, F, lane, s);
    project_compute<T, NQ>(s, p, F, Vt, k, S_f, pd, invF, lane);
}

template <typename T, int NQ>
__global__ void __launch_bounds__(256) project_pd_kernel(const T *__restrict__ S, int64_t P, int F,
                                                         const float2 *__restrict__ Vt, const int *__restrict__ k_ptr,
                                                         T *__restrict__ S_f, float *__restrict__ pd)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int k = min(*k_ptr, F);
    const float invF = 1.0f / (float)F;
    // 1.68 GB of FP32 S (2^21 pixels x 100 frames) in 0.58 ms: 43% of HBM
    // bandwidth; loading the next pixel's frames while one is filtered
    // measured the same, so the loop keeps one pixel per warp
    for (int64_t p = warp0; p < P; p += nwarps) project_pixel<T, NQ>(S, p, F, Vt, k, S_f, pd, invF, lane);
}

int pd_blocks(int64_t P);

// the projection for F <= 512 frames with the smallest frames-per-lane count
template <typename T>
fq_status launch_project(const void *S, int64_t P, int F, const float2 *Vt, const int *k, void *S_f, float *pd,
                         cudaStream_t st)
{
    const T *s = (const T *)S;
    T *sf = (T *)S_f;
    const int g = pd_blocks(P);
    if (F <= 32) project_pd_kernel<T, 1><<<g, 256, 0, st>>>(s, P, F, Vt, k, sf, pd);
    else if (F <= 64) project_pd_kernel<T, 2><<<g, 256, 0, st>>>(s, P, F, Vt, k, sf, pd);
    else if (F <= 128) project_pd_kernel<T, 4><<<g, 256, 0, st>>>(s, P, F, Vt, k, sf, pd);
    else if (F <= 256) project_pd_kernel<T, 8><<<g, 256, 0, st>>>(s, P, F, Vt, k, sf, pd);
    else project_pd_kernel<T, 16><<<g, 256, 0, st>>>(s, P, F, Vt, k, sf, pd);
    return fqi::launch_check("projection + power Doppler");
}

// ------------------------------------------------------------- batched --
template <typename T>
__global__ void __launch_bounds__(kGramThreads, kGramCtas) gram_batched_kernel(const fqb::EnsDev *__restrict__ ens, const fqb::StageQueue q)
{
    extern __shared__ float4 panel[];
    __shared__ int s_buf[2];
    fqb::Item it;
    while (fqb::next_item(q, ens, fqb::ST_GRAM, s_buf, it)) {
        const fqb::EnsDev &e = ens[it.e];
        float2 *part = (float2 *)(e.cws + e.cl_part);
        if (gram_px(e.F) == 16) gram_part<16, T>((const T *)e.iq, e.P, e.F, e.chunk_len, part, it.x, it.y, panel);
        else gram_part<8, T>((const T *)e.iq, e.P, e.F, e.chunk_len, part, it.x, it.y, panel);
    }
}

__global__ void __launch_bounds__(256) gram_reduce_batched_kernel(const fqb::EnsDev *__restrict__ ens,
                                                                  const fqb::StageQueue q)
{
    __shared__ float2 red[kGramThreads / kReduceItem][kReduceItem];
    __shared__ int s_buf[2];
    fqb::Item it;
    while (fqb::next_item(q, ens, fqb::ST_GRAM_REDUCE, s_buf, it)) {
        const fqb::EnsDev &e = ens[it.e];
        for (int i = 0; i < kReduceItems; ++i)
            gram_reduce_at((const float2 *)(e.cws + e.cl_part), e.n_chunks, e.F, (float2 *)(e.cws + e.cl_G),
                           it.x * kReduceItems + i, red);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) project_batched_kernel(const fqb::EnsDev *__restrict__ ens,
                                                              const fqb::StageQueue q)
{
    __shared__ int s_buf[2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    fqb::Item it;
    while (fqb::next_item(q, ens, fqb::ST_PROJECT, s_buf, it)) {
        const fqb::EnsDev &e = ens[it.e];
        const int *kk = e.k_used ? e.k_used : (const int *)(e.cws + e.cl_k);
        const int k = min(*kk, e.F);
        const float invF = 1.0f / (float)e.F;
        const int64_t beg = (int64_t)it.x * fqb::kItemPix;
        const int64_t end = beg + fqb::kItemPix < e.P ? beg + fqb::kItemPix : e.P;
        // the frames-per-lane count of the single-ensemble projection, so
        // that both give bit-identical results
        const T *S = (const T *)e.iq;
        const float2 *Vt = (const float2 *)(e.cws + e.cl_Vt);
        for (int64_t p = beg + wid; p < end; p += 8) {
            if (e.F <= 32) project_pixel<T, 1>(S, p, e.F, Vt, k, (T *)nullptr, e.pd, invF, lane);
            else if (e.F <= 64) project_pixel<T, 2>(S, p, e.F, Vt, k, (T *)nullptr, e.pd, invF, lane);
            else if (e.F <= 128) project_pixel<T, 4>(S, p, e.F, Vt, k, (T *)nullptr, e.pd, invF, lane);
            else if (e.F <= 256) project_pixel<T, 8>(S, p, e.F, Vt, k, (T *)nullptr, e.pd, invF, lane);
            else project_pixel<T, 16>(S, p, e.F, Vt, k, (T *)nullptr, e.pd, invF, lane);
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256) power_doppler_kernel(const T *__restrict__ S, int64_t P, int F,
                                                            float *__restrict__ pd)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = warp0; p < P; p += nwarps) {
        float e = 0.0f;
        for (int f = lane; f < F; f += 32) {
            float2 v = fqi::load_c(S, p * F + f);
            e += v.x * v.x + v.y * v.y;
        }
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0) pd[p] = e / (float)F;
    }
}

// ------------------------------------------------------------- launchers --
template <typename T>
fq_status launch_gram(const void *S, int64_t P, int F, const ClutterLayout &L, char *ws, float2 *G, cudaStream_t st)
{
    float2 *part = (float2 *)(ws + L.part);
    const size_t smem = gram_smem(F);
    auto kern = gram_px(F) == 16 ? gram_partial_kernel<16, T> : gram_partial_kernel<8, T>;
    fq_status s = fqi::cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)gram_smem_upto(kMaxF)), "fq_casorati_gram: smem attribute");
    if (s) return s;
    dim3 grid(gram_parts(F), L.n_chunks);
    kern<<<grid, kGramThreads, smem, st>>>((const T *)S, P, F, L.chunk_len, part);
    gram_reduce_kernel<<<(F * F + kReduceItem - 1) / kReduceItem, kGramThreads, 0, st>>>(part, L.n_chunks, F, G);
    return fqi::launch_check("fq_casorati_gram");
}

// Gram of gram_mode into G; the tensor-core modes use the L.tc region and
// report a timed-out wait through the status word at ws.
fq_status gram_any(const void *S, int dtype, int64_t P, int F, int gram_mode, const ClutterLayout &L, char *ws,
                   float2 *G, cudaStream_t st)
{
    const int esz = tc_esz(gram_mode);
    if (esz) return fqi::gram_tc(S, dtype, P, F, esz, G, ws + L.tc, (int *)(ws + L.status), st);
    return dtype == FQ_F32 ? launch_gram<float>(S, P, F, L, ws, G, st) : launch_gram<__nv_bfloat16>(S, P, F, L, ws, G, st);
}

fq_status launch_eig(const float2 *G, int F, float2 *big, float2 *hv, float *tau, double *lam, float2 *V, float2 *Vt,
                     int k_cut, double thresh, int *k_out, int *status, cudaStream_t st, int topk_only = 0,
                     float *ii_scr = nullptr)
{
    size_t smem = big ? 0 : sizeof(float2) * (size_t)F * (F + 1) / 2;
    const int nt = topk_only ? top_threads(F) : kEigThreads;
    auto kern = nt == kTopThreads ? eig_kernel<kTopThreads> : eig_kernel<kEigThreads>;
    if (smem > 0) {
        // the kernel's static arrays count against the same 48 KB default,
        // so the opt-in is needed for much smaller packed matrices too
        fq_status s = fqi::cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)kEigSmemMax), "eig: smem attribute");
        if (s) return s;
    }
    kern<<<1, nt, smem, st>>>(G, F, big, hv, tau, lam, V, Vt, k_cut, thresh, k_out,
                                                                status, topk_only, ii_scr);
    return fqi::launch_check("fq_hermitian_eig");
}

// ---------------------------------------------------- no-allocation variant --
// Scratch for fq_clutter_svd_noalloc: one fixed array per device that loads
// the library.  Its host-side name is only a stand-in; kernels get the
// device address that cudaGetSymbolAddress returns for the current device.
constexpr size_t kNoallocBytes = (size_t)12 << 20;
constexpr int kNoallocMaxF = 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

// The workspace layout of the clutter filter with the Gram partial sums (pixel
// chunks) that the array holds: at most 151 of the 228 that a workspace has at
// 100 frames, 34 of 91 at 200, 18 of 50 at 256; of those the count whose CTAs
// load the SMs most evenly (18 chunks of 9 parts at 256 frames would leave most SMs
// one CTA and a few two: 16).  2^21 x 100: 4.13 ms (16 chunks at any F: 18.5;
// with a workspace 3.86); 65536 x 200: 1.66 (1.95).
ClutterLayout layout_noalloc(int64_t P, int F)
{
    const ClutterLayout one = layout(P, F, FQ_GRAM_F32, false, 1);
    if (one.total > kNoallocBytes) return one;  // (the caller refuses it)
    const int most = 1 + (int)std::min<size_t>((kNoallocBytes - one.total) / (sizeof(float2) * F * F), 1 << 20);
    const int cap = std::min(most, gram_chunks(P, F)), parts = gram_parts(F);
    auto cost = [&](int n) { return (double)((n * parts + 151) / 152) / n; };  // CTAs of an SM x pixels of each
    int best = cap;
    for (int n = cap; n >= 1; --n)
        if (cost(n) < 0.97 * cost(best)) best = n;
    return layout(P, F, FQ_GRAM_F32, false, best);
}

// Unique ID of the calling thread's current CUDA context (0 if none), from
// the driver's cuCtxGetCurrent / cuCtxGetId, fetched once through the
// runtime so that the library needs no link to the driver library.
unsigned long long current_context_id()
{
    using GetCurrent = CUresult (*)(CUcontext *);
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = (GetCurrent)f;
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = (GetId)f;
    });
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

// Device address of the scratch array on the current device.  It is looked
// up (with that device current) the first time and again whenever the
// device's current context has changed since (a device reset destroys the
// context that the cached address belongs to), and cached otherwise.
fq_status noalloc_scratch(char **out)
{
    constexpr int kMaxDevices = 64;
    static void *addr[kMaxDevices] = {};
    static unsigned long long ctx_id[kMaxDevices] = {};
    static std::mutex mu;
    int dev = 0;
    fq_status s = fqi::cuda_check(cudaGetDevice(&dev), "fq_clutter_svd_noalloc: cudaGetDevice");
    if (s) return s;
    FQ_REQUIRE(dev >= 0 && dev < kMaxDevices, FQ_ERR_UNSUPPORTED, "fq_clutter_svd_noalloc: device ordinal %d", dev);
    std::lock_guard<std::mutex> lock(mu);
    const unsigned long long id = current_context_id();
    if (!addr[dev] || id == 0 || id != ctx_id[dev]) {
        void *p = nullptr;
        s = fqi::cuda_check(cudaGetSymbolAddress(&p, g_noalloc_scratch),
                            "fq_clutter_svd_noalloc: cudaGetSymbolAddress");
        if (s) return s;
        addr[dev] = p;
        ctx_id[dev] = current_context_id();  // the lookup makes the device's context current if it was not
    }
    *out = (char *)addr[dev];
    return FQ_OK;
}

int pd_blocks(int64_t P)
{
    int64_t b = (P + 7) / 8;
    return (int)(b < 152 * 16 ? b : 152 * 16);
}

}  // namespace

extern "C" {

fq_status fq_gram_workspace_size(int64_t P, int32_t F, int32_t gram_mode, size_t *bytes)
{
    FQ_REQUIRE(bytes && P >= 1 && F >= 2 && F <= 512, FQ_ERR_INVALID_ARG, "fq_gram_workspace_size: bad arguments");
    FQ_REQUIRE(gram_mode >= FQ_GRAM_F32 && gram_mode <= FQ_GRAM_BF16, FQ_ERR_INVALID_ARG,
               "fq_gram_workspace_size: gram_mode %d", gram_mode);
    const int esz = tc_esz(gram_mode);
    if (esz) {
        *bytes = 256 + fqi::gram_tc_workspace_bytes(P, F, esz);  // status word + operands + partials
        return FQ_OK;
    }
    ClutterLayout L = layout(P, F);
    *bytes = al256(sizeof(float2) * (size_t)L.n_chunks * F * F);
    return FQ_OK;
}

fq_status fq_casorati_gram(const void *S, int32_t dtype, int64_t P, int32_t F, int32_t gram_mode, float *G,
                           void *workspace, size_t workspace_bytes, void *stream)
{
    FQ_REQUIRE(S && G && P >= 1 && F >= 2 && F <= 512, FQ_ERR_INVALID_ARG, "fq_casorati_gram: bad arguments");
    FQ_REQUIRE(gram_mode >= FQ_GRAM_F32 && gram_mode <= FQ_GRAM_BF16, FQ_ERR_INVALID_ARG,
               "fq_casorati_gram: gram_mode %d", gram_mode);
    FQ_REQUIRE(dtype == FQ_F32 || dtype == FQ_BF16, FQ_ERR_UNSUPPORTED, "fq_casorati_gram: dtype");
    size_t need = 0;
    fq_gram_workspace_size(P, F, gram_mode, &need);
    FQ_REQUIRE(workspace && workspace_bytes >= need, FQ_ERR_WORKSPACE, "fq_casorati_gram: workspace needs %zu bytes",
               need);
    FQ_REQUIRE(fqi::aligned(workspace, 256) && fqi::aligned(S, 8) && fqi::aligned(G, 8), FQ_ERR_ALIGN,
               "fq_casorati_gram: alignment");
    cudaStream_t st = (cudaStream_t)stream;
    const int esz = tc_esz(gram_mode);
    if (esz) {
        fq_status s = fqi::cuda_check(cudaMemsetAsync(workspace, 0, 256, st), "fq_casorati_gram: status reset");
        if (s) return s;
        return fqi::gram_tc(S, dtype, P, F, esz, (float2 *)G, (char *)workspace + 256, (int *)workspace, st);
    }
    ClutterLayout L = layout(P, F);
    L.part = 0;  // the partials are the only workspace content here
    if (dtype == FQ_F32) return launch_gram<float>(S, P, F, L, (char *)workspace, (float2 *)G, st);
    return launch_gram<__nv_bfloat16>(S, P, F, L, (char *)workspace, (float2 *)G, st);
}

fq_status fq_eig_workspace_size(int32_t F, size_t *bytes)
{
    FQ_REQUIRE(bytes && F >= 1 && F <= 512, FQ_ERR_INVALID_ARG, "fq_eig_workspace_size: F must be in [1, 512]");
    *bytes = eig_only_bytes(F);
    return FQ_OK;
}

fq_status fq_hermitian_eig(const float *G, int32_t F, double *eigvals, float *V, void *workspace,
                           size_t workspace_bytes, void *stream)
{
    FQ_REQUIRE(G && eigvals && V && F >= 1 && F <= 512, FQ_ERR_INVALID_ARG, "fq_hermitian_eig: bad arguments");
    size_t need = eig_only_bytes(F);
    FQ_REQUIRE(workspace && workspace_bytes >= need, FQ_ERR_WORKSPACE, "fq_hermitian_eig: workspace needs %zu bytes",
               need);
    FQ_REQUIRE(fqi::aligned(workspace, 256) && fqi::aligned(G, 8) && fqi::aligned(V, 8), FQ_ERR_ALIGN,
               "fq_hermitian_eig: alignment");
    char *ws = (char *)workspace;
    size_t o = 256;
    float2 *hv = (float2 *)(ws + o); o += al256(sizeof(float2) * F * F);
    float *tau = (float *)(ws + o); o += al256(sizeof(float) * F);
    float2 *Vt = (float2 *)(ws + o); o += al256(sizeof(float2) * F * F);
    int *kk = (int *)(ws + o); o += 256;
    float2 *big = eig_in_smem(F) ? nullptr : (float2 *)(ws + o);
    cudaStream_t st = (cudaStream_t)stream;
    fq_status s = fqi::cuda_check(cudaMemsetAsync(ws, 0, 256, st), "fq_hermitian_eig: status reset");
    if (s) return s;
    return launch_eig((const float2 *)G, F, big, hv, tau, eigvals, (float2 *)V, Vt, 0, 0.0, kk, (int *)ws, st);
}

fq_status fq_clutter_svd_workspace_size(int64_t P, int32_t F, int32_t gram_mode, size_t *bytes)
{
    FQ_REQUIRE(bytes && P >= 1 && F >= 2 && F <= 512, FQ_ERR_INVALID_ARG,
               "fq_clutter_svd_workspace_size: bad arguments");
    FQ_REQUIRE(gram_mode >= FQ_GRAM_F32 && gram_mode <= FQ_GRAM_BF16, FQ_ERR_INVALID_ARG,
               "fq_clutter_svd_workspace_size: gram_mode %d", gram_mode);
    *bytes = layout(P, F, gram_mode).total;
    return FQ_OK;
}

fq_status fq_clutter_svd(const void *iq, int32_t dtype, int64_t P, int32_t F, int32_t k_cut, double energy_thresh,
                         int32_t gram_mode, void *iq_f, float *pd, double *eigvals, int32_t *k_used, void *workspace,
                         size_t workspace_bytes, void *stream)
{
    FQ_REQUIRE(iq && P >= 1 && F >= 2 && F <= 512, FQ_ERR_INVALID_ARG, "fq_clutter_svd: bad arguments");
    FQ_REQUIRE(k_cut <= F, FQ_ERR_INVALID_ARG, "fq_clutter_svd: k_cut %d > F %d", k_cut, F);
    FQ_REQUIRE(k_cut >= 0 || (energy_thresh > 0.0 && energy_thresh <= 1.0), FQ_ERR_INVALID_ARG,
               "fq_clutter_svd: energy_thresh must be in (0, 1] when k_cut < 0");
    FQ_REQUIRE(dtype == FQ_F32 || dtype == FQ_BF16, FQ_ERR_UNSUPPORTED, "fq_clutter_svd: dtype");
    FQ_REQUIRE(gram_mode >= FQ_GRAM_F32 && gram_mode <= FQ_GRAM_BF16, FQ_ERR_INVALID_ARG,
               "fq_clutter_svd: gram_mode %d", gram_mode);
    ClutterLayout L = layout(P, F, gram_mode);
    FQ_REQUIRE(workspace && workspace_bytes >= L.total, FQ_ERR_WORKSPACE,
               "fq_clutter_svd: workspace needs %zu bytes", L.total);
    FQ_REQUIRE(fqi::aligned(workspace, 256) && fqi::aligned(iq, 8) && fqi::aligned(iq_f, 8), FQ_ERR_ALIGN,
               "fq_clutter_svd: alignment");
    char *ws = (char *)workspace;
    cudaStream_t st = (cudaStream_t)stream;
    fq_status s = fqi::cuda_check(cudaMemsetAsync(ws, 0, 256, st), "fq_clutter_svd: status reset");
    if (s) return s;
    float2 *G = (float2 *)(ws + L.G);
    s = gram_any(iq, dtype, P, F, gram_mode, L, ws, G, st);
    if (s) return s;
    double *lam = eigvals ? eigvals : (double *)(ws + L.lam);
    int *kk = k_used ? (int *)k_used : (int *)(ws + L.k);
    float2 *big = eig_in_smem(F) ? nullptr : (float2 *)(ws + L.big);
    s = launch_eig(G, F, big, (float2 *)(ws + L.hv), (float *)(ws + L.tau), lam, (float2 *)(ws + L.V),
                   (float2 *)(ws + L.Vt), k_cut, energy_thresh, kk, (int *)ws, st, 1, (float *)(ws + L.ii));
    if (s) return s;
    if (!iq_f && !pd) return FQ_OK;
    if (dtype == FQ_F32) return launch_project<float>(iq, P, F, (const float2 *)(ws + L.Vt), kk, iq_f, pd, st);
    return launch_project<__nv_bfloat16>(iq, P, F, (const float2 *)(ws + L.Vt), kk, iq_f, pd, st);
}

fq_status fq_power_doppler(const void *iq_f, int32_t dtype, int64_t P, int32_t F, float *pd, void *stream)
{
    FQ_REQUIRE(iq_f && pd && P >= 1 && F >= 1, FQ_ERR_INVALID_ARG, "fq_power_doppler: bad arguments");
    FQ_REQUIRE(fqi::aligned(iq_f, 8), FQ_ERR_ALIGN, "fq_power_doppler: iq_f must be 8-byte aligned");
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == FQ_F32)
        power_doppler_kernel<float><<<pd_blocks(P), 256, 0, st>>>((const float *)iq_f, P, F, pd);
    else if (dtype == FQ_BF16)
        power_doppler_kernel<__nv_bfloat16><<<pd_blocks(P), 256, 0, st>>>((const __nv_bfloat16 *)iq_f, P, F, pd);
    else
        return fqi::set_error(FQ_ERR_UNSUPPORTED, "fq_power_doppler: dtype");
    return fqi::launch_check("fq_power_doppler");
}

fq_status fq_clutter_status(void *workspace, void *stream)
{
    if (!workspace) {  // the built-in array of fq_clutter_svd_noalloc on the current device
        char *ws = nullptr;
        fq_status s = noalloc_scratch(&ws);
        if (s) return s;
        workspace = ws;
    }
    cudaStream_t st = (cudaStream_t)stream;
    int flag = 0;
    fq_status s = fqi::cuda_check(cudaMemcpyAsync(&flag, workspace, sizeof(int), cudaMemcpyDeviceToHost, st),
                                  "fq_clutter_status: read");
    if (s) return s;
    s = fqi::cuda_check(cudaStreamSynchronize(st), "fq_clutter_status: sync");
    if (s) return s;
    s = fqi::cuda_check(cudaMemsetAsync(workspace, 0, sizeof(int), st), "fq_clutter_status: clear");
    if (s) return s;
    if (flag) return fqi::set_error((fq_status)flag, "device solver reported %s", fq_status_string((fq_status)flag));
    return FQ_OK;
}


fq_status fq_clutter_svd_noalloc(const void *iq, int32_t dtype, int64_t P, int32_t F, int32_t k_cut,
                                 double energy_thresh, void *iq_f, float *pd, double *eigvals, int32_t *k_used,
                                 void *stream)
{
    FQ_REQUIRE(iq && P >= 1 && F >= 2, FQ_ERR_INVALID_ARG, "fq_clutter_svd_noalloc: bad arguments");
    FQ_REQUIRE(F <= kNoallocMaxF, FQ_ERR_SHAPE,
               "fq_clutter_svd_noalloc: F = %d frames exceeds the built-in scratch limit of %d frames; "
               "use fq_clutter_svd with a workspace", F, kNoallocMaxF);
    FQ_REQUIRE(k_cut <= F, FQ_ERR_INVALID_ARG, "fq_clutter_svd_noalloc: k_cut %d > F %d", k_cut, F);
    FQ_REQUIRE(k_cut >= 0 || (energy_thresh > 0.0 && energy_thresh <= 1.0), FQ_ERR_INVALID_ARG,
               "fq_clutter_svd_noalloc: energy_thresh must be in (0, 1] when k_cut < 0");
    FQ_REQUIRE(dtype == FQ_F32 || dtype == FQ_BF16, FQ_ERR_UNSUPPORTED, "fq_clutter_svd_noalloc: dtype");
    FQ_REQUIRE(fqi::aligned(iq, 8) && fqi::aligned(iq_f, 8), FQ_ERR_ALIGN, "fq_clutter_svd_noalloc: alignment");
    ClutterLayout L = layout_noalloc(P, F);
    FQ_REQUIRE(L.total <= kNoallocBytes, FQ_ERR_SHAPE,
               "fq_clutter_svd_noalloc: needs %zu scratch bytes, the built-in array has %zu", L.total, kNoallocBytes);
    char *ws = nullptr;
    fq_status s = noalloc_scratch(&ws);
    if (s) return s;
    cudaStream_t st = (cudaStream_t)stream;
    // the status word must start at zero; everything else is fully rewritten
    s = fqi::cuda_check(cudaMemsetAsync(ws, 0, 256, st), "fq_clutter_svd_noalloc: status reset");
    if (s) return s;
    float2 *G = (float2 *)(ws + L.G);
    s = dtype == FQ_F32 ? launch_gram<float>(iq, P, F, L, ws, G, st) : launch_gram<__nv_bfloat16>(iq, P, F, L, ws, G, st);
    if (s) return s;
    double *lam = eigvals ? eigvals : (double *)(ws + L.lam);
    int *kk = k_used ? (int *)k_used : (int *)(ws + L.k);
    float2 *big = eig_in_smem(F) ? nullptr : (float2 *)(ws + L.big);
    s = launch_eig(G, F, big, (float2 *)(ws + L.hv), (float *)(ws + L.tau), lam, (float2 *)(ws + L.V),
                   (float2 *)(ws + L.Vt), k_cut, energy_thresh, kk, (int *)ws, st, 1, (float *)(ws + L.ii));
    if (s) return s;
    if (!iq_f && !pd) return FQ_OK;
    if (dtype == FQ_F32) return launch_project<float>(iq, P, F, (const float2 *)(ws + L.Vt), kk, iq_f, pd, st);
    return launch_project<__nv_bfloat16>(iq, P, F, (const float2 *)(ws + L.Vt), kk, iq_f, pd, st);
}

}  // extern "C"

namespace fqi {

void clutter_layout_batched(int64_t P, int F, size_t off[10], int *n_chunks, int64_t *chunk_len, size_t *total)
{
    const ClutterLayout L = layout(P, F, FQ_GRAM_F32, true);
    const size_t o[10] = {L.G, L.part, L.V, L.Vt, L.lam, L.k, L.hv, L.tau, L.big, L.ii};
    for (int i = 0; i < 10; ++i) off[i] = o[i];
    *n_chunks = L.n_chunks;
    *chunk_len = L.chunk_len;
    *total = L.total;
}

template <typename T>
fq_status launch_gram_batched(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, int F_max, cudaStream_t st)
{
    const size_t smem = gram_smem_upto(F_max);
    auto kern = gram_batched_kernel<T>;
    fq_status s = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  (int)gram_smem_upto(kMaxF)), "batched Gram: smem attribute");
    if (s) return s;
    kern<<<fqb::persistent_grid(kern, kGramThreads, smem, items), kGramThreads, smem, st>>>(ens, q);
    return launch_check("batched Gram");
}

fq_status batched_gram(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, int iq_dtype, int F_max, cudaStream_t st)
{
    return iq_dtype == FQ_F32 ? launch_gram_batched<float>(ens, q, items, F_max, st)
                              : launch_gram_batched<__nv_bfloat16>(ens, q, items, F_max, st);
}

void gram_item_counts(int F, int *parts, int *reduce_items)
{
    *parts = gram_parts(F);
    *reduce_items = (F * F + kReduceItem * kReduceItems - 1) / (kReduceItem * kReduceItems);
}

fq_status batched_gram_reduce(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, cudaStream_t st)
{
    gram_reduce_batched_kernel<<<fqb::persistent_grid(gram_reduce_batched_kernel, 256, 0, items), 256, 0, st>>>(ens,
                                                                                                               q);
    return launch_check("batched Gram reduce");
}

// Matrices too large for shared memory in a launch of their own without any: they
// live in the L1 cache as far as they fit, and shared memory for the other
// members' matrices took it from them (6 members of 240 frames 3.8 -> 2.64 ms, of
// 400 14.4 -> 9.4).  The other members' launch starts as soon as
// all CTAs of the first run (programmatic launch; it reads nothing of theirs, and
// the Gram matrices, which were complete before them, from L2) and ends after them, so that the stages that follow see both (6 members of 50 to 300
// frames: 3.97 ms, one after the other 5.33, in one launch 5.5).
fq_status batched_eig(const fqb::EnsDev *ens, const int *members, const int *F, int n, cudaStream_t st)
{
    int big = 0;
    while (big < n && !eig_in_smem(F[big])) ++big;
    if (big > 0) eig_batched_kernel<kEigThreads><<<big, kEigThreads, 0, st>>>(ens, members);
    if (big < n) {
        auto kern = eig_batched_kernel<kTopThreads>;
        fq_status s = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      (int)kEigSmemMax), "batched eig: smem attribute");
        if (s) return s;
        cudaLaunchAttribute early;
        early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        early.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n - big);
        cfg.blockDim = dim3(kTopThreads);
        cfg.dynamicSmemBytes = sizeof(float2) * (size_t)F[big] * (F[big] + 1) / 2;
        cfg.stream = st;
        cfg.attrs = &early;
        cfg.numAttrs = big > 0 ? 1 : 0;
        s = cuda_check(cudaLaunchKernelEx(&cfg, kern, ens, members + big), "batched eig");
        if (s) return s;
    }
    return launch_check("batched eig");
}

fq_status batched_project(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, int iq_dtype, cudaStream_t st)
{
    if (iq_dtype == FQ_F32)
        project_batched_kernel<float>
            <<<fqb::persistent_grid(project_batched_kernel<float>, 256, 0, items), 256, 0, st>>>(ens, q);
    else
        project_batched_kernel<__nv_bfloat16>
            <<<fqb::persistent_grid(project_batched_kernel<__nv_bfloat16>, 256, 0, items), 256, 0, st>>>(ens, q);
    return launch_check("batched projection");
}

}  // namespace fqi
