// Gridding NUFFT of the multicoil operator of Eq. (1) (Sec. 2.1):
//   forward (a2): apodise + coil-multiply + zero-pad fused into the row FFT,
//                 column FFT, Kaiser-Bessel interpolation (gather);
//   adjoint (a3): tile-owned KB spreading (shared-memory tiles, no atomics),
//                 column IFFT, row IFFT fused with crop + deapodisation +
//                 conj(S_l) coil sum.
// All grids are coil-innermost ([gy][gx][l]) so a grid tap is L contiguous
// complex values.
#include <algorithm>
#include <cstring>

#include "fft16.cuh"
#include "plan.cuh"

using namespace hqs;

// phi(t) = I0(beta sqrt(1 - (2t/W)^2)) on |t| <= W/2.
HQS_DEV float kb_phi(float t, float W, float beta) {
    const float z = 2.0f * t / W;
    const float s = 1.0f - z * z;
    return s >= 0.f ? cyl_bessel_i0f(beta * sqrtf(s)) : 0.f;
}

// image pixel held at oversampled-grid position p (centred layout), or -1
HQS_DEV int grid_to_pix(int p, int n, int G) {
    const int h = n >> 1;
    if (p < h) return p + h;
    if (p >= G - h) return p - G + h;
    return -1;
}
HQS_DEV int pix_to_grid(int i, int n, int G) {
    const int c = i - (n >> 1);
    return c >= 0 ? c : c + G;
}

// ---------------------------------------------------------------- forward
// Shared memory of the FFT passes: [G][kLines] lines | [G] twiddles.
template <int G> constexpr size_t nufft_smem_floats2() { return (size_t)G * kLines + G; }

// Row iy for the coils of chunk blockIdx.y: S_l x / (phihat phihat) placed at
// n mod G, FFT along x -> U[iy][gx][l].
template <int G>
__global__ void k_fwd_rows(const float2* __restrict__ x, const float2* __restrict__ smaps,
                           const float* __restrict__ apod, int n, int L, int LC, int nchunk,
                           float scale, const float2* __restrict__ twg, float2* __restrict__ U) {
    HQS_PDL_ENTRY();
    extern __shared__ float2 s[];
    const float2* tw = stage_twiddles<G>(s + G * kLines, twg);
    const int iy = blockIdx.x;
    const float ay = apod[iy] * scale;
    const int l0 = blockIdx.y * LC;
    const int lines = min(LC, L - l0);
    const int pst = blockDim.x / lines;
    const int l = threadIdx.x % lines, p0 = threadIdx.x / lines;
    if (p0 < pst) {
#pragma unroll 4
        for (int p = p0; p < G; p += pst) {
            const int ix = grid_to_pix(p, n, G);
            float2 v = make_float2(0.f, 0.f);
            if (ix >= 0) {
                const int64_t pix = (int64_t)iy * n + ix;
                v = cscale(cmul(smaps[pix * L + l0 + l], x[pix]), ay * apod[ix]);
            }
            s[p * kLines + l] = v;
        }
    }
    __syncthreads();
    block_fft<G, false>(s, lines, tw);
    float2* dst = U + (int64_t)iy * G * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 4
        for (int p = p0; p < G; p += pst) dst[(int64_t)p * L] = s[p * kLines + l];
    }
}

// Column gx: image rows at n mod G, zeros elsewhere, FFT along y -> Ghat.
template <int G>
__global__ void k_fwd_cols(const float2* __restrict__ U, int n, int L, int LC, int nchunk,
                           const float2* __restrict__ twg, float2* __restrict__ Gh) {
    HQS_PDL_ENTRY();
    extern __shared__ float2 s[];
    const float2* tw = stage_twiddles<G>(s + G * kLines, twg);
    const int gx = blockIdx.x;
    const int l0 = blockIdx.y * LC;
    const int lines = min(LC, L - l0);
    const int pst = blockDim.x / lines;
    const int l = threadIdx.x % lines, p0 = threadIdx.x / lines;
    const int64_t rs = (int64_t)G * L;
    const float2* col = U + (int64_t)gx * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 8
        for (int p = p0; p < G; p += pst) {
            const int iy = grid_to_pix(p, n, G);
            s[p * kLines + l] = iy >= 0 ? col[iy * rs] : make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    block_fft<G, false>(s, lines, tw);
    float2* dst = Gh + (int64_t)gx * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 4
        for (int p = p0; p < G; p += pst) dst[p * rs] = s[p * kLines + l];
    }
}

// ---- passes with the image in the lower half of each line (G = 2n)
// With G = 2n the centred placement p = (i - n/2) mod G of pixel i is the circular
// shift by n/2 of position q = i, so FFT_G of the centred line is i^k times the FFT of
// the line holding the image in its lower half [0, n), and the centred output pixels
// of an inverse transform are the lower half of the inverse of (-i)^k X[k].  Half of
// every line is then zero or not wanted, and the two-stage transforms of fft16.cuh
// apply (the rotations folded into their lane factors), at any coil count: 320^2 x 16
// coils forward 55.5 -> 51.1 us, adjoint 98.8 -> 85.5; 384^2 x 13 coils, whose passes
// were the general ones below, adjoint 178 -> 145; 320^2 x 2 coils forward 82 -> 24.  Grids of
// 32 and 64 points keep the radix-8 stages with the rotations on load and store, for
// full 16-coil chunks.
// v * i^k and v * (-i)^k, k >= 0, with selects (k differs from lane to lane: no branches)
HQS_DEV float2 mul_ipow(float2 v, int k) {
    const bool odd = k & 1, neg = k & 2;
    const float re = odd ? -v.y : v.x, im = odd ? v.x : v.y;
    return neg ? make_float2(-re, -im) : make_float2(re, im);
}
HQS_DEV float2 mul_mipow(float2 v, int k) {
    const bool odd = k & 1, neg = k & 2;
    const float re = odd ? v.y : v.x, im = odd ? -v.x : v.y;
    return neg ? make_float2(-re, -im) : make_float2(re, im);
}

// Arguments of the lower-half FFT passes of one plan (G = 2n), for the single-slice
// launches and, in a table over slices, the batched ones.
struct HalfArgs {
    const float2* x;       // forward: image
    float2* xo;            // adjoint: image (out)
    const float2* z;       // adjoint: xo = A^H y + zc z when z is given
    float zc;
    const float2* smaps;   // [n][n][L]
    const float* apod;     // [n]
    const float2* tw;      // G-point twiddles, in the order the size's transforms read
    float2* work;          // [n][G][L]
    float2* grid;          // [G][G][L]
    float2* part;          // [nchunk][n][n] coil-chunk sums (nchunk > 1)
    int n, L, LC, nchunk;
    float scale;
};
template <int G, int LINES> constexpr int half_threads() {
    return fft16_ok<G>() ? 16 * LINES : FftSize<G>::TPL * kLines;
}
template <int G, int LINES> constexpr size_t half_smem() { return ((size_t)G * LINES + G) * sizeof(float2); }
// the twiddle table, copied with cp.async (the pass waits for it before its first barrier)
template <int G> HQS_DEV void half_twiddles(float2* dst, const float2* __restrict__ tw) {
    for (int c = threadIdx.x; c < G / 2; c += blockDim.x) cp_async16(dst + 2 * c, tw + 2 * c);
}

// FFT of `lines` lines from ld(line, q) (q < n) to st(line, k)
template <int G, int LINES, class LD, class ST>
HQS_DEV void half_forward(float2* s, const float2* twg, int lines, LD&& ld, ST&& st) {
    float2* tw = s + (size_t)G * LINES;
    half_twiddles<G>(tw, twg);
    if constexpr (fft16_ok<G>()) {
        const Lane16 T(LINES);
        const bool act = T.line < lines;
        const int ln = act ? T.line : 0;
        fft16_head<G, LINES, true>(s, T, [&](int q) { return ld(ln, q); });
        cp_async_wait_all();
        __syncthreads();
        float2 v[Fft16<G>::R];
        fft16_mid_read<G, LINES>(s, T, v);
        fft16_mid_fwd<G>(T, tw, v);
        if (act) {
#pragma unroll
            for (int m = 0; m < Fft16<G>::R; ++m) st(ln, T.t + 16 * m, v[m]);
        }
    } else {
        cp_async_wait_all();
        __syncthreads();
        block_fft_io<G, false, true, false>(
            s, lines, tw, [&](int line, int q, bool) { return ld(line, q); }, NoIO{},
            [&](int line, int k, float2 v) { st(line, k, mul_ipow(v, k)); });
    }
}

// The forward passes take chunks of LINES coils, at most 8 for the two-stage transforms
// (their lines do not meet, see toep_impl in toeplitz.cu; 320^2 x 16 coils forward 48.0 ->
// 44.1 us).  The adjoint's columns, which load a whole line per thread at once, are slower
// that way (384^2 x 13 coils adjoint 94.7 -> 102 us) and keep the plan's chunks.
template <int G, int LINES> HQS_DEV void fwd_rows_h_item(const HalfArgs& A, int iy, int ch, float2* s) {
    const int n = A.n, L = A.L, l0 = ch * LINES;
    const float ay = A.apod[iy] * A.scale;
    const float2* xr = A.x + (int64_t)iy * n;
    const float2* sm = A.smaps + (int64_t)iy * n * L + l0;
    const float* apod = A.apod;
    float2* dst = A.work + (int64_t)iy * G * L + l0;
    half_forward<G, LINES>(
        s, A.tw, min(LINES, L - l0),
        [&](int line, int q) { return cscale(cmul(__ldg(sm + (int64_t)q * L + line), __ldg(xr + q)), ay * __ldg(apod + q)); },
        [&](int line, int k, float2 v) { dst[(int64_t)k * L + line] = v; });
}

template <int G, int LINES> HQS_DEV void fwd_cols_h_item(const HalfArgs& A, int gx, int ch, float2* s) {
    const int L = A.L, l0 = ch * LINES;
    const int64_t rs = (int64_t)G * L;
    const float2* col = A.work + (int64_t)gx * L + l0;
    float2* dst = A.grid + (int64_t)gx * L + l0;
    half_forward<G, LINES>(
        s, A.tw, min(LINES, L - l0), [&](int line, int q) { return __ldg(col + q * rs + line); },
        [&](int line, int k, float2 v) { dst[k * rs + line] = v; });
}

template <int G, int LINES> HQS_DEV void adj_cols_h_item(const HalfArgs& A, int gx, int ch, float2* s) {
    const int L = A.L, l0 = ch * A.LC, lines = min(A.LC, L - l0);
    const int64_t rs = (int64_t)G * L;
    const float2* col = A.grid + (int64_t)gx * L + l0;
    float2* dst = A.work + (int64_t)gx * L + l0;
    float2* tw = s + (size_t)G * LINES;
    half_twiddles<G>(tw, A.tw);
    if constexpr (fft16_ok<G>()) {
        const Lane16 T(LINES);
        const bool act = T.line < lines;
        const int ln = act ? T.line : 0;
        float2 v[Fft16<G>::R];
#pragma unroll
        for (int m = 0; m < Fft16<G>::R; ++m) v[m] = __ldg(col + (T.t + 16 * m) * rs + ln);
        cp_async_wait_all();
        __syncthreads();
        fft16_mid_inv<G>(T, tw, v);
        fft16_mid_write<G, LINES>(s, T, v);
        __syncthreads();
        fft16_tail<G, LINES, true>(s, T, [&](int, int, int q, float2 w) {
            if (act) dst[q * rs + ln] = w;
        });
    } else {
        cp_async_wait_all();
        __syncthreads();
        block_fft_io<G, true, false, true>(
            s, lines, tw, [&](int line, int p, bool) { return mul_mipow(__ldg(col + p * rs + line), p); }, NoIO{},
            [&](int line, int q, float2 v) { dst[q * rs + line] = v; });
    }
}

template <int G, int LINES> HQS_DEV void adj_rows_h_item(const HalfArgs& A, int iy, int ch, float2* s) {
    const int n = A.n, L = A.L, l0 = ch * A.LC, lines = min(A.LC, L - l0);
    const float2* src = A.work + (int64_t)iy * G * L + l0;
    const float2* sm = A.smaps + (int64_t)iy * n * L + l0;
    const float ay = A.apod[iy] * A.scale;
    float2* tw = s + (size_t)G * LINES;
    auto store = [&](int ix, float2 a) {
        if (A.nchunk == 1) {
            const int64_t e = (int64_t)iy * n + ix;
            float2 v = cscale(a, ay * A.apod[ix]);
            if (A.z) {
                const float2 zv = A.z[e];
                v.x = fmaf(A.zc, zv.x, v.x);
                v.y = fmaf(A.zc, zv.y, v.y);
            }
            A.xo[e] = v;
        } else {
            A.part[((int64_t)ch * n + iy) * n + ix] = a;
        }
    };
    half_twiddles<G>(tw, A.tw);
    if constexpr (fft16_ok<G>()) {
        constexpr int R = Fft16<G>::R, SUB = Fft16<G>::SUB;
        const Lane16 T(LINES);
        const bool act = T.line < lines;
        const int ln = act ? T.line : 0;
        float2 v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = __ldg(src + (int64_t)(T.t + 16 * m) * L + ln);
        cp_async_wait_all();
        __syncthreads();
        fft16_mid_inv<G>(T, tw, v);
        fft16_mid_write<G, LINES>(s, T, v);
        // the maps of the lane's outputs load while the CTA meets at the barrier
        float2 sv[4 * SUB];
#pragma unroll
        for (int k = 0; k < 4 * SUB; ++k) {
            const int ix = T.tp + 8 * (k >> 2) + R * (4 * T.par + (k & 3));
            sv[k] = __ldg(sm + (int64_t)ix * L + ln);
            if (!act) sv[k] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        fft16_tail_coilsum<G, LINES, true>(s, T, sv, store);
    } else {
        cp_async_wait_all();
        __syncthreads();
        block_fft_io<G, true, false, true>(
            s, lines, tw, [&](int line, int p, bool) { return mul_mipow(__ldg(src + (int64_t)p * L + line), p); }, NoIO{},
            NoIO{});
        for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
            float2 a = make_float2(0.f, 0.f);
            for (int l = 0; l < lines; ++l) a = cadd(a, cmulc(__ldg(sm + (int64_t)ix * L + l), s[ix * kLines + l]));
            store(ix, a);
        }
    }
}

// single slice: grid (rows or columns, chunks); batched: grid (rows or columns,
// largest chunk count, slices), the slice's arguments from a device table
#define HQS_HALF_KERNELS(NAME, CHUNKS)                                                                              \
    template <int G, int LINES>                                                                               \
    __global__ void __launch_bounds__(half_threads<G, LINES>(), 512 / half_threads<G, LINES>()) k_##NAME(HalfArgs A) { \
        HQS_PDL_ENTRY();                                                                                      \
        extern __shared__ __align__(16) float2 s[];                                                           \
        NAME##_item<G, LINES>(A, blockIdx.x, blockIdx.y, s);                                                  \
    }                                                                                                         \
    template <int G, int LINES>                                                                               \
    __global__ void __launch_bounds__(half_threads<G, LINES>(), 512 / half_threads<G, LINES>())               \
        k_##NAME##_b(const HalfArgs* __restrict__ tab, float zc) {                                            \
        HQS_PDL_ENTRY();                                                                                      \
        extern __shared__ __align__(16) float2 s[];                                                           \
        HalfArgs A = tab[blockIdx.z];                                                                         \
        A.zc = zc;                                                                                            \
        if ((int)blockIdx.y >= (CHUNKS ? A.nchunk : (A.L + LINES - 1) / LINES)) return;                          \
        NAME##_item<G, LINES>(A, blockIdx.x, blockIdx.y, s);                                                  \
    }
HQS_HALF_KERNELS(fwd_rows_h, false)
HQS_HALF_KERNELS(fwd_cols_h, false)
HQS_HALF_KERNELS(adj_cols_h, true)
HQS_HALF_KERNELS(adj_rows_h, true)
#undef HQS_HALF_KERNELS

// Type-2 interpolation: LPP lanes per sorted point, lane q owning VEC coils of a chunk
// (two as one 16-byte load where the coil count is even), the weights from the plan's
// table, the results straight to the caller's (coil, point) order (a sorted copy and a
// kernel to put it in order cost 8 us more).  Bound: latency of the L2 and L1 gathers of
// W^2 grid values of a point's coils, so the registers go to loads in flight (3 CTAs per
// SM with 85 registers: a 320^2 x 16-coil forward at W 6 55 us; with 128 registers 48).
template <int VEC> struct Coils;
template <> struct Coils<2> {
    float2 a, b;
    HQS_DEV void zero() { a = b = make_float2(0.f, 0.f); }
    HQS_DEV void fma_load(const float2* p, float w) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        a = cfma_r(make_float2(v.x, v.y), w, a);
        b = cfma_r(make_float2(v.z, v.w), w, b);
    }
    HQS_DEV void fma(const Coils& v, float w) {
        a = cfma_r(v.a, w, a);
        b = cfma_r(v.b, w, b);
    }
    HQS_DEV void put(float2* y, int64_t M) const {
        y[0] = a;
        y[M] = b;
    }
};
template <> struct Coils<1> {
    float2 a;
    HQS_DEV void zero() { a = make_float2(0.f, 0.f); }
    HQS_DEV void fma_load(const float2* p, float w) { a = cfma_r(__ldg(p), w, a); }
    HQS_DEV void fma(const Coils& v, float w) { a = cfma_r(v.a, w, a); }
    HQS_DEV void put(float2* y, int64_t) const { y[0] = a; }
};
template <int W, int VEC, int LPP>
__global__ void __launch_bounds__(256) k_interp(const float2* __restrict__ Gh, const int4* __restrict__ pts,
                                                const float* __restrict__ kbw, const int* __restrict__ perm, int M,
                                                int G, int L, float2* __restrict__ y) {
    HQS_PDL_ENTRY();
    const int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LPP;
    const int q = threadIdx.x % LPP;
    if (j >= M) return;
    const int4 pt = pts[j];
    const int dst = perm[j];
    float wx[8], wy[8];
    const float4* kw = reinterpret_cast<const float4*>(kbw + j * 24);
#pragma unroll
    for (int h = 0; h < (W + 3) / 4; ++h) {
        const float4 v = __ldg(kw + h);
        wx[4 * h] = v.x, wx[4 * h + 1] = v.y, wx[4 * h + 2] = v.z, wx[4 * h + 3] = v.w;
    }
#pragma unroll
    for (int h = 0; h < (W + 1) / 2; ++h) {
        const float4 v = __ldg(kw + 2 + h);
        wy[2 * h] = v.x, wy[2 * h + 1] = v.z;
    }
    int gxs[W];
#pragma unroll
    for (int b = 0; b < W; ++b) {
        const int gx = pt.x + b;
        gxs[b] = (gx >= G ? gx - G : gx) * L;
    }
    for (int l = q * VEC; l < L; l += LPP * VEC) {
        Coils<VEC> acc;
        acc.zero();
#pragma unroll
        for (int a = 0; a < W; ++a) {
            int gy = pt.y + a;
            if (gy >= G) gy -= G;
            const float2* row = Gh + (int64_t)gy * G * L + l;
            Coils<VEC> ra;
            ra.zero();
#pragma unroll
            for (int b = 0; b < W; ++b) ra.fma_load(row + gxs[b], wx[b]);
            acc.fma(ra, wy[a]);
        }
        acc.put(y + (int64_t)l * M + dst, M);
    }
}

// ---------------------------------------------------------------- adjoint
// Tile-owned type-1 spreading: each 8 x 8 tile of the grid is written once, with plain
// stores, by the warps that own it (no atomics on data, no memset, a fixed order of the
// sums).  The plan lists the points that touch each tile (2.7 tiles a point at W 6) with
// the offset of their first tap.  Lane (x, coil group) keeps the 8 rows of its cell
// column for CPL coils in registers, so a point costs its value times the lane's x
// weight once, then one packed multiply-add per exact y tap and coil, the rows selected
// by a switch on the point's y offset (registers need static names).  The weights and
// k-space values of 16 points at a time go to the warp's own shared memory with
// cp.async while the 16 before are added: a warp needs no barrier.
// A tile of at most HQS_SPREAD_LIGHT points belongs to one warp, eight such tiles to a
// CTA; a heavier one to whole CTAs of up to 8 HQS_SPREAD_LIGHT points each, whose warps'
// tiles are summed through shared memory, and, where there are several CTAs, through
// partial tiles in slot order by the last to arrive.
// Bound: latency of a point's shared-memory reads and switch, and of the list, weight and
// value reads per tile.  320^2 x 16 coils, 32,768 spiral points: a whole adjoint 85.5 ->
// 62.1 us (384^2 x 13 coils, 56,064 radial points: 145 -> 94.8) against CTAs that scanned
// the neighbouring bins' points; light tiles of up to 32, 64, 128, 256 points: 64.7, 62.1,
// 75.0, 103.5 us; without reading the next point ahead 66.1.
constexpr int kTile = 8;
constexpr int kSpreadBatch = 16;
template <int CPL> constexpr int spread_slot() { return 96 + 4 * CPL * (int)sizeof(float2); }
template <int CPL> constexpr size_t spread_smem() {
    // point slots of 8 warps, or their 8 tiles while a heavy tile is summed
    constexpr size_t a = (size_t)8 * 2 * kSpreadBatch * spread_slot<CPL>();
    constexpr size_t b = (size_t)8 * kTile * kTile * 4 * CPL * sizeof(float2);
    return a > b ? a : b;
}
template <int W, int CPL, int OY>
HQS_DEV void spread_rows(float2 (&acc)[kTile][CPL], const char* sp, const float2* u) {
    const float4* wy = reinterpret_cast<const float4*>(sp + 32);
#pragma unroll
    for (int b = 0; b < W; ++b) {
        if (OY + b < 0 || OY + b >= kTile) continue;
        const float4 w4 = wy[b >> 1];
        const float2 w = (b & 1) ? make_float2(w4.z, w4.w) : make_float2(w4.x, w4.y);
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[(OY + b) & (kTile - 1)][c] = cfma2(u[c], w, acc[(OY + b) & (kTile - 1)][c]);
    }
}
// CPL values of a lane to d: pairs as 16-byte stores, or the first n singly
template <int CPL> HQS_DEV void put_coils(float2* d, const float2* v, int n, bool pairs) {
    if (CPL >= 2 && pairs && n >= CPL) {
#pragma unroll
        for (int c = 0; c + 1 < CPL; c += 2)
            reinterpret_cast<float4*>(d)[c / 2] = make_float4(v[c].x, v[c].y, v[c + 1].x, v[c + 1].y);
    } else {
#pragma unroll
        for (int c = 0; c < CPL; ++c)
            if (c < n) d[c] = v[c];
    }
}
template <int W, int CPL>
__global__ void __launch_bounds__(256, 2)
    k_spread(const float2* __restrict__ y, const float* __restrict__ kbw, const int4* __restrict__ list,
             const int4* __restrict__ ctas, const int4* __restrict__ light, const int2* __restrict__ tinfo,
             unsigned* __restrict__ tickets, float2* __restrict__ partial, int64_t M, int nbx, int G, int L,
             float2* __restrict__ grid) {
    HQS_PDL_ENTRY();
    constexpr int T = kTile, CL = 4 * CPL, SLOT = spread_slot<CPL>(), NB = kSpreadBatch;
    static_assert(T == 8 && W <= 8 && NB == 16, "one point per half-warp of copies, eight steps a batch");
    extern __shared__ float4 smem4[];
    __shared__ int last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int xl = lane & 7, cq = lane >> 3;
    const int l0 = blockIdx.y * CL, lc = min(CL, L - l0);
    // (tile, first entry, end entry, partial slot or -1), or (-1, first light tile, end, -)
    const int4 it = ctas[blockIdx.x];
    const bool heavy = it.x >= 0;
    int tile = it.x, e0 = 0, e1 = 0;
    if (heavy) {   // this warp's eighth of the entries
        const int n = it.z - it.y;
        e0 = it.y + n * warp / 8;
        e1 = it.y + n * (warp + 1) / 8;
    } else if (it.y + warp < it.z) {
        const int4 t = light[it.y + warp];
        tile = t.x;
        e0 = t.y;
        e1 = t.z;
    }
    char* sw = reinterpret_cast<char*>(smem4) + (size_t)warp * 2 * NB * SLOT;
    float2 acc[T][CPL];
#pragma unroll
    for (int r = 0; r < T; ++r)
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[r][c] = make_float2(0.f, 0.f);
    auto entry = [&](int e) { return lane < NB && e + lane < e1 ? __ldg(list + e + lane) : make_int4(0, 0, 0, 0); };
    auto copy = [&](const int4& ent, int n, int buf) {
        const int q = lane & 15;
#pragma unroll
        for (int s = 0; s < NB / 2; ++s) {
            const int i = 2 * s + (lane >> 4);
            const int j = __shfl_sync(0xffffffffu, ent.x, i), m = __shfl_sync(0xffffffffu, ent.y, i);
            if (i >= n) continue;
            char* d = sw + (buf * NB + i) * SLOT;
            if (q < 6) cp_async16(d + 16 * q, kbw + (int64_t)j * 24 + 4 * q);
            if (q < lc) cp_async8(d + 96 + 8 * q, y + (int64_t)(l0 + q) * M + m);
        }
        cp_async_commit();
    };
    int4 cur = entry(e0), nxt = entry(e0 + NB);
    copy(cur, e1 - e0, 0);
    for (int e = e0, buf = 0; e < e1; e += NB, buf ^= 1) {
        const int4 nn = entry(e + 2 * NB);
        copy(nxt, e1 - e - NB, buf ^ 1);   // empty after the last batch
        cp_async_wait_group<1>();
        __syncwarp();
        const int n = min(NB, e1 - e);
        // the next point's offset, x weight and values are read while this one is added
        const int vl = 96 + cq * CPL * (int)sizeof(float2);
        const char* sp = sw + buf * NB * SLOT;
        int off = __shfl_sync(0xffffffffu, cur.z, 0);
        float wx;
        float2 v[CPL];
        auto fetch = [&](const char* p) {
            const int bx = xl - ((off & 255) - 16);
            const bool in = (unsigned)bx < (unsigned)W;
            wx = *reinterpret_cast<const float*>(p + (in ? 4 * bx : 0));
            wx = in ? wx : 0.f;
            if constexpr (CPL == 4) {
                const float4 v0 = *reinterpret_cast<const float4*>(p + vl), v1 = *reinterpret_cast<const float4*>(p + vl + 16);
                v[0] = make_float2(v0.x, v0.y), v[1] = make_float2(v0.z, v0.w);
                v[2] = make_float2(v1.x, v1.y), v[3] = make_float2(v1.z, v1.w);
            } else {
#pragma unroll
                for (int c = 0; c < CPL; ++c) v[c] = reinterpret_cast<const float2*>(p + vl)[c];
            }
        };
        fetch(sp);
        for (int i = 0; i < n; ++i, sp += SLOT) {
            const int oy = (off >> 8) - 16;
            float2 u[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) u[c] = cmul_r(v[c], wx);
            if (i + 1 < n) {
                off = __shfl_sync(0xffffffffu, cur.z, i + 1);
                fetch(sp + SLOT);
            }
            switch (oy) {
#define HQS_ROWS(OY)                                                 \
    case OY:                                                         \
        if constexpr (OY > -W) spread_rows<W, CPL, OY>(acc, sp, u);  \
        break;
                HQS_ROWS(-7) HQS_ROWS(-6) HQS_ROWS(-5) HQS_ROWS(-4) HQS_ROWS(-3)
                HQS_ROWS(-2) HQS_ROWS(-1) HQS_ROWS(0) HQS_ROWS(1) HQS_ROWS(2)
                HQS_ROWS(3) HQS_ROWS(4) HQS_ROWS(5) HQS_ROWS(6) HQS_ROWS(7)
#undef HQS_ROWS
            }
        }
        __syncwarp();
        cur = nxt;
        nxt = nn;
    }
    cp_async_wait_all();
    const int ncoil = lc - cq * CPL;   // coils of this lane that exist (may be <= 0)
    const bool pairs = L % 2 == 0;
    const int64_t grow = (int64_t)G * L;
    auto cell = [&](int r) {
        return grid + ((int64_t)((tile / nbx) * T + r) * G + (tile % nbx) * T + xl) * L + l0 + cq * CPL;
    };
    if (!heavy) {
        if (tile < 0) return;
        float2* g = cell(0);
#pragma unroll
        for (int r = 0; r < T; ++r) put_coils<CPL>(g + r * grow, acc[r], ncoil, pairs);
        return;
    }
    // the CTA's sum: every warp's tile to shared memory, then warp w adds row w in warp order
    __syncthreads();
    // (element c of a lane at [warp][row][c][lane], so a warp's accesses are contiguous)
    float2* st = reinterpret_cast<float2*>(smem4);
#pragma unroll
    for (int r = 0; r < T; ++r)
#pragma unroll
        for (int c = 0; c < CPL; ++c) st[((warp * T + r) * CPL + c) * 32 + lane] = acc[r][c];
    __syncthreads();
    float2 sum[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) sum[c] = make_float2(0.f, 0.f);
    for (int w = 0; w < 8; ++w)
#pragma unroll
        for (int c = 0; c < CPL; ++c) sum[c] = cadd(sum[c], st[((w * T + warp) * CPL + c) * 32 + lane]);
    if (it.w < 0) {
        put_coils<CPL>(cell(warp), sum, ncoil, pairs);
        return;
    }
    const int64_t slot = (int64_t)gridDim.y * T * T * CL;
    float2* pc = partial + ((int64_t)blockIdx.y * T * T + warp * T + xl) * CL + cq * CPL;
    put_coils<CPL>(pc + it.w * slot, sum, CPL, true);
    __threadfence();
    __syncthreads();
    const int2 ti = tinfo[tile];
    unsigned* ticket = tickets + (int64_t)tile * gridDim.y + blockIdx.y;
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == (unsigned)(ti.x - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int c = 0; c < CPL; ++c) sum[c] = make_float2(0.f, 0.f);
    for (int k = 0; k < ti.x; ++k)
#pragma unroll
        for (int c = 0; c < CPL; ++c) sum[c] = cadd(sum[c], __ldcg(pc + (ti.y + k) * slot + c));
    put_coils<CPL>(cell(warp), sum, ncoil, pairs);
    if (threadIdx.x == 0) *ticket = 0u;
}

// Column gx: IFFT along y of the spread grid, keep the image rows -> V[iy][gx][l].
template <int G>
__global__ void k_adj_cols(const float2* __restrict__ Hg, int n, int L, int LC, int nchunk,
                           const float2* __restrict__ twg, float2* __restrict__ V) {
    HQS_PDL_ENTRY();
    extern __shared__ float2 s[];
    const float2* tw = stage_twiddles<G>(s + G * kLines, twg);
    const int gx = blockIdx.x;
    const int l0 = blockIdx.y * LC;
    const int lines = min(LC, L - l0);
    const int pst = blockDim.x / lines;
    const int l = threadIdx.x % lines, p0 = threadIdx.x / lines;
    const int64_t rs = (int64_t)G * L;
    const float2* col = Hg + (int64_t)gx * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 8
        for (int p = p0; p < G; p += pst) s[p * kLines + l] = col[p * rs];
    }
    __syncthreads();
    block_fft<G, true>(s, lines, tw);
    float2* dst = V + (int64_t)gx * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 4
        for (int iy = p0; iy < n; iy += pst) dst[iy * rs] = s[pix_to_grid(iy, n, G) * kLines + l];
    }
}

// Row IFFT + crop + conj(S_l) sum over the coils of chunk blockIdx.y.  With
// one chunk the deapodised image is written directly; otherwise the chunk's
// partial sum goes to part[chunk] and k_adj_chunk_sum finishes.
template <int G>
__global__ void k_adj_rows(const float2* __restrict__ V, const float2* __restrict__ smaps,
                           const float* __restrict__ apod, int n, int L, int LC, int nchunk,
                           float scale, const float2* __restrict__ twg, float2* x,
                           float2* __restrict__ part, float zc, const float2* z) {
    HQS_PDL_ENTRY();
    extern __shared__ float2 s[];
    const float2* tw = stage_twiddles<G>(s + G * kLines, twg);
    const int iy = blockIdx.x;
    const int l0 = blockIdx.y * LC;
    const int lines = min(LC, L - l0);
    const int pst = blockDim.x / lines;
    const int l = threadIdx.x % lines, p0 = threadIdx.x / lines;
    const float2* src = V + (int64_t)iy * G * L + l0 + l;
    if (p0 < pst) {
#pragma unroll 8
        for (int p = p0; p < G; p += pst) s[p * kLines + l] = src[(int64_t)p * L];
    }
    __syncthreads();
    block_fft<G, true>(s, lines, tw);
    const float ay = apod[iy] * scale;
    for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
        const int p = pix_to_grid(ix, n, G);
        const float2* sm = smaps + ((int64_t)iy * n + ix) * L + l0;
        float2 a = make_float2(0.f, 0.f);
        for (int ll = 0; ll < lines; ++ll) {
            const float2 sv = sm[ll];
            const float2 g = s[p * kLines + ll];
            a.x += sv.x * g.x + sv.y * g.y;
            a.y += sv.x * g.y - sv.y * g.x;
        }
        if (nchunk == 1) {
            const int64_t e = (int64_t)iy * n + ix;
            float2 v = cscale(a, ay * apod[ix]);
            if (z) {
                const float2 zv = z[e];
                v.x = fmaf(zc, zv.x, v.x);
                v.y = fmaf(zc, zv.y, v.y);
            }
            x[e] = v;
        } else {
            part[((int64_t)blockIdx.y * n + iy) * n + ix] = a;
        }
    }
}

__global__ void k_adj_chunk_sum(const float2* __restrict__ part, const float* __restrict__ apod, int n,
                                int nchunk, float scale, float2* x, float zc, const float2* z) {
    HQS_PDL_ENTRY();
    const int count = n * n;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
        float2 a = make_float2(0.f, 0.f);
        for (int c = 0; c < nchunk; ++c) a = cadd(a, part[(int64_t)c * count + e]);
        const int iy = e / n, ix = e - iy * n;
        float2 v = cscale(a, apod[iy] * apod[ix] * scale);
        if (z) {
            const float2 zv = z[e];
            v.x = fmaf(zc, zv.x, v.x);
            v.y = fmaf(zc, zv.y, v.y);
        }
        x[e] = v;
    }
}

// ---------------------------------------------------------------- launchers
// the lower-half passes apply when G = 2n: at any coil count for the sizes of the
// two-stage transforms, for full 16-coil chunks below (a thread without a line would
// leave the radix-8 stages' hooks reading line 0)
inline bool half_passes(const hqs_plan_s* p) {
    return p->G == 2 * p->n && (p->G >= 128 || (p->LC == kLines && p->L % kLines == 0));
}
// lines per CTA of these passes: the smallest of 4, 8, 16 that holds the coil chunk
inline int half_lines(const hqs_plan_s* p) { return p->G >= 128 && p->LC <= 8 ? (p->LC <= 4 ? 4 : 8) : kLines; }
// lines per CTA of the passes whose lines do not meet
template <int G, int LINES> constexpr int half_free_lines() { return fft16_ok<G>() && LINES > 8 ? 8 : LINES; }
template <int G, class F> static int dispatch_half(int lines, F&& f) {
    if constexpr (fft16_ok<G>()) {
        if (lines == 4) return f.template operator()<4>();
        if (lines == 8) return f.template operator()<8>();
    }
    return f.template operator()<kLines>();
}

static HalfArgs half_args(const hqs_plan_s* p, const float2* x, float2* xo, float zc, const float2* z) {
    HalfArgs A;
    A.x = x;
    A.xo = xo;
    A.z = z;
    A.zc = zc;
    A.smaps = p->smaps;
    A.apod = p->apod;
    A.tw = p->G >= 128 ? plan_twiddles16(p, p->G) : plan_twiddles(p, p->G);
    A.work = p->work;
    A.grid = p->grid;
    A.part = p->chunk_buf;
    A.n = p->n;
    A.L = p->L;
    A.LC = p->LC;
    A.nchunk = p->nchunk;
    A.scale = p->scale;
    return A;
}

template <int G>
static int fwd_fft_impl(hqs_plan_s* p, const float2* x, cudaStream_t st) {
    const float2* tw = plan_twiddles(p, G);
    const int th = fft_threads<G>(p->LC);
    const size_t sm = nufft_smem_floats2<G>() * sizeof(float2);
    if constexpr (G % 2 == 0 && G != 16 && G != 320 && G != 384) {   // twice a supported image
        if (half_passes(p))
            return dispatch_half<G>(half_lines(p), [&]<int LN>() -> int {
                constexpr int LI = half_free_lines<G, LN>(), ht = half_threads<G, LI>();
                constexpr size_t hs = half_smem<G, LI>();
                const int nc = ceil_div(p->L, LI);
                HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_rows_h<G, LI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs));
                HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_cols_h<G, LI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs));
                const HalfArgs A = half_args(p, x, nullptr, 0.f, nullptr);
                HQS_CUDA_TRY(launch_pdl(k_fwd_rows_h<G, LI>, dim3(p->n, nc), ht, hs, st, A));
                HQS_CUDA_TRY(launch_pdl(k_fwd_cols_h<G, LI>, dim3(G, nc), ht, hs, st, A));
                HQS_CUDA_TRY(cudaGetLastError());
                return HQS_OK;
            });
    }
    HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_rows<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_cols<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HQS_CUDA_TRY(launch_pdl(k_fwd_rows<G>, dim3(p->n, p->nchunk), th, sm, st, x, p->smaps, p->apod, p->n, p->L, p->LC,
                            p->nchunk, p->scale, tw, p->work));
    HQS_CUDA_TRY(launch_pdl(k_fwd_cols<G>, dim3(G, p->nchunk), th, sm, st, p->work, p->n, p->L, p->LC, p->nchunk, tw,
                            p->grid));
    HQS_CUDA_TRY(cudaGetLastError());
    return HQS_OK;
}

template <int G>
static int adj_fft_impl(hqs_plan_s* p, float2* x, float zc, const float2* z, cudaStream_t st) {
    const float2* tw = plan_twiddles(p, G);
    const int th = fft_threads<G>(p->LC);
    const size_t sm = nufft_smem_floats2<G>() * sizeof(float2);
    if constexpr (G % 2 == 0 && G != 16 && G != 320 && G != 384) {
        if (half_passes(p)) {
            const int rc = dispatch_half<G>(half_lines(p), [&]<int LN>() -> int {
                constexpr int ht = half_threads<G, LN>();
                constexpr size_t hs = half_smem<G, LN>();
                HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_cols_h<G, LN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs));
                HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_rows_h<G, LN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs));
                const HalfArgs A = half_args(p, nullptr, x, zc, z);
                HQS_CUDA_TRY(launch_pdl(k_adj_cols_h<G, LN>, dim3(G, p->nchunk), ht, hs, st, A));
                HQS_CUDA_TRY(launch_pdl(k_adj_rows_h<G, LN>, dim3(p->n, p->nchunk), ht, hs, st, A));
                return HQS_OK;
            });
            if (rc != HQS_OK) return rc;
            return launch_adj_chunks(p, x, zc, z, st);
        }
    }
    HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_cols<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_rows<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HQS_CUDA_TRY(launch_pdl(k_adj_cols<G>, dim3(G, p->nchunk), th, sm, st, p->grid, p->n, p->L, p->LC, p->nchunk, tw,
                            p->work));
    HQS_CUDA_TRY(launch_pdl(k_adj_rows<G>, dim3(p->n, p->nchunk), th, sm, st, p->work, p->smaps, p->apod, p->n, p->L,
                            p->LC, p->nchunk, p->scale, tw, x, p->chunk_buf, zc, z));
    if (p->nchunk > 1)
        HQS_CUDA_TRY(launch_pdl(k_adj_chunk_sum, dim3(std::min(ceil_div(p->n * p->n, 256), 1024)), dim3(256), 0, st,
                                p->chunk_buf, p->apod, p->n, p->nchunk, p->scale, x, zc, z));
    HQS_CUDA_TRY(cudaGetLastError());
    return HQS_OK;
}

template <int W>
static int interp_impl(hqs_plan_s* p, float2* y, cudaStream_t st) {
    if (p->M == 0) return HQS_OK;
    auto go = [&]<int VEC, int LPP>() -> int {
        HQS_CUDA_TRY(launch_pdl(k_interp<W, VEC, LPP>, dim3((unsigned)ceil_div64(p->M * LPP, 256)), dim3(256), 0, st,
                                p->grid, p->pts, p->spread.kbw, p->perm, (int)p->M, p->G, p->L, y));
        HQS_CUDA_TRY(cudaGetLastError());
        return HQS_OK;
    };
    // lanes per point: as many as the coils fill (pairs of coils need an even count)
    if (p->L % 2 == 0) return p->L > 4 ? go.template operator()<2, 8>() : go.template operator()<2, 2>();
    return p->L > 4 ? go.template operator()<1, 16>() : go.template operator()<1, 4>();
}

// Kaiser-Bessel weights of the sorted points, 24 floats each: x taps [8], y taps as
// pairs [8][2] (the operand of packed multiply-adds); zero beyond W.
__global__ void k_point_weights(const int4* __restrict__ pts, int M, int W, float beta, float* __restrict__ kbw) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)M * 16) return;
    const int j = (int)(e >> 4), h = (int)(e & 15), b = h & 7;
    const int4 pt = pts[j];
    const float t = __int_as_float(h < 8 ? pt.z : pt.w) - (float)b;
    const float w = b < W ? kb_phi(t, (float)W, beta) : 0.f;
    float* o = kbw + (int64_t)j * 24;
    if (h < 8) o[b] = w;
    else o[8 + 2 * b] = o[9 + 2 * b] = w;
}

int launch_point_weights(const hqs_plan_s* p, const int4* pts, float* kbw, cudaStream_t st) {
    if (p->M == 0) return HQS_OK;
    k_point_weights<<<(unsigned)ceil_div64(p->M * 16, 256), 256, 0, st>>>(pts, (int)p->M, p->W, (float)p->beta, kbw);
    HQS_CUDA_TRY(cudaGetLastError());
    return HQS_OK;
}

// The tiles (up to two per axis) that a point's footprint touches: f(tile, offsets).
template <class F> HQS_DEV void touched_tiles(int4 p, int W, int G, F&& f) {
    constexpr int T = kTile;
    const int i0[2] = {p.x, p.y};
    int t[2][2], o[2][2], n[2];
    for (int a = 0; a < 2; ++a) {
        int e = i0[a] + W - 1;
        e -= e >= G ? G : 0;
        t[a][0] = i0[a] / T;
        o[a][0] = i0[a] - t[a][0] * T;
        t[a][1] = e / T;
        const int d = i0[a] - t[a][1] * T;
        o[a][1] = d > 0 ? d - G : d;   // taps that wrap start before cell 0
        n[a] = t[a][1] != t[a][0] ? 2 : 1;
    }
    for (int b = 0; b < n[1]; ++b)
        for (int a = 0; a < n[0]; ++a) f(t[1][b] * (G / T) + t[0][a], (o[0][a] + 16) | ((o[1][b] + 16) << 8));
}
__global__ void k_tile_count(const int4* __restrict__ pts, int M, int W, int G, int* __restrict__ counts) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < M) touched_tiles(pts[j], W, G, [&](int t, int) { atomicAdd(&counts[t], 1); });
}
__global__ void k_tile_fill(const int4* __restrict__ pts, const int* __restrict__ perm, int M, int W, int G,
                            int* __restrict__ cursor, int4* __restrict__ list) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < M)
        touched_tiles(pts[j], W, G,
                      [&](int t, int off) { list[atomicAdd(&cursor[t], 1)] = make_int4(j, perm[j], off, 0); });
}

int launch_tile_count(const hqs_plan_s* p, int* counts, cudaStream_t st) {
    if (p->M > 0) k_tile_count<<<(unsigned)ceil_div64(p->M, 256), 256, 0, st>>>(p->pts, (int)p->M, p->W, p->G, counts);
    HQS_CUDA_TRY(cudaGetLastError());
    return HQS_OK;
}
int launch_tile_fill(const hqs_plan_s* p, const int4* pts, const int* perm, int* cursor, int4* list, cudaStream_t st) {
    if (p->M > 0)
        k_tile_fill<<<(unsigned)ceil_div64(p->M, 256), 256, 0, st>>>(pts, perm, (int)p->M, p->W, p->G, cursor, list);
    HQS_CUDA_TRY(cudaGetLastError());
    return HQS_OK;
}

template <int W>
static int spread_impl(hqs_plan_s* p, const float2* y, cudaStream_t st) {
    const int cpl = spread_cpl(p->L), nch = ceil_div(p->L, 4 * cpl);
    const hqs_plan_s::Spread& S = p->spread;
    auto go = [&]<int CPL>() -> int {
        constexpr size_t sm = spread_smem<CPL>();
        HQS_CUDA_TRY(cudaFuncSetAttribute(k_spread<W, CPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        HQS_CUDA_TRY(launch_pdl(k_spread<W, CPL>, dim3(S.nctas, nch), dim3(256), sm, st, y, S.kbw, S.list, S.ctas, S.light,
                                S.tile_info, S.tickets, S.partial, p->M, p->G / kTile, p->G, p->L, p->grid));
        HQS_CUDA_TRY(cudaGetLastError());
        return HQS_OK;
    };
    return cpl == 1 ? go.template operator()<1>() : (cpl == 2 ? go.template operator()<2>() : go.template operator()<4>());
}

template <class F> static int dispatch_w(int W, F&& f) {
    switch (W) {
        case 2: return f.template operator()<2>();
        case 3: return f.template operator()<3>();
        case 4: return f.template operator()<4>();
        case 5: return f.template operator()<5>();
        case 6: return f.template operator()<6>();
        case 7: return f.template operator()<7>();
        case 8: return f.template operator()<8>();
        default: return HQS_ERR_INVALID_ARG;
    }
}

int launch_fwd(hqs_plan_s* p, const float2* x, float2* y, cudaStream_t st) {
    int rc = dispatch_fft_size(p->G, [&]<int GG>() { return fwd_fft_impl<GG>(p, x, st); });
    if (rc != HQS_OK) return rc;
    return dispatch_w(p->W, [&]<int WW>() { return interp_impl<WW>(p, y, st); });
}

int launch_adj_axpy(hqs_plan_s* p, const float2* y, float zc, const float2* z, float2* x, cudaStream_t st) {
    // every grid cell is written by the tile-owned spreading: no memset
    int rc = dispatch_w(p->W, [&]<int WW>() { return spread_impl<WW>(p, y, st); });
    if (rc != HQS_OK) return rc;
    return dispatch_fft_size(p->G, [&]<int GG>() { return adj_fft_impl<GG>(p, x, zc, z, st); });
}

// ---- the passes of several plans in one launch per pass (batched operators)
bool plan_half_passes(const hqs_plan_s* p) { return half_passes(p); }
int plan_half_lines(const hqs_plan_s* p) { return half_lines(p); }
size_t half_args_bytes() { return sizeof(HalfArgs); }
void fill_half_args(const hqs_plan_s* p, const float2* x, float2* xo, const float2* z, void* dst) {
    const HalfArgs A = half_args(p, x, xo, 0.f, z);
    std::memcpy(dst, &A, sizeof(HalfArgs));
}

// `count` plans with grid G = 2n and `lines` lines per CTA whose arguments are the
// consecutive HalfArgs at d_tab: the forward's row and column passes (adjoint 0)
// or the adjoint's column and row passes (adjoint 1), grid (lines, chunks, plans);
// maxchunk, maxcoils: the largest chunk and coil count among them
int launch_half_group(int G, int n, int lines, int maxchunk, int maxcoils, int count, const void* d_tab, int adjoint, float zc,
                      cudaStream_t st) {
    return dispatch_fft_size(G, [&]<int GG>() -> int {
        if constexpr (GG == 16 || GG == 320 || GG == 384) {
            return HQS_ERR_UNSUPPORTED;
        } else {
            return dispatch_half<GG>(lines, [&]<int LN>() -> int {
                const HalfArgs* tab = static_cast<const HalfArgs*>(d_tab);
                if (adjoint) {
                    constexpr int th = half_threads<GG, LN>();
                    constexpr size_t sm = half_smem<GG, LN>();
                    HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_cols_h_b<GG, LN>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
                    HQS_CUDA_TRY(cudaFuncSetAttribute(k_adj_rows_h_b<GG, LN>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
                    HQS_CUDA_TRY(launch_pdl(k_adj_cols_h_b<GG, LN>, dim3(GG, maxchunk, count), th, sm, st, tab, zc));
                    HQS_CUDA_TRY(launch_pdl(k_adj_rows_h_b<GG, LN>, dim3(n, maxchunk, count), th, sm, st, tab, zc));
                } else {
                    constexpr int LI = half_free_lines<GG, LN>(), th = half_threads<GG, LI>();
                    constexpr size_t sm = half_smem<GG, LI>();
                    const int nc = ceil_div(maxcoils, LI);
                    HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_rows_h_b<GG, LI>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
                    HQS_CUDA_TRY(cudaFuncSetAttribute(k_fwd_cols_h_b<GG, LI>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
                    HQS_CUDA_TRY(launch_pdl(k_fwd_rows_h_b<GG, LI>, dim3(n, nc, count), th, sm, st, tab, zc));
                    HQS_CUDA_TRY(launch_pdl(k_fwd_cols_h_b<GG, LI>, dim3(GG, nc, count), th, sm, st, tab, zc));
                }
                HQS_CUDA_TRY(cudaGetLastError());
                return HQS_OK;
            });
        }
    });
}

// the parts of the operators outside the lower-half passes, per plan
int launch_spread(hqs_plan_s* p, const float2* y, cudaStream_t st) {
    return dispatch_w(p->W, [&]<int WW>() { return spread_impl<WW>(p, y, st); });
}
int launch_interp(hqs_plan_s* p, float2* y, cudaStream_t st) {
    return dispatch_w(p->W, [&]<int WW>() { return interp_impl<WW>(p, y, st); });
}
int launch_adj_chunks(hqs_plan_s* p, float2* x, float zc, const float2* z, cudaStream_t st) {
    if (p->nchunk <= 1) return HQS_OK;
    HQS_CUDA_TRY(launch_pdl(k_adj_chunk_sum, dim3(std::min(ceil_div(p->n * p->n, 256), 1024)), dim3(256), 0, st,
                            p->chunk_buf, p->apod, p->n, p->nchunk, p->scale, x, zc, z));
    return HQS_OK;
}

int launch_adj(hqs_plan_s* p, const float2* y, float2* x, cudaStream_t st) {
    return launch_adj_axpy(p, y, 0.f, nullptr, x, st);
}

extern "C" int hqs_forward(hqs_plan p, const hqs_c64* x, hqs_c64* y, void* stream) {
    if (!p || !x || (!y && p->M > 0)) return HQS_ERR_INVALID_ARG;
    return launch_fwd(p, reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y),
                      (cudaStream_t)stream);
}

extern "C" int hqs_adjoint(hqs_plan p, const hqs_c64* y, hqs_c64* x, void* stream) {
    if (!p || !x || (!y && p->M > 0)) return HQS_ERR_INVALID_ARG;
    return launch_adj(p, reinterpret_cast<const float2*>(y), reinterpret_cast<float2*>(x),
                      (cudaStream_t)stream);
}

extern "C" int hqs_adjoint_axpy(hqs_plan p, const hqs_c64* y, float c, const hqs_c64* z, hqs_c64* x,
                                void* stream) {
    if (!p || !x || !z || (!y && p->M > 0)) return HQS_ERR_INVALID_ARG;
    return launch_adj_axpy(p, reinterpret_cast<const float2*>(y), c, reinterpret_cast<const float2*>(z),
                           reinterpret_cast<float2*>(x), (cudaStream_t)stream);
}
