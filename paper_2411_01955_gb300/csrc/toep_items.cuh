// Device bodies of the three A^H A passes, shared by the per-stage kernels
// and the persistent solver.
#pragma once

#include "fft16.cuh"
#include "solve.cuh"

namespace hqs {

// ------------------------------------------------------------ A^H A passes
// Each CTA handles one row/column for the coils of chunk `ch` (<= 16 coils);
// the FFT body must not sit inside a runtime loop (register allocation
// collapses), so coil chunks are a grid dimension.

// Shared memory of the A^H A passes: [N2][LINES] lines | [n] image row |
// [N2] twiddles.  LINES: lines an item holds; the radix-8 transforms of the small
// sizes always use kLines.
template <int N2, int LINES = kLines> constexpr size_t toep_smem_floats2(int n) { return (size_t)N2 * LINES + n + N2; }
// threads of a CTA that runs these items
template <int N2, int LINES = kLines> constexpr int toep_threads() {
    return fft16_ok<N2>() ? 16 * LINES : FftSize<N2>::TPL * kLines;
}

// Twiddles of the item in shared memory: given (already staged), or copied now with
// cp.async, complete after the item's cp_async_wait_all and barrier.
template <int N2> HQS_DEV const float2* toep_twiddles(float2* dst, const ToepArgs& A, const float2* tws) {
    if (tws) return tws;
    for (int c = threadIdx.x; c < N2 / 2; c += blockDim.x) cp_async16(dst + 2 * c, A.tw + 2 * c);
    return dst;
}

// P1: v = src (or p = src + beta p when fused, single chunk only), S_l v,
// zero-pad to N2, FFT along x.
// src_row, when given, is the row already in shared memory (the persistent
// solver rebuilds z there); otherwise the row is read from src.  tws, when given,
// holds the 2n-point twiddles already staged in shared memory.  Vectors
// written by other CTAs earlier in the same launch are read with ld.global.cg
// (L2), never from a possibly stale L1 line.
template <int N2, int LINES = kLines>
HQS_DEV void toep_rows_fwd_item(const ToepArgs& A, int iy, int ch, const float2* __restrict__ src,
                                float2* __restrict__ pvec, float beta, bool fuse, float2* s,
                                const float2* src_row = nullptr, const float2* tws = nullptr) {
    const int n = A.n, L = A.L;
    float2* rowv = s + N2 * LINES;
    const float2* tw = toep_twiddles<N2>(rowv + n, A, tws);
    for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
        const int64_t e = (int64_t)iy * n + ix;
        float2 v = src_row ? src_row[ix] : __ldcg(src + e);
        if (fuse) {
            if (beta != 0.f) {
                const float2 pv = __ldcg(pvec + e);
                v.x = fmaf(beta, pv.x, v.x);
                v.y = fmaf(beta, pv.y, v.y);
            }
            pvec[e] = v;
        }
        rowv[ix] = v;
    }
    const int l0 = ch * A.LC;
    const int lines = min(A.LC, L - l0);
    const float2* sm = A.smaps + (int64_t)iy * n * L + l0;
    float2* dst = A.T + (int64_t)iy * N2 * L + l0;
    cp_async_wait_all();
    __syncthreads();
    if constexpr (fft16_ok<N2>()) {
        const Lane16 T(LINES);
        const bool act = T.line < lines;
        const float2* sml = sm + (act ? T.line : 0);
        fft16_head<N2, LINES>(s, T, [&](int p) { return cmul(__ldg(sml + (int64_t)p * L), rowv[p]); });
        __syncthreads();
        float2 v[Fft16<N2>::R];
        fft16_mid_read<N2, LINES>(s, T, v);
        fft16_mid_fwd<N2>(T, tw, v);
        if (act) {
            float2* d = dst + (int64_t)T.t * L + T.line;
#pragma unroll
            for (int m = 0; m < Fft16<N2>::R; ++m) __stcg(d + (int64_t)(16 * m) * L, v[m]);
        }
    } else {
        // S_l v straight into the first radix stage (upper half is the zero
        // padding), last stage straight to T
        block_fft_io<N2, false, true, false>(
            s, lines, tw, [&](int line, int p, bool) { return cmul(sm[(int64_t)p * L + line], rowv[p]); }, NoIO{},
            [&](int line, int p, float2 v) { dst[(int64_t)p * L + line] = v; });
    }
    __syncthreads();
}

// P2 of `nl` lines at col (element p of line f at col[f + p rs]): zero-pad, FFT along
// y, * kf(line, p), IFFT, keep the first n rows.  khs is the image-row region.
template <int N2, int LINES, class KF>
HQS_DEV void toep_cols_body(const ToepArgs& A, float2* col, int nl, float2* s, const float2* tw, KF&& kf) {
    const int64_t rs = (int64_t)N2 * A.L;
    if constexpr (fft16_ok<N2>()) {
        constexpr int R = Fft16<N2>::R;
        const Lane16 T(LINES);
        const bool act = T.line < nl;
        float2* c = col + (act ? T.line : 0);
        fft16_head<N2, LINES>(s, T, [&](int p) { return __ldcg(c + p * rs); });
        cp_async_wait_all();
        __syncthreads();
        // a thread reads and rewrites its own (i, kk) column: no barrier in between
        float2 v[R];
        fft16_mid_read<N2, LINES>(s, T, v);
        fft16_mid_fwd<N2>(T, tw, v);
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = cscale(v[m], kf(act ? T.line : 0, T.t + 16 * m));
        fft16_mid_inv<N2>(T, tw, v);
        fft16_mid_write<N2, LINES>(s, T, v);
        __syncthreads();
        // addresses afresh (a volatile copy of the stride): kept from the head's loads they
        // would hold 4 R / 5 registers through the transforms
        const Lane16 T2(LINES);
        int64_t rs2 = rs;
        asm volatile("" : "+l"(rs2));
        float2* c2 = col + T2.line;
        fft16_tail<N2, LINES>(s, T2, [&](int, int, int p, float2 w) {
            if (T2.line < nl) __stcg(c2 + p * rs2, w);
        });
    } else {
        cp_async_wait_all();
        __syncthreads();
        // column straight into the first stage (zero-padded upper half), * Khat between
        // the last forward and the first inverse stage (on registers), IFFT, first n rows
        // straight back to T
        block_fft_pair<N2, true, true>(
            s, nl, tw, [&](int line, int p, bool) { return __ldcg(col + line + p * rs); },
            [&](int line, int p, float2 v) { return cscale(v, kf(line, p)); },
            [&](int line, int p, float2 v) { col[line + p * rs] = v; });
    }
    __syncthreads();
}

// P2: column kx: zero-pad, FFT along y, * Khat, IFFT, keep the first n rows.
template <int N2, int LINES = kLines>
HQS_DEV void toep_cols_item(const ToepArgs& A, int kx, int ch, float2* s, const float2* tws = nullptr) {
    const int n = A.n, L = A.L;
    const float2* tw = toep_twiddles<N2>(s + N2 * LINES + n, A, tws);
    const int l0 = ch * A.LC;
    const int lines = min(A.LC, L - l0);
    const float* kh = A.khat + (int64_t)kx * N2;   // Khat stored transposed: column kx contiguous
    // the column of Khat (N2 floats) goes to the image-row region asynchronously while
    // the forward head runs
    float* khs = reinterpret_cast<float*>(s + N2 * LINES);
    for (int c = threadIdx.x; c < N2 / 4; c += blockDim.x) cp_async16(khs + 4 * c, kh + 4 * c);
    toep_cols_body<N2, LINES>(A, A.T + (int64_t)kx * L + l0, lines, s, tw, [&](int, int p) { return khs[p]; });
}

// P2 over nl consecutive (column, coil) lines of the flattened index f = kx L + l
// (f0 .. f0 + nl - 1, nl <= kLines): the data of line f at position p is
// T[f + p N2 L], so an item's lines are contiguous whichever columns they belong
// to, and chunks of fewer than kLines coils need not leave threads idle.  Khat of
// the item's first column is staged with cp.async; a line of a later column reads
// its Khat through L1.
template <int N2, int LINES = kLines>
HQS_DEV void toep_cols_flat_item(const ToepArgs& A, int f0, int nl, float2* s, const float2* tws = nullptr) {
    const int n = A.n, L = A.L;
    const float2* tw = toep_twiddles<N2>(s + N2 * LINES + n, A, tws);
    const int kx0 = f0 / L;
    const float* kh0 = A.khat + (int64_t)kx0 * N2;
    const float* khat = A.khat;
    float* khs = reinterpret_cast<float*>(s + N2 * LINES);
    for (int c = threadIdx.x; c < N2 / 4; c += blockDim.x) cp_async16(khs + 4 * c, kh0 + 4 * c);
    toep_cols_body<N2, LINES>(A, A.T + f0, nl, s, tw, [&](int line, int p) {
        const int kx = (f0 + line) / L;
        return kx == kx0 ? khs[p] : __ldg(khat + (int64_t)kx * N2 + p);
    });
}

// CG epilogue on one pixel: mode 0 returns v = A^H A p; mode 1 returns
// q = a v + b p and adds Re<p, q> to part.
HQS_DEV float2 toep_epilogue_pv(float2 v, float2 pv, float a, float b, double& part) {
    v = make_float2(fmaf(a, v.x, b * pv.x), fmaf(a, v.y, b * pv.y));
    part += (double)pv.x * v.x + (double)pv.y * v.y;
    return v;
}
HQS_DEV float2 toep_epilogue(float2 v, int64_t e, const float2* __restrict__ pvec, float a, float b,
                             int mode, double& part) {
    if (mode == 1) v = toep_epilogue_pv(v, __ldcg(pvec + e), a, b, part);
    return v;
}

// P3: row iy: IFFT along x, keep n, sum_l conj(S_l) . over the chunk's coils.
// One chunk: epilogue and store here (returns the thread's partial); several
// chunks: the raw chunk sum goes to A.chunk[ch] for k_toep_chunk_epilogue.
template <int N2, int LINES = kLines>
HQS_DEV double toep_rows_adj_item(const ToepArgs& A, int iy, int ch, float2* __restrict__ out,
                                  const float2* __restrict__ pvec, float a, float b, int mode,
                                  float2* s, const float2* tws = nullptr) {
    const int n = A.n, L = A.L;
    const float2* tw = toep_twiddles<N2>(s + N2 * LINES + n, A, tws);
    const int l0 = ch * A.LC;
    const int lines = min(A.LC, L - l0);
    const float2* src = A.T + (int64_t)iy * N2 * L + l0;
    const float2* sm = A.smaps + (int64_t)iy * n * L + l0;
    double part = 0.0;
    auto store = [&](int ix, float2 acc) {
        const int64_t e = (int64_t)iy * n + ix;
        if (A.nchunk == 1)
            out[e] = toep_epilogue(acc, e, pvec, a, b, mode, part);
        else
            A.chunk[(int64_t)ch * n * n + e] = acc;
    };
    if constexpr (fft16_ok<N2>()) {
        constexpr int R = Fft16<N2>::R, SUB = Fft16<N2>::SUB;
        const Lane16 T(LINES);
        const bool act = T.line < lines;
        const int ln = act ? T.line : 0;
        float2 v[R];
        {
            const float2* g = src + (int64_t)T.t * L + ln;
#pragma unroll
            for (int m = 0; m < R; ++m) v[m] = __ldcg(g + (int64_t)(16 * m) * L);
        }
        cp_async_wait_all();
        __syncthreads();   // twiddles staged; the previous item's reads of s are done
        fft16_mid_inv<N2>(T, tw, v);
        fft16_mid_write<N2, LINES>(s, T, v);
        // the maps of the lane's outputs load while the CTA meets at the barrier
        float2 sv[4 * SUB];
#pragma unroll
        for (int k = 0; k < 4 * SUB; ++k) {
            const int ix = T.tp + 8 * (k >> 2) + R * (4 * T.par + (k & 3));
            sv[k] = __ldg(sm + (int64_t)ix * L + ln);
            if (!act) sv[k] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        fft16_tail_coilsum<N2, LINES>(s, T, sv, store);
    } else {
        cp_async_wait_all();
        __syncthreads();
        // row straight from T into the first stage; only the first n columns are kept
        block_fft_io<N2, true, false, true>(
            s, lines, tw, [&](int line, int p, bool) { return __ldcg(src + (int64_t)p * L + line); }, NoIO{}, NoIO{});
        for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
            float2 acc = make_float2(0.f, 0.f);
            const float2* smx = sm + (int64_t)ix * L;
            for (int ll = 0; ll < lines; ++ll) {
                const float2 w = smx[ll];
                const float2 g = s[ix * kLines + ll];
                acc.x += w.x * g.x + w.y * g.y;
                acc.y += w.x * g.y - w.y * g.x;
            }
            store(ix, acc);
        }
    }
    __syncthreads();
    return part;
}

HQS_DEV double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += red[w];
    __syncthreads();
    return t;
}


}  // namespace hqs
