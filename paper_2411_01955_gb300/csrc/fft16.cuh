// Two-stage transforms of 2n-point lines (N = 2n = 16 R) whose input half is zero or
// whose output half is not wanted: the transforms of the Toeplitz passes and of the
// NUFFT's lower-half passes at 128 points and more (fft16_ok; shorter lines keep the
// radix-8 stages of fft.cuh).
//
//   X[kk + 16 m] = sum_{i < R} w_R^(i m) w_N^(i kk) sum_{r < 8} w_16^(r kk) x[i + R r],   kk < 16, m < R
//
// Head (per i): a radix-16 DFT of 8 inputs, split over a pair of lanes: the lane of
// parity par computes the 8 outputs kk = 2k + par.  Mid (per kk): the twiddles
// w_N^(i kk) and one radix-R DFT held in one thread's registers, whose outputs leave
// for global memory, or, for a forward x factor x inverse pair, are multiplied and
// transformed back in place.  The inverse runs the same two steps backwards (tail).
// One shared-memory round trip per transform and two per pair, against two and four
// of the three-stage radix-8 transforms, and one barrier for each; 16 threads per line
// at every size, so a CTA holds the same 16 lines whatever N is.
//
// Thread layout: tid = t * LINES + line, t < 16 (LINES = 16 or 8), so the lanes of a
// pair (t = 2 tp + par) are LINES apart in one warp.  Element (i, kk) of a line lies at
// s[(i * 16 + kk) * LINES + line]: a half-warp always touches 128 contiguous bytes.
// The 8 inputs of a pair are loaded half by each lane and exchanged by shuffles, which
// halves the global loads; the tail sums the two parities the same way, and each lane
// keeps 4 of the pair's 8 outputs.
//
// Bound: shared-memory wavefronts and FP32 issue.  A^H A at 320^2 x 16 coils (5,120 row
// pairs, 10,240 column pairs of 640 points): 68.5 -> 50.8 us with these transforms in
// place of the 8 x 8 x 10 stages (GB300, CUDA events over back-to-back applies).
#pragma once

#include "fft.cuh"

namespace hqs {

// Radix 32 = 4 x 8 with twiddles: n = n1 + 4 n2, k = k1 + 8 k2,
// X[k1 + 8 k2] = sum_n1 w4^(n1 k2) w32^(n1 k1) sum_n2 w8^(n2 k1) x[n1 + 4 n2].
template <bool INV> struct Dft<32, INV> {
    HQS_DEV static void run(float2* v) {
        constexpr float c[8] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                                0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                                0.19509032201612826785f};
        float2 y[4][8];
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < 8; ++n2) y[n1][n2] = v[n1 + 4 * n2];
            Dft<8, INV>::run(y[n1]);
#pragma unroll
            for (int k1 = 1; k1 < 8; ++k1) {
                if (n1 == 0) continue;
                // angle 2 pi n1 k1 / 32, n1 k1 <= 21: (cos, sin) from the first octant's table
                const int q = n1 * k1;
                const float cq = q <= 8 ? (q == 8 ? 0.f : c[q]) : (q <= 16 ? (q == 16 ? -1.f : -c[16 - q]) : -c[q - 16]);
                const float sq = q <= 8 ? (q == 8 ? 1.f : c[8 - q]) : (q <= 16 ? (q == 16 ? 0.f : c[q - 8]) : -c[24 - q]);
                y[n1][k1] = cmul(y[n1][k1], make_float2(cq, INV ? sq : -sq));
            }
        }
#pragma unroll
        for (int k1 = 0; k1 < 8; ++k1) {
            float2 t[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
            Dft<4, INV>::run(t);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 8 * k2] = t[k2];
        }
    }
};
template <bool INV> struct Dft<48, INV> : DftPfa<16, 3, INV> {};

// Sizes these transforms cover (R = 8, 16, 32, 40, 48); smaller lines leave lane
// pairs idle in the head and keep the radix-8 stages of fft.cuh.
template <int N> constexpr bool fft16_ok() { return N == 128 || N == 256 || N == 512 || N == 640 || N == 768; }
template <int N> struct Fft16 {
    static constexpr int R = N / 16;
    static constexpr int SUB = R / 8;   // (input or output) columns i per lane pair
};

struct Lane16 {
    int line, t, tp, par;
    HQS_DEV Lane16(int lines_) {
        int tid;
        asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));   // see block_fft
        line = tid % lines_;
        t = tid / lines_;
        tp = t >> 1;
        par = t & 1;
    }
};

// (cos, sin) of pi m / 8, m = 0..9
HQS_DEV float2 w16(int m) {
    constexpr float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f;
    switch (m) {
        case 0: return make_float2(1.f, 0.f);
        case 1: return make_float2(c1, s1);
        case 2: return make_float2(kSqrtHalf, kSqrtHalf);
        case 3: return make_float2(s1, c1);
        case 4: return make_float2(0.f, 1.f);
        case 5: return make_float2(-s1, c1);
        case 6: return make_float2(-kSqrtHalf, kSqrtHalf);
        case 7: return make_float2(-c1, s1);
        case 8: return make_float2(-1.f, 0.f);
        default: return make_float2(-c1, -s1);
    }
}
HQS_DEV float2 sel(bool p, float2 a, float2 b) { return make_float2(p ? a.x : b.x, p ? a.y : b.y); }
template <int LINES> HQS_DEV float2 swap_pair(float2 v) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, LINES), __shfl_xor_sync(0xffffffffu, v.y, LINES));
}

// Forward head: ld(pos) reads the line's element pos < N/2 (the upper half is zero).
// Every thread of the CTA calls it (the loads of threads without a line read the
// caller's clamped line); no barrier inside.  ROT: output k times i^k (the image's
// centring, i^(kk + 16 m) = i^kk, folded into the lane factors).
// fft16_head_load and fft16_head_do are its two halves, for callers that load ahead.
template <int N, class LD> HQS_DEV void fft16_head_load(float2 (&o)[Fft16<N>::SUB][4], const Lane16& T, LD&& ld) {
    constexpr int R = Fft16<N>::R, SUB = Fft16<N>::SUB;
#pragma unroll
    for (int b = 0; b < SUB; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q) o[b][q] = ld(T.tp + 8 * b + R * (4 * T.par + q));
}
template <int N, int LINES, bool ROT = false>
HQS_DEV void fft16_head_do(float2* s, const Lane16& T, const float2 (&o)[Fft16<N>::SUB][4]) {
    constexpr int SUB = Fft16<N>::SUB;
    const bool odd = T.par != 0;
    // lane factors of the sums and differences: w16^(par q) and (-1)^par w16^((2 + par) q)
    float2 ca[4], cb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 a = sel(odd, w16(q), make_float2(1.f, 0.f));
        const float2 b = sel(odd, make_float2(-w16(3 * q).x, -w16(3 * q).y), w16(2 * q));
        ca[q] = make_float2(a.x, -a.y);
        cb[q] = make_float2(b.x, -b.y);
        if (ROT) {   // kk = 4 m + par for the sums, 4 m + 2 + par for the differences
            ca[q] = sel(odd, make_float2(-ca[q].y, ca[q].x), ca[q]);
            cb[q] = sel(odd, make_float2(cb[q].y, -cb[q].x), make_float2(-cb[q].x, -cb[q].y));
        }
    }
#pragma unroll
    for (int b = 0; b < SUB; ++b) {
        float2 e[4], f[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 p = swap_pair<LINES>(o[b][q]);
            // even lane: own x[q], other x[q + 4]; odd lane: own x[q + 4] times -i, other x[q]
            const float2 w = sel(odd, make_float2(o[b][q].y, -o[b][q].x), o[b][q]);
            e[q] = cadd(w, p);
            f[q] = csub(w, p);
            if (q > 0 || ROT) {
                e[q] = cmul(e[q], ca[q]);
                f[q] = cmul(f[q], cb[q]);
            } else {
                f[q] = cscale(f[q], cb[0].x);
            }
        }
        Dft<4, false>::run(e);
        Dft<4, false>::run(f);
        float2* dst = s + ((T.tp + 8 * b) * 16 + T.par) * LINES + T.line;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            dst[(4 * m) * LINES] = e[m];
            dst[(4 * m + 2) * LINES] = f[m];
        }
    }
}

template <int N, int LINES, bool ROT = false, class LD> HQS_DEV void fft16_head(float2* s, const Lane16& T, LD&& ld) {
    float2 o[Fft16<N>::SUB][4];
    fft16_head_load<N>(o, T, ld);
    fft16_head_do<N, LINES, ROT>(s, T, o);
}

// Inverse tail: the lane's 4 outputs of each of its SUB columns go to put(b, q, pos, v),
// pos = tp + 8 b + R (4 par + q) < N/2.  ROT: the transformed line was (-i)^k times the
// one given.
template <int N, int LINES, bool ROT = false, class PUT> HQS_DEV void fft16_tail(const float2* s, const Lane16& T, PUT&& put) {
    constexpr int R = Fft16<N>::R, SUB = Fft16<N>::SUB;
    const bool odd = T.par != 0;
    float2 ca[4], cb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ca[q] = sel(odd, w16(q), make_float2(1.f, 0.f));
        cb[q] = sel(odd, w16(3 * q), w16(2 * q));
        if (ROT) {
            ca[q] = sel(odd, make_float2(ca[q].y, -ca[q].x), ca[q]);
            cb[q] = sel(odd, make_float2(-cb[q].y, cb[q].x), make_float2(-cb[q].x, -cb[q].y));
        }
    }
#pragma unroll
    for (int b = 0; b < SUB; ++b) {
        const float2* src = s + ((T.tp + 8 * b) * 16 + T.par) * LINES + T.line;
        float2 e[4], f[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            e[m] = src[(4 * m) * LINES];
            f[m] = src[(4 * m + 2) * LINES];
        }
        Dft<4, true>::run(e);
        Dft<4, true>::run(f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q > 0 || ROT) {
                e[q] = cmul(e[q], ca[q]);
                f[q] = cmul(f[q], cb[q]);
            }
            const float2 S = cadd(e[q], f[q]), D0 = csub(e[q], f[q]);
            const float2 D = sel(odd, make_float2(-D0.y, D0.x), D0);
            const float2 g = swap_pair<LINES>(sel(odd, S, D));
            put(b, q, T.tp + 8 * b + R * (4 * T.par + q), cadd(sel(odd, D, S), g));
        }
    }
}

// Mid steps of a thread's kk = t: reads or writes the line's R values (i, kk).
template <int N, int LINES> HQS_DEV void fft16_mid_read(const float2* s, const Lane16& T, float2* v) {
    const float2* p = s + T.t * LINES + T.line;
#pragma unroll
    for (int i = 0; i < Fft16<N>::R; ++i) v[i] = p[i * 16 * LINES];
}
template <int N, int LINES> HQS_DEV void fft16_mid_write(float2* s, const Lane16& T, const float2* v) {
    float2* p = s + T.t * LINES + T.line;
#pragma unroll
    for (int i = 0; i < Fft16<N>::R; ++i) p[i * 16 * LINES] = v[i];
}
// twiddle table [R][16] in shared memory: w_N^(i kk) at i * 16 + kk (plan_twiddles16).
// The inverse reads it again with volatile loads: kept from a pair's forward step the
// table would take 2 R registers.
template <int N> HQS_DEV void fft16_mid_fwd(const Lane16& T, const float2* tw, float2* v) {
#pragma unroll
    for (int i = 1; i < Fft16<N>::R; ++i) v[i] = cmul(v[i], tw[i * 16 + T.t]);
    Dft<Fft16<N>::R, false>::run(v);
}
template <int N> HQS_DEV void fft16_mid_inv(const Lane16& T, const float2* tw, float2* v) {
    Dft<Fft16<N>::R, true>::run(v);
    const unsigned base = (unsigned)__cvta_generic_to_shared(tw + T.t);
#pragma unroll
    for (int i = 1; i < Fft16<N>::R; ++i) {
        float2 w;
        asm volatile("ld.volatile.shared.v2.f32 {%0, %1}, [%2];" : "=f"(w.x), "=f"(w.y) : "r"(base + i * 128));
        v[i] = cmulc(w, v[i]);
    }
}

// Sums over the LINES lanes of a line group (low lane bits) of CNT values per lane at
// once, halving the values a lane carries at each exchange while there are several:
// 15 exchanges for 16 values over 16 lanes against 64 for one butterfly per value; the
// order of the sum is fixed.  Afterwards lane j holds in w[0 .. PER) the totals of the
// values j PER + k (PER = CNT / LINES >= 1), or in w[0] that of value j >> SH, shared by
// 2^SH lanes (CNT < LINES).
template <int CNT, int LINES> HQS_DEV void lanes_sum(float2* w, int lane) {
    int c = CNT;
#pragma unroll
    for (int bit = LINES / 2; bit > 0; bit >>= 1) {
        if (c > 1) {
            c >>= 1;
            const bool up = (lane & bit) != 0;
#pragma unroll
            for (int k = 0; k < CNT / 2; ++k) {
                if (k >= c) continue;
                const float2 give = sel(up, w[k], w[k + c]), keep = sel(up, w[k + c], w[k]);
                w[k] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, give.x, bit),
                                   keep.y + __shfl_xor_sync(0xffffffffu, give.y, bit));
            }
        } else {
            w[0] = make_float2(w[0].x + __shfl_xor_sync(0xffffffffu, w[0].x, bit),
                               w[0].y + __shfl_xor_sync(0xffffffffu, w[0].y, bit));
        }
    }
}
template <int CNT, int LINES, class F> HQS_DEV void lanes_sum_each(float2* w, int lane, F&& f) {
    lanes_sum<CNT, LINES>(w, lane);
    if constexpr (CNT >= LINES) {
        constexpr int PER = CNT / LINES;
#pragma unroll
        for (int k = 0; k < PER; ++k) f(lane * PER + k, w[k]);
    } else {
        constexpr int REP = LINES / CNT;
        if ((lane & (REP - 1)) == 0) f(lane / REP, w[0]);
    }
}

// Inverse tail of a row of coils (line = coil) with the weighted coil sum fused:
// put(ix, sum_l conj(S_l[ix]) v_l[ix]) once for each pixel ix < n of the row.  sv: the
// lane's maps at its 4 SUB outputs (index 4 b + q), zero for lanes without a coil.
// COILS < LINES: the lines are rows of COILS coils each, summed row by row.
template <int N, int LINES, bool ROT = false, int COILS = LINES, class PUT>
HQS_DEV void fft16_tail_coilsum(const float2* s, const Lane16& T, const float2* sv, PUT&& put) {
    constexpr int R = Fft16<N>::R, CNT = 4 * Fft16<N>::SUB;
    constexpr int C1 = CNT >= 16 ? 16 : CNT, C2 = CNT - C1;   // 16 + 4 at 640, 16 + 8 at 768
    float2 w[CNT];
    fft16_tail<N, LINES, ROT>(s, T, [&](int b, int q, int, float2 v) { w[4 * b + q] = cmulc(sv[4 * b + q], v); });
    auto out = [&](int j, float2 v) { put(T.tp + 8 * (j >> 2) + R * (4 * T.par + (j & 3)), v); };
    const int lane = T.line % COILS;
    lanes_sum_each<C1, COILS>(w, lane, out);
    if constexpr (C2 > 0) lanes_sum_each<C2, COILS>(w + C1, lane, [&](int j, float2 v) { out(C1 + j, v); });
}

}  // namespace hqs
