// pair_rule.cuh -- the written rule of the unique pair list (library-internal),
// shared by the solve's pair-list kernel and the allocation-free entry point so
// that both lists agree bit for bit.
//
// For i <= j (Sec. III A, Step II; Eq. l2g): s = h^-1 C (row sums left to
// right, no FMA); ds = s_j - s_i - round(ds); the lattice image k in
// {-1,0,1}^3 with the smallest |h(ds+k)|^2 (first in lexicographic k on ties),
// kept when that is <= R_pair^2.  Grid-resolved centre
// g = NINT(N (s_i + (ds + k)/2)) mod N, NINT rounding half away from zero
// (round()).  Every product and sum is an explicit round-to-nearest intrinsic,
// so nothing is contracted and the operation order is the one the oracle uses.
// The list of 1024 orbitals (count, scan, fill) on one GB300: 789 us with the rule on every pair, 98 us screened.
#pragma once

namespace exx {

__device__ __forceinline__ double pair_dot3_rn(const double *r, double a, double b, double c)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(r[0], a), __dmul_rn(r[1], b)), __dmul_rn(r[2], c));
}

// Fractional coordinates s = h^-1 C of one orbital.
// Cell: any structure with double h[3][3], hinv[3][3], r_pair2, int n[3] and
// const double *centres ([n_orb][3] Cartesian, device memory).
template <class Cell>
__device__ __forceinline__ void pair_frac(const Cell &C, int i, double *s)
{
    const double *c = C.centres + 3 * i;
    for (int al = 0; al < 3; ++al) s[al] = pair_dot3_rn(C.hinv[al], c[0], c[1], c[2]);
}

// FP32 screen of the rule.  FP64 runs at 1/64 of the FP32 rate and the 27 images of a
// pair take 800 FP64 operations, while about one pair in twenty is near: the
// distances are formed in FP32 first, and the rule itself runs only for pairs that
// the screen cannot rule out, over the images that it cannot rule out.
struct PairScreen {
    float h[3][3];
    float H;   // largest sum of |h| over a row: a component's error per unit of coordinate error
    float r;   // R_pair
    template <class Cell>
    __device__ explicit PairScreen(const Cell &C)
    {
        H = 0.f;
        for (int a = 0; a < 3; ++a) {
            float t = 0.f;
            for (int b = 0; b < 3; ++b) {
                h[a][b] = (float)C.h[a][b];
                t += fabsf(h[a][b]);
            }
            H = fmaxf(H, t);
        }
        r = sqrtf((float)C.r_pair2) * (1.f + 0x1p-20f);
    }
    // error of a Cartesian component of h (ds + k) in FP32: es, that of ds, and the roundings of the
    // sums (|ds + k| < 2; 16 half-ulps cover them)
    __device__ float delta(float es) const { return 1.01f * H * (es + 0x1p-19f); }
    // squared distances of the 27 images; f(index, squared distance)
    template <class F>
    __device__ __forceinline__ void images(const float *ds, F f) const
    {
#pragma unroll
        for (int k0 = -1; k0 <= 1; ++k0) {
            const float t0 = ds[0] + (float)k0;
            const float a0 = h[0][0] * t0, a1 = h[1][0] * t0, a2 = h[2][0] * t0;
#pragma unroll
            for (int k1 = -1; k1 <= 1; ++k1) {
                const float t1 = ds[1] + (float)k1;
                const float b0 = a0 + h[0][1] * t1, b1 = a1 + h[1][1] * t1, b2 = a2 + h[2][1] * t1;
#pragma unroll
                for (int k2 = -1; k2 <= 1; ++k2) {
                    const float t2 = ds[2] + (float)k2;
                    const float x = b0 + h[0][2] * t2, y = b1 + h[1][2] * t2, z = b2 + h[2][2] * t2;
                    f((k0 + 1) * 9 + (k1 + 1) * 3 + k2 + 1, x * x + y * y + z * z);
                }
            }
        }
    }
    // false only when the rule cannot accept the pair: si, sj rounded to FP32 (a coordinate
    // difference next to +-1/2, whose image base may differ in FP64, passes)
    __device__ __forceinline__ bool near(const float *si, const float *sj) const
    {
        float ds[3], es = 0.f;
        bool pass = false;
        for (int al = 0; al < 3; ++al) {
            const float d = sj[al] - si[al];
            const float e = 0x1p-22f * (fabsf(si[al]) + fabsf(sj[al]) + 1.f);
            ds[al] = d - rintf(d);
            es = fmaxf(es, e);
            pass |= !(fabsf(ds[al]) < 0.5f - e);
        }
        float m = __int_as_float(0x7f800000);
        images(ds, [&](int, float d2) { m = fminf(m, d2); });
        const float lim = (r + 2.f * delta(es)) * (1.f + 0x1p-20f);
        return pass || !(m > lim * lim);   // a NaN passes
    }
    // images that may be the nearest one, from the FP64 ds of the rule
    __device__ __forceinline__ unsigned mask(const double *d) const
    {
        const float ds[3] = {(float)d[0], (float)d[1], (float)d[2]};
        float m = __int_as_float(0x7f800000);
        images(ds, [&](int, float d2) { m = fminf(m, d2); });
        const float lim = (sqrtf(m) + 4.f * delta(0x1p-22f)) * (1.f + 0x1p-20f), lim2 = lim * lim;
        unsigned w = 0;
        images(ds, [&](int k, float d2) { w |= d2 > lim2 ? 0u : 1u << k; });
        return w;
    }
};

// The rule.
template <class Cell>
__device__ __forceinline__ bool pair_rule(const Cell &C, const PairScreen &scr, int i, int j, int *kb, int *g)
{
    double si[3], ds[3];
    pair_frac(C, i, si);
    pair_frac(C, j, ds);
    for (int al = 0; al < 3; ++al) {
        const double d = __dadd_rn(ds[al], -si[al]);
        ds[al] = __dadd_rn(d, -round(d));
    }
    double best = 1.0 / 0.0;
    kb[0] = kb[1] = kb[2] = 0;
    for (unsigned w = scr.mask(ds); w; w &= w - 1) {   // ascending: the lexicographic order of k
        const int im = __ffs(w) - 1, k0 = im / 9 - 1, k1 = im / 3 % 3 - 1, k2 = im % 3 - 1;
        const double t0 = __dadd_rn(ds[0], (double)k0), t1 = __dadd_rn(ds[1], (double)k1),
                     t2 = __dadd_rn(ds[2], (double)k2);
        const double d0 = pair_dot3_rn(C.h[0], t0, t1, t2);
        const double d1 = pair_dot3_rn(C.h[1], t0, t1, t2);
        const double d2 = pair_dot3_rn(C.h[2], t0, t1, t2);
        const double dd = __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
        if (dd < best) {
            best = dd;
            kb[0] = k0;
            kb[1] = k1;
            kb[2] = k2;
        }
    }
    if (!(best <= C.r_pair2)) return false;
    for (int al = 0; al < 3; ++al) {
        const double sm = __dadd_rn(si[al], __dmul_rn(__dadd_rn(ds[al], (double)kb[al]), 0.5));
        const long long gg = (long long)round(__dmul_rn((double)C.n[al], sm));
        long long r = gg % C.n[al];
        if (r < 0) r += C.n[al];
        g[al] = (int)r;
    }
    return true;
}

// Rows i0 .. i0 + kPairRows - 1 of the list by one CTA of kPairThreads: screens every
// j >= i of each row in FP32, collects the survivors in shared memory and runs the
// rule on them with full warps.  emit(row, position, j, k, g) receives the pairs of a row in
// ascending j, position counting from 0; returns the rows' pair counts in cnt (every thread).
constexpr int kPairRows = 4, kPairThreads = 256, kPairList = 1024;
template <class Cell, class Emit>
__device__ void pair_rows_block(const Cell &C, int n_orb, int i0, int *cnt, Emit emit)
{
    __shared__ int s_list[kPairRows][kPairList];
    __shared__ int s_warp[kPairRows][kPairThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const PairScreen scr(C);
    float si[kPairRows][3];
#pragma unroll
    for (int r = 0; r < kPairRows; ++r) {
        double s[3] = {0.0, 0.0, 0.0};
        if (i0 + r < n_orb) pair_frac(C, i0 + r, s);
        for (int al = 0; al < 3; ++al) si[r][al] = (float)s[al];
        cnt[r] = 0;
    }
    int len[kPairRows] = {};
    // sum over the CTA's warps of a per-warp count, and the part of the warps before this one
    auto scan = [&](int r, int mine, int &before, int &total) {
        if (lane == 0) s_warp[r][w] = mine;
        __syncthreads();
        before = total = 0;
        for (int k = 0; k < kPairThreads / 32; ++k) {
            if (k < w) before += s_warp[r][k];
            total += s_warp[r][k];
        }
    };
    auto flush = [&](int r) {   // the rule on the row's survivors, in order
        __syncthreads();
        for (int p0 = 0; p0 < len[r]; p0 += kPairThreads) {
            int kb[3], g[3];
            const int j = p0 + tid < len[r] ? s_list[r][p0 + tid] : -1;
            const bool ok = j >= 0 && pair_rule(C, scr, i0 + r, j, kb, g);
            const unsigned bal = __ballot_sync(0xffffffffu, ok);
            int before, total;
            scan(r, __popc(bal), before, total);
            if (ok) emit(r, cnt[r] + before + __popc(bal & ((1u << lane) - 1u)), j, kb, g);
            cnt[r] += total;
            __syncthreads();
        }
        len[r] = 0;
    };
    for (int j0 = i0; j0 < n_orb; j0 += kPairThreads) {
        const int j = j0 + tid;
        float sj[3] = {0.f, 0.f, 0.f};
        if (j < n_orb) {
            double s[3];
            pair_frac(C, j, s);
            for (int al = 0; al < 3; ++al) sj[al] = (float)s[al];
        }
        unsigned bal[kPairRows];
#pragma unroll
        for (int r = 0; r < kPairRows; ++r) {
            bal[r] = __ballot_sync(0xffffffffu, j < n_orb && j >= i0 + r && i0 + r < n_orb && scr.near(si[r], sj));
            if (lane == 0) s_warp[r][w] = __popc(bal[r]);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kPairRows; ++r) {
            int before = len[r], total = 0;
            for (int k = 0; k < kPairThreads / 32; ++k) {
                if (k < w) before += s_warp[r][k];
                total += s_warp[r][k];
            }
            if (bal[r] >> lane & 1u) s_list[r][before + __popc(bal[r] & ((1u << lane) - 1u))] = j;
            len[r] += total;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kPairRows; ++r)
            if (len[r] > kPairList - kPairThreads) flush(r);
    }
#pragma unroll
    for (int r = 0; r < kPairRows; ++r) flush(r);
}

}  // namespace exx
