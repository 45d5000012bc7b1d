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
// The list of 1024 orbitals (count, scan, fill) on one GB300, one pair in twenty near: 822 us with the rule on every
// pair, 60 us screened; of 4 orbitals 37.6 -> 20.3, of 128 that are all near 41.6 -> 23.1, of 1024 that are 832 -> 222.
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
    float r;   // R_pair
    float H;   // largest sum of |h| over a row: a component's error per unit of coordinate error
    // by the lanes of one warp, for the CTA (conversions from FP64 are slow): h and r
    template <class Cell>
    __device__ void fill(const Cell &C, int lane)
    {
        if (lane < 9) h[lane / 3][lane % 3] = (float)C.h[lane / 3][lane % 3];
        if (lane == 9) r = sqrtf((float)C.r_pair2) * (1.f + 0x1p-20f);
    }
    __device__ void set_norm()
    {
        H = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) H = fmaxf(H, fabsf(h[a][0]) + fabsf(h[a][1]) + fabsf(h[a][2]));
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

// The rule.  si: the fractional coordinates of i; g is formed with GRID only.
template <bool GRID, class Cell>
__device__ __forceinline__ bool pair_rule(const Cell &C, const PairScreen &scr, const double *si, int j, int *kb, int *g)
{
    double ds[3];
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
    if constexpr (GRID) {
        for (int al = 0; al < 3; ++al) {
            const double sm = __dadd_rn(si[al], __dmul_rn(__dadd_rn(ds[al], (double)kb[al]), 0.5));
            const long long gg = (long long)round(__dmul_rn((double)C.n[al], sm));
            long long r = gg % C.n[al];
            if (r < 0) r += C.n[al];
            g[al] = (int)r;
        }
    }
    return true;
}

// Rows i0 .. i0 + R - 1 of the list by one CTA of kPairThreads: screens every j >= i of each
// row in FP32, collects the survivors in shared memory (a list per row) and runs the rule on the
// lists of all rows together, a warp on 32 survivors of one row, so that no warp of the CTA
// waits while another row's survivors are ruled.  What every thread needs in FP64 of the
// rows and the cell is formed once per CTA.  emit(r, position, j, k, g) receives the pairs of row
// i0 + r in ascending j, position counting from 0 (FILL only); cnt: the rows' pair counts (every thread).
constexpr int kPairThreads = 256, kPairWarps = kPairThreads / 32, kPairList = 1024;
template <int R, bool FILL, class Cell, class Emit>
__device__ __forceinline__ void pair_rows_block(const Cell &C, int n_orb, int i0, int (&cnt)[R], Emit emit)
{
    __shared__ PairScreen s_scr;
    __shared__ double s_si[R][3];
    __shared__ float s_sif[R][3];
    __shared__ int s_list[R][kPairList];
    __shared__ int s_warp[2][R][kPairWarps];   // two buffers: one barrier per step
    __shared__ int s_run[2][kPairWarps];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    if (w == 0 && lane < 3 * R) {
        const int r = lane / 3, al = lane - 3 * r;
        double s = 0.0;
        if (i0 + r < n_orb) {
            const double *c = C.centres + 3 * (i0 + r);
            s = pair_dot3_rn(C.hinv[al], c[0], c[1], c[2]);
        }
        s_si[r][al] = s;
        s_sif[r][al] = (float)s;
    }
    if (w == 1) s_scr.fill(C, lane);
    __syncthreads();
    PairScreen scr = s_scr;
    scr.set_norm();
    int len[R];
#pragma unroll
    for (int r = 0; r < R; ++r) cnt[r] = len[r] = 0;
    auto pick = [](const int (&v)[R], int r) {   // v[r] from registers
        int x = 0;
#pragma unroll
        for (int k = 0; k < R; ++k) x = k == r ? v[k] : x;
        return x;
    };
    auto flush = [&]() {   // the rule on the survivors of every row, in order
        __syncthreads();
        int nw = 0;   // warps' worth of survivors
#pragma unroll
        for (int r = 0; r < R; ++r) nw += (len[r] + 31) >> 5;
        for (int q0 = 0, buf = 0; q0 < nw; q0 += kPairWarps, buf ^= 1) {
            int r = 0, b = q0 + w;   // this warp's row, and its place in the row's list
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const int n = (len[k] + 31) >> 5;
                if (r == k && b >= n) {
                    b -= n;
                    ++r;
                }
            }
            const int p = (b << 5) + lane;
            int kb[3], g[3], j = -1;
            bool ok = false;
            if (r < R && p < pick(len, r)) {
                j = s_list[r][p];
                ok = pair_rule<FILL>(C, scr, s_si[r], j, kb, g);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, ok);
            if (lane == 0) s_run[buf][w] = r << 8 | __popc(bal);
            __syncthreads();
            if constexpr (FILL) {
                int pos = r < R ? pick(cnt, r) + __popc(bal & below) : 0;
#pragma unroll
                for (int k = 0; k < kPairWarps; ++k)
                    if (k < w && s_run[buf][k] >> 8 == r) pos += s_run[buf][k] & 255;
                if (ok) emit(r, pos, j, kb, g);
            }
#pragma unroll
            for (int k = 0; k < kPairWarps; ++k) {
                const int rk = s_run[buf][k] >> 8, n = s_run[buf][k] & 255;
#pragma unroll
                for (int x = 0; x < R; ++x) cnt[x] += rk == x ? n : 0;
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) len[r] = 0;
        __syncthreads();
    };
    for (int j0 = i0, buf = 0; j0 < n_orb; j0 += kPairThreads, buf ^= 1) {
        const int j = j0 + tid;
        unsigned bal[R];
#pragma unroll
        for (int r = 0; r < R; ++r) bal[r] = 0;
        if (j0 + 32 * w < n_orb) {   // (the whole warp; FP64 below)
            float sj[3] = {0.f, 0.f, 0.f};
            if (j < n_orb) {
                double s[3];
                pair_frac(C, j, s);
                for (int al = 0; al < 3; ++al) sj[al] = (float)s[al];
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                bal[r] = __ballot_sync(0xffffffffu, j < n_orb && j >= i0 + r && i0 + r < n_orb && scr.near(s_sif[r], sj));
        }
        if (lane == 0)
#pragma unroll
            for (int r = 0; r < R; ++r) s_warp[buf][r][w] = __popc(bal[r]);
        __syncthreads();
        bool full = false;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            int before = len[r], total = 0;
#pragma unroll
            for (int k = 0; k < kPairWarps; ++k) {
                if (k < w) before += s_warp[buf][r][k];
                total += s_warp[buf][r][k];
            }
            if (bal[r] >> lane & 1u) s_list[r][before + __popc(bal[r] & below)] = j;
            len[r] += total;
            full |= len[r] > kPairList - kPairThreads;
        }
        if (full) flush();
    }
    flush();
}

// Rows per CTA (R) for a list of n rows: the rows of a CTA share the FP64 coordinates of the columns,
// which bound the screen, but their survivors share its warps and the grid shrinks.  Measured, one
// GB300, the whole list of n orbitals in us with R = 1 / 2 / 4, one pair in twenty near, and all:
//    n =  256   23.6 /  23.2 /  27.2    36.0 /  43.6 /  68.4
//    n =  512   39.5 /  31.3 /  35.4    83.1 /  86.5 / 125
//    n = 1024   76.4 /  60.3 /  59.9     208 /   222 /  292
//    n = 1500    132 /  98.8 /  90.7     410 /   410 /  507
//    n = 2048    221 /   154 /   132     734 /   698 /  754
//    n = 4096    762 /   505 /   384    2830 /  2620 /  2550
// Two rows once they leave each of the 152 SMs a CTA, four once that leaves two.
inline int pair_rows_per_cta(int n) { return n < 2 * 152 ? 1 : n < 8 * 152 ? 2 : 4; }

}  // namespace exx
