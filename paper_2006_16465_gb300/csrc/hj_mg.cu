// hj_mg.cu -- hierarchical Jacobi as the smoother of a geometric multigrid
// V-cycle (the use the paper's conclusion names; the V-cycle is the textbook
// one of the multigrid tutorial it cites).
//
// Levels: level 0 is the caller's 2D grid; level l + 1 halves the interior
// ((n - 1) / 2 points per axis, coarse point (I, J) on fine point (2I, 2J)),
// and its operator rediscretises the stencil on the doubled spacing (every
// h^-2 coefficient divided by 4, sigma_const kept).
//
// Kernels (one launch each, all captured in one CUDA graph per handle):
//   * mg_smooth_kernel: one weighted hierarchical cycle, a thread per point of
//     up to four rows, the subdomain plus halo in two shared-memory
//     containers, k damped Jacobi subiterations u' = u + omega (jac - u)
//     with the halo frozen (binary32 subdomains 32 wide and a multiple of four
//     high: mg_smooth_rows_kernel, four rows a warp in registers);
//   * mg_restrict_kernel (binary32), mg_restrict_tile_kernel (binary64): the fine
//     residual f - A u at the nine fine points around each coarse point,
//     full-weighted into the coarse right-hand side (fused, no residual array),
//     and the coarse correction set to zero;
//   * mg_prolong_kernel: u + bilinear interpolation of the coarse correction,
//     one thread per coarse cell writing the 2 x 2 fine points from its first
//     coarse point on.
// The graph also holds the residual norm of the level-0 iterate and its copy
// to pinned host memory, so a V-cycle costs one graph launch and one wait.
//
// Binary64 evaluates every sum in the oracle's order with separately rounded
// operations (no fused multiply-add), so the GPU V-cycle equals the oracle's
// bit for bit; binary32 uses fused chains.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "hj_runtime.cuh"

namespace hj {

namespace {

struct MgXferArgs {
    const void *f;       // fine right-hand side (restriction)
    const void *u;       // fine iterate (restriction: input; prolongation: u_in)
    void *uout;          // prolongation output (may equal u)
    void *fc;            // coarse right-hand side (restriction output)
    void *ec;            // coarse correction (restriction: zeroed; prolongation: input)
    long long ld, ldc;
    int nx, ny, ncx, ncy;
    double d, cW, cE, cS, cN;
};

// What a smoothing launch stages besides its level's iterate and RHS:
//   MG_PLAIN:    u and f of the level;
//   MG_RESTRICT: (binary32) the level's first smoothing after the restriction: the RHS is
//                the full-weighted fine residual (x: the finer level), formed
//                here and also stored as the level's f, and the iterate (the
//                coarse correction) starts at zero;
//   MG_PROLONG:  the level's first smoothing after the coarse solve: the
//                iterate is u + the bilinear interpolation of the coarse
//                correction (x: this level as the fine one), formed here for
//                the subdomain and its halo.
enum MgStage { MG_PLAIN = 0, MG_RESTRICT = 1, MG_PROLONG = 2 };

struct MgSmoothArgs {
    const void *f;
    const void *uin;
    void *uout;
    long long ld;
    int nx, ny, k, stage;   // stage: MgStage (the kernel instance is chosen by it)
    double cW, cE, cS, cN, invd, omega;
    float fW, fE, fS, fN, finvd, fomega;   // binary32: -c/d, 1/d, omega
    MgXferArgs x;                          // MG_RESTRICT / MG_PROLONG
};

template <typename T>
__device__ __forceinline__ T ld_g(const T *p) {
    return __ldg(p);
}

// whether two values differ in any bit
__device__ __forceinline__ bool bits_differ(double x, double y) {
    return __double_as_longlong(x) != __double_as_longlong(y);
}
__device__ __forceinline__ bool bits_differ(float x, float y) { return __float_as_uint(x) != __float_as_uint(y); }

// x * 2^-n (n = 1, 2, ..), correctly rounded, by an integer subtraction in the
// exponent field where x and the result are normal, else by the multiplication.
template <int N>
__device__ __forceinline__ double scale_down(double x) {
    const int hi = __double2hiint(x);
    const unsigned e = (unsigned)hi & 0x7ff00000u;
    if (e - ((unsigned)(N + 1) << 20) < (0x7fe00000u - ((unsigned)N << 20)))
        return __hiloint2double(hi - (N << 20), __double2loint(x));
    return __dmul_rn(x, 1.0 / (1 << N));
}

// x * c, correctly rounded, on the integer pipes where they cover it (mul_const)
__device__ __forceinline__ double mul_rn(double x, const MulConst &m, double c) {
    unsigned bad = 0;
    double r = mul_const(x, m, bad);
    if (bad > m.span) r = __dmul_rn(x, c);
    return r;
}

// Binary32: f - A u at fine index q as a fused chain
__device__ __forceinline__ float mg_resid(const MgXferArgs &x, const float *u, const float *f, long long q) {
    float r = fmaf(-(float)x.d, u[q], f[q]);
    r = fmaf(-(float)x.cW, u[q - 1], r);
    r = fmaf(-(float)x.cE, u[q + 1], r);
    r = fmaf(-(float)x.cS, u[q - x.ld], r);
    r = fmaf(-(float)x.cN, u[q + x.ld], r);
    return r;
}

// Binary32: the full-weighted fine residual at coarse point (I, J), the restriction
// (binary64: mg_restrict_tile_kernel).
__device__ __forceinline__ float restrict_at(const MgXferArgs &x, int I, int J) {
    const float *u = (const float *)x.u, *f = (const float *)x.f;
    const long long q = 2LL * J * x.ld + 2LL * I, ld = x.ld;
    const float r00 = mg_resid(x, u, f, q);
    const float s1 = (mg_resid(x, u, f, q - 1) + mg_resid(x, u, f, q + 1)) +
                     (mg_resid(x, u, f, q - ld) + mg_resid(x, u, f, q + ld));
    const float s2 = (mg_resid(x, u, f, q - ld - 1) + mg_resid(x, u, f, q - ld + 1)) +
                     (mg_resid(x, u, f, q + ld - 1) + mg_resid(x, u, f, q + ld + 1));
    return (4.0f * r00 + 2.0f * s1 + s2) * 0.0625f;
}

// Bilinear interpolation of the coarse correction: a fine point between four
// coarse points (both indices odd), between two (one odd), or on one.
template <typename T, bool EXACT>
__device__ __forceinline__ T avg2(T x, T y) {
    if constexpr (EXACT) return scale_down<1>(__dadd_rn(x, y));
    else return (x + y) * (T)0.5;
}

template <typename T, bool EXACT>
__device__ __forceinline__ T avg4(T e00, T e10, T e01, T e11) {
    if constexpr (EXACT) {
        double t = __dadd_rn(e00, e10);
        t = __dadd_rn(t, e01);
        t = __dadd_rn(t, e11);
        return scale_down<2>(t);
    } else {
        return ((e00 + e10) + (e01 + e11)) * (T)0.25;
    }
}

// The correction at interior fine point (i, j); coarse point (I, J) lies on
// fine point (2I, 2J), and the coarse ghost ring holds zeros.  Columns
// i >> 1 and (i + 1) >> 1 are the two coarse columns around an odd i and both
// the one under an even i (rows likewise); the value for each parity of i is
// formed and one is selected, so neighbouring lanes (alternating parities) do
// not diverge.  Each value is the prolongation kernel's formula for its parity.
template <typename T, bool EXACT>
__device__ __forceinline__ T prolong_at(const MgXferArgs &x, int i, int j) {
    const T *e = (const T *)x.ec;
    const long long ldc = x.ldc;
    const int cl = i >> 1, cr = (i + 1) >> 1;
    const bool odd_i = i & 1;
    const T *r0 = e + (long long)(j >> 1) * ldc;
    if (j & 1) {
        const T *r1 = r0 + ldc;
        const T e00 = r0[cl], e10 = r0[cr], e01 = r1[cl], e11 = r1[cr];
        if constexpr (EXACT) {
            // both parities from one chain of sums (avg2 is its first, avg4 all three)
            const double t1 = __dadd_rn(e00, odd_i ? e10 : e01);
            const double t3 = __dadd_rn(__dadd_rn(t1, e01), e11);
            const double v2 = scale_down<1>(t1), v4 = scale_down<2>(t3);
            return odd_i ? v4 : v2;
        }
        const T vo = avg4<T, EXACT>(e00, e10, e01, e11), ve = avg2<T, EXACT>(e00, e01);
        return odd_i ? vo : ve;
    }
    const T e00 = r0[cl], e10 = r0[cr];
    const T vo = avg2<T, EXACT>(e00, e10);
    return odd_i ? vo : e00;
}

// RPT rows per thread: thread (tx, ty) of a (TX, BY) block owns rows
// ty + m BY (m < RPT) of a TX x (BY RPT) subdomain, so each thread keeps RPT
// independent loads of u and f in flight (one point per thread leaves too
// few bytes in flight per SM to cover HBM latency).
template <typename T, bool EXACT, int RPT, int STAGE>
__global__ void __launch_bounds__(1024 / RPT, (RPT == 1 && STAGE == MG_PLAIN) ? 2 : 1)
    mg_smooth_kernel(const MgSmoothArgs a) {
    extern __shared__ __align__(16) unsigned char mg_smem[];
    const int TX = blockDim.x, BY = blockDim.y, TY = BY * RPT, lw = TX + 2, lh = TY + 2;
    T *buf0 = (T *)mg_smem, *buf1 = buf0 + lw * lh;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int i = 1 + blockIdx.x * TX + tx, j0 = 1 + blockIdx.y * TY;
    const int nx = a.nx, ny = a.ny;
    const long long ld = a.ld;
    const T *__restrict__ u = (const T *)a.uin;
    constexpr int stage = STAGE;
    auto ld_u = [&](int jj, int ii) -> T {
        if (ii > nx + 1 || jj > ny + 1 || stage == MG_RESTRICT) return (T)0;
        T v = ld_g(u + (long long)jj * ld + ii);
        if (stage == MG_PROLONG && ii >= 1 && ii <= nx && jj >= 1 && jj <= ny) {
            const T c = prolong_at<T, EXACT>(a.x, ii, jj);
            v = EXACT ? (T)__dadd_rn(v, c) : v + c;
        }
        return v;
    };
    // every global load first, then the shared-memory stores
    T v0[RPT], hw[RPT], he[RPT], g[RPT];
    bool in[RPT];
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
        const int j = j0 + ty + m * BY;
        in[m] = i <= nx && j <= ny;
        v0[m] = ld_u(j, i);
        if constexpr (EXACT && stage == MG_PROLONG) {
            // one call for both edge columns: here each is binary64 work for the whole warp
            hw[m] = he[m] = (T)0;
            if (tx == 0 || tx == TX - 1) {
                const T h = ld_u(j, tx == 0 ? i - 1 : i + 1);
                if (tx == 0) hw[m] = h;
                if (tx == TX - 1) he[m] = TX == 1 ? ld_u(j, i + 1) : h;
            }
        } else {
            hw[m] = tx == 0 ? ld_u(j, i - 1) : (T)0;
            he[m] = tx == TX - 1 ? ld_u(j, i + 1) : (T)0;
        }
        T fv = (T)0;
        if (in[m]) {
            if constexpr (stage == MG_RESTRICT) {
                fv = restrict_at(a.x, i, j);
                ((T *)a.x.fc)[(long long)j * ld + i] = fv;
            } else {
                fv = ld_g((const T *)a.f + (long long)j * ld + i);
            }
        }
        g[m] = EXACT ? fv : fv * (T)a.finvd;
    }
    const T hs = ty == 0 ? ld_u(j0 - 1, i) : (T)0;
    const T hn = ty == BY - 1 ? ld_u(j0 + TY, i) : (T)0;
    // Binary64 with four equal coefficients: the containers hold the products
    // c u_p, each formed once by its point's thread instead of once per
    // neighbour, and a thread keeps its own values in registers (12 FP64
    // operations a point and subiteration become 9, every rounding unchanged;
    // the FP64 pipe bounds this kernel, see update_from_products; 1023 x 1023 to
    // 1e-8: 5.94 -> 5.30 ms).  Otherwise they hold the values.
    bool share = false;
    if constexpr (EXACT) share = same_bits(a.cW, a.cE) && same_bits(a.cS, a.cN) && same_bits(a.cW, a.cS);
    // The three products by constants of a shared update (c u, (f - sum)/d and the
    // damping) run on the integer pipes; a thread that meets a value they do not
    // cover repeats its points on the FP64 pipe (mul_const: 9 become 6 there).
    auto run = [&](auto share_tag) {
        constexpr bool SH = decltype(share_tag)::value;
        MulConst mc, mi, mo;
        if constexpr (SH) {
            mc = make_mul_const(a.cW);
            mi = make_mul_const(a.invd);
            mo = make_mul_const(a.omega);
        }
        auto term = [&](T v) -> T {
            if constexpr (SH) return (T)mul_rn(v, mc, a.cW);
            else return v;
        };
#pragma unroll
        for (int m = 0; m < RPT; ++m) {
            const int me = (ty + m * BY + 1) * lw + tx + 1;
            const T p0 = term(v0[m]);
            buf0[me] = p0;
            buf1[me] = p0;
            if (tx == 0) { const T w = term(hw[m]); buf0[me - 1] = w; buf1[me - 1] = w; }
            if (tx == TX - 1) { const T e = term(he[m]); buf0[me + 1] = e; buf1[me + 1] = e; }
        }
        if (ty == 0) { const T w = term(hs); buf0[tx + 1] = w; buf1[tx + 1] = w; }
        if (ty == BY - 1) { const T w = term(hn); buf0[(TY + 1) * lw + tx + 1] = w; buf1[(TY + 1) * lw + tx + 1] = w; }
        __syncthreads();
        // one point from its neighbours' terms; INT: collects in bad what it cannot do
        auto update = [&](int m, const T *src, auto int_tag, T &prod, unsigned &bad) -> T {
            constexpr bool INT = decltype(int_tag)::value;
            const int me = (ty + m * BY + 1) * lw + tx + 1;
            const T old = v0[m];
            const T W = src[me - 1], E = src[me + 1], Sv = src[me - lw], Nv = src[me + lw];
            T nv;
            if constexpr (EXACT) {
                double acc;
                if constexpr (SH) {
                    acc = __dadd_rn(W, E);
                    acc = __dadd_rn(acc, Sv);
                    acc = __dadd_rn(acc, Nv);
                } else {
                    acc = __dmul_rn(a.cW, W);
                    acc = __dadd_rn(acc, __dmul_rn(a.cE, E));
                    acc = __dadd_rn(acc, __dmul_rn(a.cS, Sv));
                    acc = __dadd_rn(acc, __dmul_rn(a.cN, Nv));
                }
                const double t = __dsub_rn(g[m], acc);
                if constexpr (INT) {
                    unsigned b0 = 0, b1 = 0, b2 = 0;
                    const double jac = mul_const(t, mi, b0);
                    nv = __dadd_rn(old, mul_const(__dsub_rn(jac, old), mo, b1));
                    prod = mul_const(nv, mc, b2);
                    bad |= (unsigned)(b0 > mi.span) | (unsigned)(b1 > mo.span) | (unsigned)(b2 > mc.span);
                } else {
                    const double jac = __dmul_rn(t, a.invd);
                    nv = __dadd_rn(old, __dmul_rn(a.omega, __dsub_rn(jac, old)));
                    prod = SH ? __dmul_rn(a.cW, nv) : nv;
                }
            } else {
                T t = g[m];
                t = fmaf(a.fN, Nv, t);
                t = fmaf(a.fS, Sv, t);
                t = fmaf(a.fE, E, t);
                t = fmaf(a.fW, W, t);
                nv = fmaf(a.fomega, t - old, old);
                prod = nv;
            }
            return nv;
        };
        // one subiteration; WATCH: true once it leaves every value of the CTA as it was
        const T *src = buf0;
        T *dst = buf1;
        auto step = [&](int s, auto watch_tag) -> bool {
            constexpr bool WATCH = decltype(watch_tag)::value;
            const bool more = s + 1 < a.k;   // the last subiteration's values go to global memory from registers
            T nv[RPT], prod[RPT];
            unsigned bad = 0;
#pragma unroll
            for (int m = 0; m < RPT; ++m) {
                unsigned b = 0;
                nv[m] = update(m, src, std::integral_constant<bool, SH>(), prod[m], b);
                if (in[m]) bad |= b;
            }
            if constexpr (SH) {
                if (bad) {
#pragma unroll
                    for (int m = 0; m < RPT; ++m)
                        nv[m] = update(m, src, std::integral_constant<bool, false>(), prod[m], bad);
                }
            }
            bool changed = false;
#pragma unroll
            for (int m = 0; m < RPT; ++m) {
                if (!in[m]) continue;
                if constexpr (WATCH) changed = changed || bits_differ(nv[m], v0[m]);
                v0[m] = nv[m];
                if (more) dst[(ty + m * BY + 1) * lw + tx + 1] = prod[m];
            }
            if (!more) return false;
            const T *t = src;
            src = dst;
            dst = const_cast<T *>(t);
            if constexpr (WATCH) return !__syncthreads_or(changed);
            __syncthreads();
            return false;
        };
        // Long runs (the coarsest level's) end at their fixed point: once a
        // subiteration leaves every value as it was, bit for bit, so do all that
        // follow.  A level of one point is there after two of its 256 (79 us of a
        // V-cycle in binary64).  Binary32 looks after 2, 8, 32 subiterations and every
        // 64 from there, in a body of its own: the comparison and the vote cost 75 ns a
        // subiteration (6 V-cycles of 63 x 63 with a coarsest level of 15 x 15, which
        // is never there: 263 us without, 376 with one in every subiteration, 276 so).
        int s = 0;
        for (int w = a.k < 16 ? a.k : EXACT ? 0 : 1;; w = EXACT ? w + 1 : w < 31 ? 4 * w + 3 : w + 64) {
            const int plain = min(w, a.k);
            for (; s < plain; ++s) step(s, std::integral_constant<bool, false>());
            if (s >= a.k || step(s, std::integral_constant<bool, true>())) break;
            ++s;
        }
    };
    if constexpr (EXACT) {
        if (share) run(std::integral_constant<bool, true>());
        else run(std::integral_constant<bool, false>());
    } else {
        run(std::integral_constant<bool, false>());
    }
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
        const int j = j0 + ty + m * BY;
        if (in[m]) ((T *)a.uout)[(long long)j * ld + i] = v0[m];
    }
}

__global__ void __launch_bounds__(256) mg_restrict_kernel(const MgXferArgs x) {
    const int I = 1 + blockIdx.x * 32 + threadIdx.x, J = 1 + blockIdx.y * 8 + threadIdx.y;
    if (I > x.ncx || J > x.ncy) return;
    const long long qc = (long long)J * x.ldc + I;
    ((float *)x.fc)[qc] = restrict_at(x, I, J);
    ((float *)x.ec)[qc] = 0.f;
}

// Binary32 smoothing of subdomains 32 columns wide and 4, 8, .. 32 high: a warp owns
// four rows, a lane one column of them, in registers; W/E neighbours come by
// shuffle and only the warps' edge rows pass through shared memory (as in
// vc2d_rows_kernel; the sums are those of mg_smooth_kernel, bit for bit).  Bound by
// HBM on the fine levels: 4095 x 4095, 32 x 8, k = 2
// 57.8 -> 50.6 us.
__global__ void __launch_bounds__(256) mg_smooth_rows_kernel(const MgSmoothArgs a) {
    constexpr int R = 4;
    constexpr unsigned ALL = 0xffffffffu;
    __shared__ float edge[2][8][2][32];   // [parity][warp][first, last row][column]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nx = a.nx, ny = a.ny;
    const long long ld = a.ld;
    const int i = 1 + blockIdx.x * 32 + lane, j0 = 1 + (blockIdx.y * nw + w) * R;
    const float *__restrict__ u = (const float *)a.uin, *__restrict__ f = (const float *)a.f;
    auto ld_u = [&](int jj, int ii) -> float {
        return ii <= nx + 1 && jj <= ny + 1 ? __ldg(u + (long long)jj * ld + ii) : 0.f;
    };
    const bool edge_lane = lane == 0 || lane == 31;
    float v[R], hx[R], g[R];
    bool in[R];
    float top = ld_u(j0 - 1, i), bot = ld_u(j0 + R, i);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = j0 + r;
        in[r] = i <= nx && j <= ny;
        v[r] = ld_u(j, i);
        hx[r] = edge_lane ? ld_u(j, lane == 0 ? i - 1 : i + 1) : 0.f;
        g[r] = in[r] ? __ldg(f + (long long)j * ld + i) : 0.f;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) g[r] = g[r] * a.finvd;
    for (int s = 0; s < a.k; ++s) {
        float prev = top;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float cur = v[r];
            float W = __shfl_up_sync(ALL, cur, 1), E = __shfl_down_sync(ALL, cur, 1);
            if (lane == 0) W = hx[r];
            if (lane == 31) E = hx[r];
            float t = g[r];
            t = fmaf(a.fN, r < R - 1 ? v[r < R - 1 ? r + 1 : 0] : bot, t);
            t = fmaf(a.fS, prev, t);
            t = fmaf(a.fE, E, t);
            t = fmaf(a.fW, W, t);
            v[r] = in[r] ? fmaf(a.fomega, t - cur, cur) : cur;
            prev = cur;
        }
        if (nw > 1 && s + 1 < a.k) {
            const int par = s & 1;
            edge[par][w][0][lane] = v[0];
            edge[par][w][1][lane] = v[R - 1];
            __syncthreads();
            if (w > 0) top = edge[par][w - 1][1][lane];
            if (w < nw - 1) bot = edge[par][w + 1][0][lane];
        }
    }
    float *__restrict__ uo = (float *)a.uout;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (in[r]) uo[(long long)(j0 + r) * ld + i] = v[r];
}

// Binary64 restriction of a block of 32 x 8 coarse points: the 65 x 17 fine
// residuals around them are formed once each in shared memory and weighted from
// there.  A thread per coarse point (the binary32 kernel above) forms nine residuals of ten operations per coarse
// point; each fine one is needed 2.25 times on average, so on the FP64 pipe, which
// bounds both, 104 operations a coarse point become some 50 (30 with the products
// by constants, shared between neighbours where the coefficients are equal, on
// the integer pipes).  Sums in restrict_at's order; 4 r + 2 s + t with exact
// powers of two is 2 (2 r + s) + t, two fused operations with the same roundings.
// 4095 x 4095 fine points: 327 us; a coarse level's launch 4 to 7 us, where forming
// nine residuals a point inside the next smoothing made that launch 13 us longer.
__global__ void __launch_bounds__(256) mg_restrict_tile_kernel(const MgXferArgs x) {
    constexpr int BW = 32, BH = 8, RW = 2 * BW + 1, RH = 2 * BH + 1, UW = RW + 2, UH = RH + 2;
    __shared__ double U[UH][UW], P[UH][UW];   // u and c u on the residuals' points and one around
    __shared__ double R[RH][RW + 1];
    const double *u = (const double *)x.u, *f = (const double *)x.f;
    const int I0 = 1 + blockIdx.x * BW, J0 = 1 + blockIdx.y * BH;
    const int fx = 2 * I0 - 2, fy = 2 * J0 - 2;   // fine point of U[0][0]
    const int tid = threadIdx.x + 32 * threadIdx.y;
    const bool iso = same_bits(x.cW, x.cE) && same_bits(x.cS, x.cN) && same_bits(x.cW, x.cS);
    const MulConst mc = make_mul_const(x.cW), md = make_mul_const(x.d);
    // every load first: one round of memory latency per CTA, which is most of what
    // a coarse level's launch costs
    constexpr int NU = (UW * UH + 255) / 256, NR = (RW * RH + 255) / 256;
    double uv[NU], fv[NR];
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = tid + 256 * k, c = t % UW, r = t / UW;
        uv[k] = 0.0;
        if (t < UW * UH && fx + c <= x.nx + 1 && fy + r <= x.ny + 1) uv[k] = __ldg(u + (long long)(fy + r) * x.ld + fx + c);
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int t = tid + 256 * k, gx = fx + 1 + t % RW, gy = fy + 1 + t / RW;
        fv[k] = 0.0;
        if (t < RW * RH && gx <= x.nx && gy <= x.ny) fv[k] = __ldg(f + (long long)gy * x.ld + gx);
    }
#pragma unroll
    for (int k = 0; k < NU; ++k) {
        const int t = tid + 256 * k, c = t % UW, r = t / UW;
        if (t >= UW * UH) continue;
        U[r][c] = uv[k];
        if (iso) P[r][c] = mul_rn(uv[k], mc, x.cW);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int t = tid + 256 * k, c = t % RW, r = t / RW;
        if (t >= RW * RH || fx + 1 + c > x.nx || fy + 1 + r > x.ny) continue;   // (no coarse point here has such a neighbour)
        double au = mul_rn(U[r + 1][c + 1], md, x.d);
        if (iso) {
            au = __dadd_rn(au, P[r + 1][c]);
            au = __dadd_rn(au, P[r + 1][c + 2]);
            au = __dadd_rn(au, P[r][c + 1]);
            au = __dadd_rn(au, P[r + 2][c + 1]);
        } else {
            au = __dadd_rn(au, __dmul_rn(x.cW, U[r + 1][c]));
            au = __dadd_rn(au, __dmul_rn(x.cE, U[r + 1][c + 2]));
            au = __dadd_rn(au, __dmul_rn(x.cS, U[r][c + 1]));
            au = __dadd_rn(au, __dmul_rn(x.cN, U[r + 2][c + 1]));
        }
        R[r][c] = __dsub_rn(fv[k], au);
    }
    __syncthreads();
    const int I = I0 + (int)threadIdx.x, J = J0 + (int)threadIdx.y;
    if (I > x.ncx || J > x.ncy) return;
    const int c = 2 * threadIdx.x + 1, r = 2 * threadIdx.y + 1;   // R of fine point (2I, 2J)
    double s1 = __dadd_rn(R[r][c - 1], R[r][c + 1]);
    s1 = __dadd_rn(s1, R[r - 1][c]);
    s1 = __dadd_rn(s1, R[r + 1][c]);
    double s2 = __dadd_rn(R[r - 1][c - 1], R[r - 1][c + 1]);
    s2 = __dadd_rn(s2, R[r + 1][c - 1]);
    s2 = __dadd_rn(s2, R[r + 1][c + 1]);
    const double t = __fma_rn(2.0, __fma_rn(2.0, R[r][c], s1), s2);
    const long long qc = (long long)J * x.ldc + I;
    ((double *)x.fc)[qc] = scale_down<4>(t);
    ((double *)x.ec)[qc] = 0.0;
}

// One thread per coarse cell (ca, cb), ca in [0, ncx], cb in [0, ncy]: the fine
// points (2ca | 2ca+1, 2cb | 2cb+1), each with the oracle's formula for its parity
// (row and column 0 are ghosts and left alone).  The two points of a row are one
// aligned vector, so a warp reads and writes whole lines of every fine row (as
// the cell's inner points, 2ca+1 | 2ca+2, they were two strided halves: 4095 x
// 4095 binary32 58.8 -> 25.3 us; binary64, bound by its sums, 100 -> 107).
template <typename T, bool EXACT>
__global__ void __launch_bounds__(256) mg_prolong_kernel(const MgXferArgs x) {
    const int ca = blockIdx.x * 32 + threadIdx.x, cb = blockIdx.y * 8 + threadIdx.y;
    if (ca > x.ncx || cb > x.ncy) return;
    const T *e = (const T *)x.ec;
    const long long r0 = (long long)cb * x.ldc, r1 = r0 + x.ldc;
    const T e00 = e[r0 + ca], e10 = e[r0 + ca + 1], e01 = e[r1 + ca], e11 = e[r1 + ca + 1];
    struct alignas(2 * sizeof(T)) Pair {
        T x, y;
    };
    auto add = [](T u, T v) -> T { return EXACT ? (T)__dadd_rn(u, v) : u + v; };
    auto put = [&](int jj, T ve, T vo) {   // corrections of the row's even and odd column
        const long long q = (long long)jj * x.ld + 2 * ca;
        const T *ui = (const T *)x.u + q;
        T *uo = (T *)x.uout + q;
        if (ca > 0) {
            const Pair u = *(const Pair *)ui;
            *(Pair *)uo = Pair{add(u.x, ve), add(u.y, vo)};
        } else {
            uo[1] = add(ui[1], vo);
        }
    };
    if (cb > 0) put(2 * cb, e00, avg2<T, EXACT>(e00, e10));
    put(2 * cb + 1, avg2<T, EXACT>(e00, e01), avg4<T, EXACT>(e00, e10, e01, e11));
}

MgSmoothArgs smooth_args(const MgLevel &L, const void *f, const void *uin, void *uout, int k, double omega,
                         double sigma_const) {
    MgSmoothArgs a;
    memset(&a, 0, sizeof(a));
    a.f = f;
    a.uin = uin;
    a.uout = uout;
    a.ld = L.ld;
    a.nx = L.nx;
    a.ny = L.ny;
    a.k = k;
    a.stage = MG_PLAIN;
    a.cW = L.cW; a.cE = L.cE; a.cS = L.cS; a.cN = L.cN;
    a.invd = 1.0 / (L.cD + sigma_const);
    a.omega = omega;
    a.fW = (float)(-L.cW * a.invd); a.fE = (float)(-L.cE * a.invd);
    a.fS = (float)(-L.cS * a.invd); a.fN = (float)(-L.cN * a.invd);
    a.finvd = (float)a.invd;
    a.fomega = (float)omega;
    return a;
}

// Launch one smoothing cycle on level l (buffer cur -> 1 - cur); tile tx x ty.
// x: the transfer a MG_RESTRICT / MG_PROLONG launch forms while staging.
void launch_smooth(hj_handle *h, int l, int cur, int tx, int ty, int k, double omega, cudaStream_t s,
                   int stage = MG_PLAIN, const MgXferArgs *x = nullptr) {
    const MgLevel &L = h->mg[l];
    void *buf[2] = {L.a, L.b};
    MgSmoothArgs a = smooth_args(L, L.f, buf[cur], buf[1 - cur], k, omega, h->d.sigma_const);
    if (x) {
        a.stage = stage;
        a.x = *x;
    }
    // rows per thread: 4 (or 2) when the subdomain height allows, 1 otherwise
    const bool f64 = h->fam_outer == FAM_F64;
    int rpt = (ty % 4 == 0 && ty >= 8) ? 4 : (ty % 2 == 0 && ty >= 4) ? 2 : 1;
    // binary64 is bound by the FP64 pipes, one per sub-partition: at least four
    // warps a CTA before rows are added to a thread
    while (f64 && rpt > 1 && tx * (ty / rpt) < 128) rpt /= 2;
    const dim3 block(tx, ty / rpt), grid((L.nx + tx - 1) / tx, (L.ny + ty - 1) / ty);
    if (!f64 && a.stage == MG_PLAIN && tx == 32 && ty % 4 == 0 && ty <= 32) {
        mg_smooth_rows_kernel<<<grid, 32 * (ty / 4), 0, s>>>(a);
        return;
    }
    const int smem = 2 * (tx + 2) * (ty + 2) * (f64 ? 8 : 4);
#define HJ_MG_SMOOTH(T, EX, ST)                                                            \
    do {                                                                                   \
        if (rpt == 4) mg_smooth_kernel<T, EX, 4, ST><<<grid, block, smem, s>>>(a);         \
        else if (rpt == 2) mg_smooth_kernel<T, EX, 2, ST><<<grid, block, smem, s>>>(a);    \
        else mg_smooth_kernel<T, EX, 1, ST><<<grid, block, smem, s>>>(a);                  \
    } while (0)
#define HJ_MG_SMOOTH_ST(T, EX)                                        \
    do {                                                              \
        if (a.stage == MG_PROLONG) HJ_MG_SMOOTH(T, EX, MG_PROLONG); \
        else HJ_MG_SMOOTH(T, EX, MG_PLAIN);                           \
    } while (0)
    if (f64) HJ_MG_SMOOTH_ST(double, true);
    else if (a.stage == MG_RESTRICT) HJ_MG_SMOOTH(float, false, MG_RESTRICT);   // (binary32 only, record_level)
    else HJ_MG_SMOOTH_ST(float, false);
#undef HJ_MG_SMOOTH_ST
#undef HJ_MG_SMOOTH
}

MgXferArgs xfer_args(const hj_handle *h, int l) {
    const MgLevel &F = h->mg[l], &Cc = h->mg[l + 1];
    MgXferArgs x;
    memset(&x, 0, sizeof(x));
    x.ld = F.ld;
    x.ldc = Cc.ld;
    x.nx = F.nx; x.ny = F.ny;
    x.ncx = Cc.nx; x.ncy = Cc.ny;
    x.d = F.cD + h->d.sigma_const;
    x.cW = F.cW; x.cE = F.cE; x.cS = F.cS; x.cN = F.cN;
    return x;
}

// Levels up to this many points fold the transfers into their smoothing
// launches (record_level).
constexpr long long kMgFuseMaxPoints = 512LL * 512;

void launch_restrict(const hj_handle *h, const MgXferArgs &x, int ncx, int ncy, cudaStream_t s) {
    const dim3 g((ncx + 31) / 32, (ncy + 7) / 8), b(32, 8);
    if (h->fam_outer == FAM_F64) mg_restrict_tile_kernel<<<g, b, 0, s>>>(x);
    else mg_restrict_kernel<<<g, b, 0, s>>>(x);
}

// The V-cycle below level l, starting from buffer cur of level l; returns the
// buffer that holds the level's result.  rin: the restriction from the finer
// level, still to be formed (by this level's first smoothing launch, or by a
// restriction launch when the level starts without one); null at level 0.
//
// Launch count: on levels of a few hundred thousand points or fewer a launch
// costs its fixed latency (a few microseconds) whatever its size, so there the
// transfers are folded into the launches next to them where the result is the
// same: in binary32 the restriction into the coarse level's first smoothing (which forms
// the coarse RHS for its subdomain while staging, stores it for the level's
// later launches, and starts from a zero correction, as the restriction sets
// it; in binary64, bound by the sums that the subdomains' halos would repeat, it stays a
// launch) and the prolongation into the fine level's first post-smoothing (which
// stages u + P e for its subdomain and halo).  On larger levels the separate
// transfer kernels stay: they form each value once with coalesced accesses,
// where a smoothing launch would recompute the halo's.  The coarsest level's
// cycles are always one launch (one subdomain whose halo is the level's fixed
// zero boundary, so c cycles of k subiterations are c k subiterations).
int record_level(hj_handle *h, int l, int cur, cudaStream_t s, const MgXferArgs *rin) {
    const hj_params &p = h->p;
    const int levels = (int)h->mg.size();
    const MgLevel &L = h->mg[l];
    if (l == levels - 1) {
        if (p.mg_coarse_cycles <= 0) {
            if (rin) launch_restrict(h, *rin, L.nx, L.ny, s);
            return cur;
        }
        if (l > 0) {
            const bool own = h->fam_outer == FAM_F64;   // its own restriction launch
            if (own) launch_restrict(h, *rin, L.nx, L.ny, s);
            launch_smooth(h, l, cur, L.nx, L.ny, p.mg_coarse_k * p.mg_coarse_cycles, 1.0, s, MG_RESTRICT,
                          own ? nullptr : rin);
            return cur ^ 1;
        }
        for (int c = 0; c < p.mg_coarse_cycles; ++c) {
            launch_smooth(h, l, cur, L.nx, L.ny, p.mg_coarse_k, 1.0, s);
            cur ^= 1;
        }
        return cur;
    }
    const bool small = (long long)L.nx * L.ny <= kMgFuseMaxPoints;
    const MgXferArgs *pending = rin;
    // (binary64: forming nine residuals per point in the smoother's staging costs
    // more FP64 time than the tiled restriction's launch: see mg_restrict_tile_kernel)
    if (pending && (!small || p.mg_pre == 0 || h->fam_outer == FAM_F64)) {
        launch_restrict(h, *pending, L.nx, L.ny, s);
        pending = nullptr;
    }
    for (int c = 0; c < p.mg_pre; ++c) {
        launch_smooth(h, l, cur, p.tile_x, p.tile_y, p.k, p.mg_omega, s, MG_RESTRICT, pending);
        pending = nullptr;
        cur ^= 1;
    }
    MgXferArgs x = xfer_args(h, l);
    const MgLevel &Cc = h->mg[l + 1];
    x.f = L.f;
    x.u = cur ? L.b : L.a;
    x.fc = Cc.f;
    x.ec = Cc.a;
    const int ce = record_level(h, l + 1, 0, s, &x);
    x.ec = ce ? Cc.b : Cc.a;
    x.u = cur ? L.b : L.a;
    // level 0 must end in buffer a (the graph is replayed from there): when
    // pre + post is odd, a prolongation launch writes the other buffer
    const bool flip = l == 0 && ((p.mg_pre + p.mg_post) & 1);
    const bool fuse = small && p.mg_post > 0 && !flip;
    if (!fuse) {
        x.uout = flip ? (cur ? L.a : L.b) : const_cast<void *>(x.u);
        const dim3 g((Cc.nx + 1 + 31) / 32, (Cc.ny + 1 + 7) / 8), b(32, 8);   // coarse cells 0..ncx x 0..ncy
        if (h->fam_outer == FAM_F64) mg_prolong_kernel<double, true><<<g, b, 0, s>>>(x);
        else mg_prolong_kernel<float, false><<<g, b, 0, s>>>(x);
        if (flip) cur ^= 1;
    }
    for (int c = 0; c < p.mg_post; ++c) {
        launch_smooth(h, l, cur, p.tile_x, p.tile_y, p.k, p.mg_omega, s, MG_PROLONG, (fuse && c == 0) ? &x : nullptr);
        cur ^= 1;
    }
    return cur;
}

RedArgs store_red(const hj_handle *h) {
    RedArgs r;
    memset(&r, 0, sizeof(r));
    r.partials = h->partials;
    r.gpart = h->gpart;
    r.gcnt = h->gcnt;
    r.fcnt = h->fcnt;
    r.hist = h->hist;
    r.out = h->rstore;
    r.ctl = h->ctl;
    r.mode = RED_STORE;
    r.scale = 1.0;
    return r;
}

// ||f - A u||^2 of the level-0 buffer a into pinned host memory (h_rstore).
cudaError_t record_residual(hj_handle *h, cudaStream_t s) {
    const MgLevel &L = h->mg[0];
    const hj_desc &d = h->d;
    cudaError_t e = launch_residual_ex(2, d.dtype == HJ_F64, L.f, L.a, nullptr, d.ld, d.ld, d.nx, d.ny, d.cW, d.cE,
                                       d.cS, d.cN, d.cD + d.sigma_const, 0, nullptr, store_red(h), s);
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(h->h_rstore, h->rstore, sizeof(double), cudaMemcpyDeviceToHost, s);
}

}  // namespace

int mg_levels_of(int nx, int ny) {
    int L = 1;
    while (nx > 1 && ny > 1 && (nx & 1) && (ny & 1)) {
        nx = (nx - 1) / 2;
        ny = (ny - 1) / 2;
        ++L;
    }
    return L;
}

int mg_setup(hj_handle *h, int levels) {
    const hj_desc &d = h->d;
    const size_t esz = h->esz;
    h->mg.resize(levels);
    int nx = d.nx, ny = d.ny;
    double cW = d.cW, cE = d.cE, cS = d.cS, cN = d.cN, cD = d.cD;
    size_t total = 0;
    for (int l = 0; l < levels; ++l) {
        MgLevel &L = h->mg[l];
        L.nx = nx;
        L.ny = ny;
        L.ld = l == 0 ? d.ld : ((long long)nx + 2 + 31) / 32 * 32;
        L.cW = cW; L.cE = cE; L.cS = cS; L.cN = cN; L.cD = cD;
        total += 3 * (size_t)(ny + 2) * L.ld * esz;
        nx = (nx - 1) / 2;
        ny = (ny - 1) / 2;
        cW /= 4.0; cE /= 4.0; cS /= 4.0; cN /= 4.0; cD /= 4.0;
    }
    if (dmalloc(&h->mg_arena, total) != cudaSuccess) {
        cudaGetLastError();
        return seterr(HJ_ERR_NO_MEMORY, "cudaMalloc of %zu bytes failed (multigrid levels)", total);
    }
    CKR(cudaMemset(h->mg_arena, 0, total));
    unsigned char *p = (unsigned char *)h->mg_arena;
    for (int l = 0; l < levels; ++l) {
        MgLevel &L = h->mg[l];
        const size_t b = (size_t)(L.ny + 2) * L.ld * esz;
        L.a = p; p += b;
        L.b = p; p += b;
        L.f = p; p += b;
    }
    return HJ_OK;
}

// V-cycles until ||r_c|| <= tol ||r_0|| (or fixed_cycles V-cycles), u in/out.
int solve_mg(hj_handle *h, const void *f, void *u, cudaStream_t s, hj_stats *st) {
    const MgLevel &L0 = h->mg[0];
    CKR(cudaMemcpyAsync(L0.a, u, h->grid_bytes, cudaMemcpyDeviceToDevice, s));
    CKR(cudaMemcpyAsync(L0.b, u, h->grid_bytes, cudaMemcpyDeviceToDevice, s));
    CKR(cudaMemcpyAsync(L0.f, f, h->grid_bytes, cudaMemcpyDeviceToDevice, s));
    // one graph per kind of run: a converging run's V-cycle ends with the
    // level-0 residual norm (binary64 arithmetic, a large share of a binary32
    // V-cycle on this part's FP64 pipe) and its copy to pinned host memory; a
    // fixed-cycle run reads no residual, so its V-cycle has neither
    const long long fixed = h->p.fixed_cycles;
    cudaGraphExec_t &exec = fixed > 0 ? h->mg_exec_fixed : h->mg_exec;
    if (!exec) {
        cudaGraph_t graph;
        CKR(cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal));
        const int fin = record_level(h, 0, 0, h->cap, nullptr);
        cudaError_t le = cudaGetLastError();
        if (le == cudaSuccess && fixed <= 0) le = record_residual(h, h->cap);
        cudaError_t ee = cudaStreamEndCapture(h->cap, &graph);
        if (le != cudaSuccess) return seterr(HJ_ERR_CUDA, "multigrid capture: %s", cudaGetErrorString(le));
        if (ee != cudaSuccess) return seterr(HJ_ERR_CUDA, "cudaStreamEndCapture: %s", cudaGetErrorString(ee));
        if (fin != 0) {
            cudaGraphDestroy(graph);
            return seterr(HJ_ERR_CUDA, "internal: V-cycle does not end in the level-0 buffer");
        }
        cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ie != cudaSuccess) {
            exec = nullptr;
            return seterr(HJ_ERR_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(ie));
        }
    }
    long long c = 0, hl = 0;
    bool stalled = false;
    int status = HJ_OK;
    double r0 = -1.0, rc = -1.0;
    if (fixed > 0) {
        for (c = 0; c < fixed; ++c) CKR(cudaGraphLaunch(exec, s));
    } else {
        CKR(record_residual(h, s));
        CKR(cudaStreamSynchronize(s));
        r0 = rc = sqrt(std::max(h->h_rstore[0], 0.0));
        status = HJ_ERR_NOT_CONVERGED;
        // the last kStall + 1 residuals: a V-cycle contracts by a fixed factor
        // until the storage precision's floor (binary32 u: about eps |u| / h^2
        // relative), so a drop of less than 1 % over kStall V-cycles ends the solve
        constexpr int kStall = 4;
        double ring[kStall + 1];
        for (;;) {
            if (st && st->history && hl < st->history_cap) st->history[hl++] = rc;
            ring[c % (kStall + 1)] = rc;
            if (!std::isfinite(rc)) { status = HJ_ERR_DIVERGED; break; }
            if (rc <= h->p.tol * r0) { status = HJ_OK; break; }
            if (c >= h->p.max_cycles) break;
            if (c >= kStall && rc > 0.99 * ring[(c - kStall) % (kStall + 1)]) { stalled = true; break; }
            CKR(cudaGraphLaunch(exec, s));
            CKR(cudaStreamSynchronize(s));
            rc = sqrt(std::max(h->h_rstore[0], 0.0));
            ++c;
        }
    }
    CKR(cudaMemcpyAsync(u, L0.a, h->grid_bytes, cudaMemcpyDeviceToDevice, s));
    CKR(cudaStreamSynchronize(s));
    if (st) {
        st->cycles = c;
        st->cycles_launched = c;
        st->inner_cycles = 0;
        st->outer_steps = 0;
        st->res0 = r0;
        st->res_final = rc;
        st->rel_final = r0 > 0 ? rc / r0 : 0.0;
        st->history_len = hl;
        st->persistent = 0;
    }
    if (status == HJ_ERR_DIVERGED) return seterr(HJ_ERR_DIVERGED, "residual became non-finite at V-cycle %lld", c);
    if (status == HJ_ERR_NOT_CONVERGED)
        return seterr(HJ_ERR_NOT_CONVERGED, "tolerance %g not met after %lld V-cycles (rel %g%s)", h->p.tol, c,
                      r0 > 0 ? rc / r0 : 0.0, stalled ? "; the residual stopped falling" : "");
    return HJ_OK;
}

}  // namespace hj
