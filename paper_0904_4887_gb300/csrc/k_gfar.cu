// The smooth part of the Eq. 9 sum through its Fourier series.
//
// gamma(r) = sum over atoms a and all their periodic images of q_a exp(-d),
// q_a = exp(rvdw_a), needs every image within ~41 A of a point: 2,400 images per
// point for 288 atoms in a 26 x 26 x 52 A cell. Split exp(-d) = near(d) + far(d)
// with far(d) = exp(-d) w(d), w(d) = erfc((d0 - d)/s)/2. near falls below the bound
// on the dropped tail within rn (8 A at K = 15: 18 images per point) and is summed on
// the grid. far is smooth (its cusp at d = 0 is suppressed by w(0) = 1e-15), so its
// transform
//     F(k) = (4 pi/|k|) int_0^R d exp(-d) w(d) sin(|k| d) dd      (R the sum's radius)
// falls like exp(-(k s)^2/4) to ~1e-15 at K, and
//     gamma_far(r) = (1/V) sum_{|k| <= K} F(k) S(k) exp(i k.r),  S(k) = sum_a q_a exp(-i k.R_a)
// is exact to rounding. It is Ewald's idea (Ann. Phys. 369, 253, 1921), the
// splitting function multiplying exp(-d) so that both parts decay. The series is
// summed by the band-limited FFT of k_fft.cu. The force's sum_i W_i d gamma_i/d R_a is the
// adjoint: the forward transform of W, then a sum over modes per atom.
//
// On the 192 x 192 x 384 slab with 288 atoms (K = 15): eps 80.8 -> 4.3 ms, of which near
// 3.0, modes 0.5, transforms 0.8; its force 74.9 -> 5.0 ms, of which near 2.8, modes 1.3,
// transforms 0.8. Errors against 64-bit sums on seven slabs: eps 1.2e-14 to 3.6e-14 of its
// largest value (direct sums 1.2e-14 to 4.2e-14), forces 7e-15 to 2e-14 (1.7e-13 to 3.6e-12:
// the direct sum's far pairs are in FP32).
#include "df.cuh"
#include "gp_common.cuh"

namespace gp {
namespace {

constexpr double kSqrtPi = 1.7724538509055160273;

__device__ __forceinline__ double near_of(double d, double d0, double s) {
    return exp(-d) * 0.5 * erfc((d - d0) / s);
}

// -near'(d)/d
__device__ __forceinline__ double near_slope(double d, double d0, double s) {
    const double u = (d - d0) / s;
    return exp(-d) * (0.5 * erfc(u) + exp(-u * u) / (s * kSqrtPi)) / d;
}

// values at the n Chebyshev points of the first kind -> monomial coefficients in t
// (discrete cosine transform, then T_{m+1} = 2 t T_m - T_{m-1}; as for the switching tables)
template <int n>
__device__ void cheb_monomials(const double* fv, double* mono) {
    double c[n], Tm1[n], Tm[n];
    for (int m = 0; m < n; ++m) {
        double acc = 0.0;
        for (int j = 0; j < n; ++j) acc += fv[j] * cospi(m * (j + 0.5) / n);
        c[m] = acc * 2.0 / n;
    }
    c[0] *= 0.5;
    for (int e = 0; e < n; ++e) { Tm1[e] = Tm[e] = 0.0; mono[e] = 0.0; }
    Tm1[0] = 1.0;
    Tm[1] = 1.0;
    mono[0] = c[0];
    mono[1] = c[1];
    for (int m = 2; m < n; ++m) {
        double Tn[n];
        for (int e = 0; e < n; ++e) Tn[e] = (e > 0 ? 2.0 * Tm[e - 1] : 0.0) - Tm1[e];
        for (int e = 0; e < n; ++e) { mono[e] += c[m] * Tn[e]; Tm1[e] = Tm[e]; Tm[e] = Tn[e]; }
    }
}

// One block per interval of |k|: the transform at the interval's Chebyshev points
// by the trapezoidal rule (the integrand is entire, vanishes at both ends and is
// band-limited to ~K + 12, so a step of 0.2 A is exact to rounding), a warp a point.
__global__ void k_far_ftab(GammaFar f) {
    __shared__ double v[kFarDeg + 1];
    const int iv = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double dk = f.K / kFarIv;
    const int nq = (int)ceil(f.rcut / 0.2);
    const double step = f.rcut / nq;
    if (w <= kFarDeg) {
        const double k = (iv + 0.5 + 0.5 * cospi((w + 0.5) / (kFarDeg + 1))) * dk;
        double acc = 0.0;
        for (int q = 1 + lane; q <= nq; q += 32) {
            const double d = q * step;
            const double t = d * exp(-d) * 0.5 * erfc((f.d0 - d) / f.s) * sin(k * d);
            acc += q == nq ? 0.5 * t : t;
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) v[w] = acc * step * 4.0 * kPi / k;
    }
    __syncthreads();
    if (threadIdx.x == 0) cheb_monomials<kFarDeg + 1>(v, f.ftab + iv * (kFarDeg + 1));
}

__device__ __forceinline__ double far_transform(const GammaFar& f, double k) {
    const double x = k * (kFarIv / f.K);
    const int iv = min((int)x, kFarIv - 1);
    const double t = 2.0 * (x - iv) - 1.0;
    const double* c = f.ftab + iv * (kFarDeg + 1);
    double acc = c[kFarDeg];
#pragma unroll
    for (int e = kFarDeg - 1; e >= 0; --e) acc = fma(acc, t, c[e]);
    return acc;
}

// near(d) and -near'(d)/d on each interval of d^2: kNearSplit float pairs, then singles.
// A warp an interval: its lanes take the nodes, its first lane the coefficients.
__global__ void k_near_tabs(GammaFar f) {
    __shared__ double v[kNearDeg + 1], mono[kNearDeg + 1];
    const bool slope = blockIdx.x >= kNearIv;
    const int iv = slope ? blockIdx.x - kNearIv : blockIdx.x, lane = threadIdx.x;
    const double dq = f.rn * f.rn / kNearIv;
    if (lane <= kNearDeg) {
        const double d = sqrt((iv + 0.5 + 0.5 * cospi((lane + 0.5) / (kNearDeg + 1))) * dq);
        v[lane] = slope ? near_slope(d, f.d0, f.s) : near_of(d, f.d0, f.s);
    }
    __syncwarp();
    if (lane == 0) cheb_monomials<kNearDeg + 1>(v, mono);
    __syncwarp();
    // float o of the row: pairs (hi, lo) of the first kNearSplit coefficients, then single ones
    float* dst = reinterpret_cast<float*>((slope ? f.htab : f.ntab) + kNearVec * iv);
    if (lane < 4 * kNearVec) {
        const int e = lane < 2 * kNearSplit ? lane >> 1 : lane - kNearSplit;
        const double c = e <= kNearDeg ? mono[e] : 0.0;
        const float hi = (float)c;
        dst[lane] = lane < 2 * kNearSplit && (lane & 1) ? (float)(c - (double)hi) : hi;
    }
}

// phases exp(i 2 pi m x_a / L) of every atom, axis and mode index
__global__ void k_far_phases(Geo g, Atoms at, GammaFar f) {
    const int nx = f.mx + 1, ny = f.my + 1, nz = f.mz + 1, per = nx + ny + nz;
    const long total = (long)at.n * per;
    for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < total; q += (long)gridDim.x * blockDim.x) {
        const int a = (int)(q / per), r = (int)(q % per);
        const int axis = r < nx ? 0 : (r < nx + ny ? 1 : 2);
        const int m = axis == 0 ? r : (axis == 1 ? r - nx : r - nx - ny);
        const double L = axis == 0 ? g.lx : (axis == 1 ? g.ly : g.lz);
        double es, ec;
        sincospi(2.0 * m * (at.w64[3 * a + axis] / L), &es, &ec);
        const float2 c = split_to_float2(ec), sn = split_to_float2(es);
        const float4 e = make_float4(c.x, c.y, sn.x, sn.y);
        if (axis == 0) f.ex[(long)a * nx + m] = e;
        else if (axis == 1) f.ey[(long)a * ny + m] = e;
        else {
            f.ez[(long)a * nz + m] = e;
            f.ezt[(long)m * at.n + a] = e;
        }
    }
}

// kind 2: the range of planes where some but not all of the lower atoms lie above
__global__ void k_far_split(int n, int nz, const GAtom* ga, int* kz) {
    __shared__ int hi, lo;
    if (threadIdx.x == 0) { hi = 0; lo = nz; }
    __syncthreads();
    for (int a = threadIdx.x; a < n; a += blockDim.x) {
        const int k = ga[a].kzl;
        if (k > 0) { atomicMax(&hi, k); atomicMin(&lo, k); }
    }
    __syncthreads();
    if (threadIdx.x == 0) { kz[0] = hi; kz[1] = lo; }
}

// a complex number as two float pairs
struct cdf { df re, im; };
__device__ __forceinline__ cdf as_cdf(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ df df_neg(df a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ cdf cdf_mul(cdf a, cdf b) {
    return {df_add(df_mul(a.re, b.re), df_neg(df_mul(a.im, b.im))), df_add(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}

// e^{i (kx x + ky y)} of an atom, ky < 0 by conjugating its y factor
__device__ __forceinline__ cdf xy_phase(const GammaFar& f, long a, int kx, int ky) {
    cdf y = as_cdf(f.ey[a * (f.my + 1) + (ky < 0 ? -ky : ky)]);
    if (ky < 0) y.im = df_neg(y.im);
    return cdf_mul(as_cdf(f.ex[a * (f.mx + 1) + kx]), y);
}

// sums of products in df, four of them
struct Acc4 {
    float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
    __device__ __forceinline__ double get(int i) const { return (double)s[i] + (double)c[i]; }
};

// Structure factor times F/V. One block per (kx, ky) column, a thread per kz >= 0; the
// four real products of an atom's x-y factor with its z phase serve kz and -kz. They
// run in df64 (a product and its sum take 15 FP32 instructions; an FP64 FMA holds the
// FP64 pipe for 64 issue slots): relative errors of ~2^-46 of sums whose F/V-weighted
// total, far's part of gamma, is below 0.3. Modes beyond K are zero.
constexpr int kFarCh = 128;                    // atoms staged at a time

__global__ void k_far_modes(int n, GammaFar f, const GAtom* ga) {
    __shared__ cdf cs[kFarCh];
    __shared__ int low[kFarCh];
    const int kx = blockIdx.x % (f.mx + 1), jy = blockIdx.x / (f.mx + 1), ky = jy - f.my, m = threadIdx.x;
    const double gx = kx * f.bx, gy = ky * f.by, gz = m * f.bz;
    const double k2 = gx * gx + gy * gy + gz * gz;
    const bool in = m <= f.mz && k2 <= f.K * f.K;
    Acc4 L, O;                                 // lower atoms (kind 2), the others
    if (gx * gx + gy * gy <= f.K * f.K) {      // the block's column reaches into the sphere
        for (int a0 = 0; a0 < n; a0 += kFarCh) {
            const int na = min(kFarCh, n - a0);
            __syncthreads();
            for (int a = threadIdx.x; a < na; a += blockDim.x) {
                const GAtom g = ga[a0 + a];
                const cdf e = xy_phase(f, a0 + a, kx, ky);
                cs[a] = {df_mul(as_df(g.a), e.re), df_neg(df_mul(as_df(g.a), e.im))};
                low[a] = f.up && g.kzl > 0;
            }
            __syncthreads();
            if (!in) continue;
            auto add = [](Acc4& A, const cdf& c, const cdf& z) {
                df_acc_norm(A.s[0], A.c[0], c.re, z.re);
                df_acc_norm(A.s[1], A.c[1], c.im, z.im);
                df_acc_norm(A.s[2], A.c[2], c.re, z.im);
                df_acc_norm(A.s[3], A.c[3], c.im, z.re);
            };
#pragma unroll 2
            for (int a = 0; a < na; ++a) {
                const cdf c = cs[a], z = as_cdf(__ldg(f.ez + (long)(a0 + a) * (f.mz + 1) + m));
                if (low[a]) add(L, c, z);
                else add(O, c, z);
            }
        }
    }
    if (m > f.mz) return;
    const double w = in ? far_transform(f, sqrt(k2)) * f.inv_v : 0.0;
    const int cols = 2 * f.my + 1, pitch = f.mx + 1;
    auto put = [&](double2* S, double a, double b, double c, double d) {
        S[((long)(f.mz + m) * cols + jy) * pitch + kx] = make_double2(w * (a + b), w * (d - c));
        if (m > 0) S[((long)(f.mz - m) * cols + jy) * pitch + kx] = make_double2(w * (a - b), w * (d + c));
    };
    if (f.up) {
        put(f.s_up, O.get(0), O.get(1), O.get(2), O.get(3));
        put(f.s_all, O.get(0) + L.get(0), O.get(1) + L.get(1), O.get(2) + L.get(2), O.get(3) + L.get(3));
    } else {
        put(f.s_all, O.get(0), O.get(1), O.get(2), O.get(3));
    }
}

// The force's far part. Blocks share the (kx, ky) columns (x) and the atoms (y), one
// atom a thread. With P = F W^ (W^ the modes of W) and E = exp(i k.R_a),
//   S_a += (q_a/V) sum_k k (-Im[P E]),
// modes of kx > 0 counted twice. Along z, U = P(kz) + P(-kz) and V = i (P(kz) - P(-kz))
// turn a pair of modes into four products for sum P e^{i kz z} and four for its z slope
// (with U and V scaled by kz). In df64 as the structure factor; the columns' results
// are summed in FP64.
constexpr int kFarAt = 128;
constexpr int kFarKz = 32;                     // kz staged at a time

struct FarRow { cdf u, v, zu, zv; };           // U, V, kz U, kz V

__global__ void __launch_bounds__(kFarAt) k_far_force(int n, GammaFar f, const GAtom* ga, double* S) {
    __shared__ FarRow row[2][kFarKz];          // [0] of the lower atoms' W, [1] of the others'
    const int a = blockIdx.y * kFarAt + threadIdx.x, ncol = (f.mx + 1) * (2 * f.my + 1);
    const bool have = a < n;
    const int set = have && f.up && ga[a].kzl > 0 ? 0 : 1;
    const int cols = 2 * f.my + 1, pitch = f.mx + 1;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    auto split = [](double re, double im) {
        const float2 a = split_to_float2(re), b = split_to_float2(im);
        return cdf{{a.x, a.y}, {b.x, b.y}};
    };
    for (int col = blockIdx.x; col < ncol; col += gridDim.x) {
        const int kx = col % pitch, jy = col / pitch, ky = jy - f.my;
        const double gx = kx * f.bx, gy = ky * f.by, kk = gx * gx + gy * gy;
        if (kk > f.K * f.K) continue;
        const int mend = min(f.mz, (int)(sqrt(f.K * f.K - kk) / f.bz));      // the column inside the sphere
        Acc4 A;                                // T0.re, T0.im, X.re, X.im
        for (int m0 = 0; m0 <= mend; m0 += kFarKz) {
            const int nm = min(kFarKz, mend + 1 - m0);
            __syncthreads();
            for (int q = threadIdx.x; q < nm; q += kFarAt) {
                const int m = m0 + q;
                const double gz = m * f.bz;
                const double w = far_transform(f, sqrt(kk + gz * gz));
                auto at = [&](const double2* A, int mm) { return A[((long)(f.mz + mm) * cols + jy) * pitch + kx]; };
                double2 p = at(f.s_all, m), r = at(f.s_all, -m);
                auto put = [&](int s, double2 p, double2 r) {
                    if (m == 0) r = make_double2(0.0, 0.0);
                    const double ur = w * (p.x + r.x), ui = w * (p.y + r.y), vr = -w * (p.y - r.y), vi = w * (p.x - r.x);
                    row[s][q] = {split(ur, ui), split(vr, vi), split(gz * ur, gz * ui), split(-gz * vr, -gz * vi)};
                };
                if (f.up) {
                    put(0, p, r);
                    const double2 pu = at(f.s_up, m), ru = at(f.s_up, -m);
                    p.x += pu.x; p.y += pu.y; r.x += ru.x; r.y += ru.y;
                }
                put(1, p, r);
            }
            __syncthreads();
            if (!have) continue;
            for (int q = 0; q < nm; ++q) {
                const cdf z = as_cdf(__ldg(f.ezt + (long)(m0 + q) * n + a));
                const FarRow& r = row[set][q];
                df_acc_norm(A.s[0], A.c[0], z.re, r.u.re);
                df_acc_norm(A.s[0], A.c[0], z.im, r.v.re);
                df_acc_norm(A.s[1], A.c[1], z.re, r.u.im);
                df_acc_norm(A.s[1], A.c[1], z.im, r.v.im);
                df_acc_norm(A.s[2], A.c[2], z.im, r.zu.re);       // X = sum kz (sin U - cos V)
                df_acc_norm(A.s[2], A.c[2], z.re, r.zv.re);
                df_acc_norm(A.s[3], A.c[3], z.im, r.zu.im);
                df_acc_norm(A.s[3], A.c[3], z.re, r.zv.im);
            }
        }
        if (!have) continue;
        const cdf e = xy_phase(f, a, kx, ky);
        auto pair = [&](int i) { return df_quick(A.s[i], A.c[i]); };
        const df im = df_add(df_mul(e.re, pair(1)), df_mul(e.im, pair(0)));          // Im[E sum P e^{ikz z}]
        const df sl = df_add(df_mul(e.re, pair(2)), df_neg(df_mul(e.im, pair(3))));  // the slope is i E X
        const double two = kx > 0 ? 2.0 : 1.0, imd = two * df_to(im);
        fx -= gx * imd;
        fy -= gy * imd;
        fz -= two * df_to(sl);
    }
    if (!have) return;
    const double q = ((double)ga[a].a.x + (double)ga[a].a.y) * f.inv_v;
    atomicAdd(&S[3 * a + 0], q * fx);
    atomicAdd(&S[3 * a + 1], q * fy);
    atomicAdd(&S[3 * a + 2], q * fz);
}

template <typename T>
T* take(char*& p, size_t n) {
    T* r = reinterpret_cast<T*>(p);
    p += (n * sizeof(T) + 255) / 256 * 256;
    return r;
}

}  // namespace

// p null: only the size
static size_t far_layout(char* p, int n_atoms, GammaFar& f, const Geo& g) {
    char* const p0 = p;
    const size_t n = (size_t)(n_atoms > 0 ? n_atoms : 1), nx = f.mx + 1, ny = f.my + 1, nz = f.mz + 1;
    const size_t modes = (2 * nz - 1) * (2 * ny - 1) * nx, work = nx * g.ny * g.nz;
    f.ftab = take<double>(p, kFarIv * (kFarDeg + 1));
    f.ntab = take<float4>(p, kNearVec * kNearIv);
    f.htab = take<float4>(p, kNearVec * kNearIv);
    f.kz = take<int>(p, 2);
    f.ex = take<float4>(p, n * nx);
    f.ey = take<float4>(p, n * ny);
    f.ez = take<float4>(p, n * nz);
    f.ezt = take<float4>(p, n * nz);
    f.s_all = take<double2>(p, modes);
    f.c_all = take<double2>(p, work);
    f.s_up = f.c_up = nullptr;
    if (f.up) {
        f.s_up = take<double2>(p, modes);
        f.c_up = take<double2>(p, work);
    }
    return (size_t)(p - p0);
}

size_t gamma_far_bytes(int n_atoms, const GammaFar& f, const Geo& g) {
    GammaFar t = f;
    return far_layout(nullptr, n_atoms, t, g);
}

void gamma_far_view(void* base, int n_atoms, GammaFar& f, const Geo& g) {
    far_layout(static_cast<char*>(base), n_atoms, f, g);
}

void launch_gamma_far_consts(const GammaFar& f, cudaStream_t s) {
    k_far_ftab<<<kFarIv, 32 * (kFarDeg + 1), 0, s>>>(f);
    k_near_tabs<<<2 * kNearIv, 32, 0, s>>>(f);
}

void launch_gamma_far_modes(const Geo& g, Atoms at, const GammaFar& f, const GAtom* ga, cudaStream_t s) {
    if (f.up) k_far_split<<<1, 256, 0, s>>>(at.n, g.nz, ga, f.kz);
    const long total = (long)at.n * (f.mx + f.my + f.mz + 3);
    k_far_phases<<<(int)((total + 127) / 128 < 152L * 16 ? (total + 127) / 128 : 152L * 16), 128, 0, s>>>(g, at, f);
    const int threads = (f.mz + 1 + 31) / 32 * 32;
    k_far_modes<<<(f.mx + 1) * (2 * f.my + 1), threads, 0, s>>>(at.n, f, ga);
}

void launch_gamma_far_force(const Geo& g, int n_atoms, const GammaFar& f, const GAtom* ga, double* S, cudaStream_t s) {
    const int ay = (n_atoms + kFarAt - 1) / kFarAt, ncol = (f.mx + 1) * (2 * f.my + 1);
    // four blocks per SM share the columns; each ends in three FP64 atomics an atom
    const int bx = ncol < 608 / ay + 1 ? ncol : 608 / ay + 1;
    k_far_force<<<dim3(bx, ay), kFarAt, 0, s>>>(n_atoms, f, ga, S);
}

}  // namespace gp
