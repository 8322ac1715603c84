// ism_geometry.cu -- per-RIR geometry tables and the FP64 Sabine helper.
//
// The image grid of Section 2.1 factorises per axis: the image of index n sits
// at n L + x_s (n even) or (n + 1) L - x_s (n odd) (eq. (1)), so its offset to
// the receiver along one axis depends on n alone, and the reflection product
// of eq. (4) is a product of one factor per axis.  This kernel tabulates, for
// every RIR and every index of every axis,
//   S[n] = ((x_n - x_r) f_s / c)^2   (squared offset in samples^2, FP64, stored
//                                     as a float-float pair hi + lo)
//   F[n] = beta_0^{e0(n)} beta_1^{e1(n)}  (wall hits along that axis)
//   D[n] = (x_n - x_r) f_s / c           (signed offset, FP32: the direction
//                                          of arrival for polar patterns)
// so that image (nx, ny, nz) has s^2 = Sx + Sy + Sz and weight Fx Fy Fz.  For
// the backward pass it also tabulates x_n - x_r (metres), dF/dbeta_0,
// dF/dbeta_1 (product form, valid at beta = 0) and d x_n / d x_s = +-1
// (even / odd n).  It
// also checks that source and receiver lie strictly inside the room (and that
// a patterned receiver has a non-zero orientation); a pair that does not gets
// S = +inf everywhere, i.e. no image survives.
//
// Bound: the chain of FP64 instructions of a CTA.  GB300 starts an FP64 warp instruction
// on a quarter of an SM every ~64 cycles, so each one of a chain costs that much, whether
// one lane or 32 need it.  Hence a CTA per RIR and axis (a launch of 1 to 50 RIRs leaves
// most SMs idle), each wall's powers once per CTA instead of two to six per image, the
// checks in FP32 (exact: the values are FP32) on one warp and f_s / c on another.  Under
// the profiler, per launch: one RIR 5.6 -> 4.1 us, 128 RIRs 9.5 -> 6.5, 51 rooms with the
// backward's tables 9.0 -> 5.6, one room of 64 taps with its coefficient tables 8.9 -> 7.7;
// 512 RIRs of few images per axis, bound by the CTAs' start, 10.3 as before.
#include <cmath>

#include "ism_device.cuh"

namespace {

__device__ double dpow_int(double b, int e)
{
    double r = 1.0;  // 0^0 = 1: the direct path keeps weight 1
    while (e > 0) {
        if (e & 1) r *= b;
        b *= b;
        e >>= 1;
    }
    return r;
}

// Chebyshev coefficients of 8 of the tap functions g_t(f) = delta'(t - H + 1 - f) (eq. (6))
// of a window of N_w taps, f = (u + 1) / 2: interpolated at the Chebyshev-Gauss nodes
// u_k = cos(pi (k + 1/2) / N), c_i = (2 / N) sum_k g_t(u_k) T_i(u_k), c_0 halved, in FP64.
// (8 taps per CTA spread the ~100 values a tap over the SMs; the chain of FP64 instructions
// is what takes the time, so the cosines of T_i and 1 / N are one warp's work meanwhile.)
__device__ void cheb_table(const JobDev& J, int N, int tap0, float* tab)
{
    __shared__ double gv[8][ISM_CHEB_MAX], cs[ISM_CHEB_MAX + 1], inv_s;   // g_t(u_k); cos(pi j / 2 N); 1 / N
    if (threadIdx.x >= 96) {   // the last warp, while the others evaluate the tap functions
        const int j = threadIdx.x - 96;
        if (j <= N) cs[j] = cospi(0.5 * j / N);
        if (j == 0) inv_s = 1.0 / N;
    } else {
        for (int e = threadIdx.x; e < 8 * N; e += 96) {
            const int k = e % N, t = tap0 + e / N;
            const double f = 0.5 * (cospi((k + 0.5) / N) + 1.0);
            const int j = t - J.H + 1;
            const double x = (double)j - f, Nw = (double)J.Nw;
            double v = 0.0;
            if (t < 2 * J.H && fabs(x) < 0.5 * Nw)   // sin(pi (j - f)) = (-1)^(j + 1) sin(pi f)
                v = 0.5 * (1.0 + cospi(2.0 * x / Nw)) * ((j & 1) ? 1.0 : -1.0) * sinpi(f) /
                    (3.141592653589793238462643383279502884 * x);
            gv[e / N][k] = v;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 8 * N; e += blockDim.x) {
        const int i = e / 8, t = tap0 + e % 8;
        double c = 0.0;
        for (int k = 0; k < N; ++k) {   // T_i(u_k) = cos(pi i (2 k + 1) / 2 N), folded into the first quarter
            int q = i * (2 * k + 1) % (4 * N);
            q = q > 2 * N ? 4 * N - q : q;
            c += gv[e % 8][k] * (q > N ? -cs[2 * N - q] : cs[q]);
        }
        c *= i == 0 ? inv_s : 2.0 * inv_s;
        tab[i * 32 * J.slots + t] = (float)c;
        if (i == 0) tab[N * 32 * J.slots + t] = (float)(c - (double)(float)c);   // the rest of c_0, after the terms
    }
}

__global__ void __launch_bounds__(128) geometry_kernel(const __grid_constant__ JobTable t, float4* tbl,
                                                       float4* dtbl, uint32_t* status, float* tabs, int n_rir)
{
    if ((int)blockIdx.x >= n_rir) {   // the coefficient tables: ISM_CHEB_TAB_CTAS CTAs each
        if (blockIdx.y > 0) return;
        const int k = ((int)blockIdx.x - n_rir) / ISM_CHEB_TAB_CTAS, c = ((int)blockIdx.x - n_rir) % ISM_CHEB_TAB_CTAS;
        for (int i = 0; i < t.n_jobs; ++i) {
            const JobDev& J = t.j[i];
            const int N = J.use_cheb > J.adj_cheb ? J.use_cheb : J.adj_cheb;
            if (N < ISM_CHEB_NW || J.lut_base != k * ISM_CHEB_TAB) continue;
            if (8 * c < 32 * J.slots) cheb_table(J, N, 8 * c, tabs + J.lut_base);
            return;
        }
        return;
    }
    const long long g = blockIdx.x;  // one CTA per RIR of the launch set and axis
    const int a = blockIdx.y;
    const int jid = ism_find_job(t, g, [](const JobDev& j) { return j.rir_base; });
    const JobDev& J = t.j[jid];
    const int r = (int)(g - J.rir_base);
    const int i_src = r / J.n_rcv, i_rcv = r % J.n_rcv;
    const float* ps = J.pos_src + 3 * i_src;
    const float* pr = J.pos_rcv + 3 * i_rcv;

    __shared__ int ok_s;
    __shared__ double k_s, pw[2][32], pw32[2];   // f_s / c; beta_w^0 .. beta_w^31 of the axis's walls, beta_w^32
    const double xs = (double)ps[a], xr = (double)pr[a];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 2) {
        double b = (double)ism_job_beta(J, 2 * a + warp), p = 1.0;   // 0^0 = 1: the direct path keeps weight 1
        for (int i = 0; i < 5 && 4 << i <= J.N[a] + 4; ++i, b *= b)   // (exponents up to N / 4 + 1)
            if (lane >> i & 1) p *= b;
        pw[warp][lane] = p;
        if (lane == 0) pw32[warp] = b;
    } else if (warp == 2) {   // all in FP32, exactly: the coordinates and coefficients are FP32 values
        bool in = true, apart = false, dir = false, beta = true;
        if (lane < 3) {
            const float s = ps[lane], m = pr[lane];
            in = s > 0.0f && m > 0.0f && (double)fmaxf(s, m) < J.L[lane];   // (a NaN fails s > 0 or m > 0)
            apart = s != m;
            if (J.mic_alpha != 1.0f) {
                const float o = J.orient_rcv[3 * i_rcv + lane];
                in = in && fabsf(o) < __int_as_float(0x7f800000);
                dir = o != 0.0f;
            } else {
                dir = true;
            }
        }
        if (lane < 6 && J.beta_dev) beta = fabsf(ism_job_beta(J, lane)) <= 1.0f;   // (else checked on the host)
        const bool ok = __all_sync(~0u, in) && __any_sync(~0u, apart) && __any_sync(~0u, dir);
        beta = __all_sync(~0u, beta);
        if (lane == 0) {
            if (!beta) atomicOr(status, (uint32_t)ISM_DEVICE_FLAG_BETA);
            if (!ok) atomicOr(status, (uint32_t)ISM_DEVICE_FLAG_POSITION);
            ok_s = ok && beta;
        }
    } else if (lane == 0) {
        k_s = (double)J.fs / (double)J.c;
    }
    __syncthreads();

    const auto power = [&](int w, int e) {
        const double p = pw[w][e & 31];
        return e < 32 ? p : p * dpow_int(pw32[w], e >> 5);   // (an axis of more than 124 images)
    };
    const int n_axis = J.N[0] + J.N[1] + J.N[2];
    const double k = k_s, L = J.L[a];
    const long long first = J.tbl_base + (long long)r * n_axis + (a > 0 ? J.N[0] : 0) + (a > 1 ? J.N[1] : 0);
    for (int i = threadIdx.x; i < J.N[a]; i += blockDim.x) {
        int n = J.nlo[a] + i;
        bool even = (n % 2) == 0;
        // eq. (1): image coordinate minus receiver coordinate
        double m = even ? (double)n : (double)(n + 1);
        double off = (even ? xs : -xs) - xr;
        double u = (m * L + off) * k;
        double S = u * u;
        // eq. (4): hits of the near (x0) and far (x1) wall along this axis
        int an = n < 0 ? -n : n;
        int e0 = even ? an / 2 : (n - 1 < 0 ? 1 - n : n - 1) / 2;
        int e1 = even ? an / 2 : (n + 1 < 0 ? -(n + 1) : n + 1) / 2;
        const double f0 = power(0, e0), f1 = power(1, e1);
        double F = f0 * f1;
        float hi = (float)S;
        float lo = (float)(S - (double)hi);
        if (!ok_s) {
            hi = __int_as_float(0x7f800000);  // +inf: every image of this pair is culled
            lo = 0.0f;
            F = 0.0;
        }
        tbl[first + i] = make_float4(hi, lo, (float)F, (float)u);
        if (dtbl) {
            const double d0 = e0 > 0 ? (double)e0 * power(0, e0 - 1) * f1 : 0.0;
            const double d1 = e1 > 0 ? (double)e1 * f0 * power(1, e1 - 1) : 0.0;
            dtbl[first + i] = make_float4((float)(m * L + off), ok_s ? (float)d0 : 0.0f, ok_s ? (float)d1 : 0.0f,
                                          even ? 1.0f : -1.0f);
        }
    }
}

// Inverse of eq. (7) in FP64: alpha_i = w_i alpha_0, sum_i S_i alpha_i =
// 0.161 V / T60, beta_i = +-sqrt(1 - alpha_i).
__global__ void beta_sabine_kernel(const double* L, const double* T60, const double* w, int negative,
                                   int n, double* beta_out, int* status)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double Lx = L[3 * i], Ly = L[3 * i + 1], Lz = L[3 * i + 2];
    double S[6] = {Ly * Lz, Ly * Lz, Lx * Lz, Lx * Lz, Lx * Ly, Lx * Ly};
    double wt[6];
    double sw = 0.0;
    for (int k = 0; k < 6; ++k) {
        wt[k] = w ? w[k] : 1.0;
        sw += S[k] * wt[k];
    }
    int st = 0;
    double a0 = 0.0;
    if (!(sw > 0.0) || !(T60[i] > 0.0) || !(Lx > 0.0 && Ly > 0.0 && Lz > 0.0)) st = ISM_ERR_INFEASIBLE;
    else a0 = 0.161 * Lx * Ly * Lz / (T60[i] * sw);
    for (int k = 0; k < 6 && st == 0; ++k) {
        double a = wt[k] * a0;
        if (a >= 1.0 || a < 0.0) st = ISM_ERR_INFEASIBLE;
    }
    for (int k = 0; k < 6; ++k) {
        double b = st ? 0.0 : sqrt(1.0 - wt[k] * a0);
        beta_out[6 * i + k] = negative ? -b : b;
    }
    status[i] = st;
}

}  // namespace

int ism_launch_geometry(const JobTable& t, const WsPlan& p, char* ws, void* stream)
{
    long long n_rir = p.rir_total;
    if (n_rir <= 0) return 0;
    geometry_kernel<<<dim3((unsigned)(n_rir + ISM_CHEB_TAB_CTAS * p.cheb_tabs), 3), 128, 0, (cudaStream_t)stream>>>(
        t, reinterpret_cast<float4*>(ws + p.tbl_off), p.dtbl_off ? reinterpret_cast<float4*>(ws + p.dtbl_off) : nullptr,
        reinterpret_cast<uint32_t*>(ws + p.status_off), reinterpret_cast<float*>(ws + p.lut_off), (int)n_rir);
    return (int)cudaGetLastError();
}

int ism_launch_beta_sabine(const double* L, const double* T60, const double* w, int negative, int n,
                           double* beta_out, int* status, void* stream)
{
    if (n <= 0) return 0;
    beta_sabine_kernel<<<(n + 127) / 128, 128, 0, (cudaStream_t)stream>>>(L, T60, w, negative, n, beta_out,
                                                                          status);
    return (int)cudaGetLastError();
}
