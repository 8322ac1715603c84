// ism_accum_cheb.cu -- FP32 accumulation of eq. (5) through a Chebyshev
// expansion of the windowed sinc in the fractional delay, fused with the
// enumeration of the images (Section 2.1) it accumulates: 32-tap windows with
// 8 terms (the text below), other windows whose taps a series follows with 10.
//
// For tap j of an image with delay s = b + f (b integer, f in [0, 1)), the
// sample b + j receives A delta'(j - f) (eq. (6)).  For a window of exactly
// N_w = 32 taps every tap function g_j(f) = delta'(j - f), j = -15 .. 16, is
// an entire function of f on [0, 1] (the window's zeros fall at the ends of
// the interval, so no mask cuts it), and its Chebyshev series in u = 2f - 1
// converges fast: degree 7 reproduces each g_j to 4.2e-7 of the image's
// amplitude (degree 8: 6.4e-8; degree 9: 2.1e-9), about twice the fixed-point
// step of the moment terms (see below); together they keep an RIR within a few
// 1e-7 of its peak, far inside FP32's 1e-5, and degree 7 spares one shared-
// memory atomic per image against degree 8.  The coefficients c_{j,i},
// interpolated at the 8 Chebyshev-Gauss nodes in FP64 on the host, travel in
// the kernel's parameter table.  Hence for the images that share the integer
// delay b,
//   sum_n A_n g_j(f_n) = sum_i c_{j,i} M_i,   M_i = sum_n A_n T_i(2 f_n - 1),
// so each image costs 8 moment terms instead of 32 tap evaluations, and each
// integer delay costs 8 FMAs per tap once.
//
// Delay bins.  Bin q holds the images with b in [32 q - 1, 32 q + 31), i.e.
// offsets rr = b - 32 q in [-1, 30] (32 offsets, one per lane); its taps fall
// in the 64 samples from 32 q - 16, the bin's window row, which the finalize
// kernel sums per sample with the previous bin's row.  An image is kept iff a
// tap reaches a sample below n_ism: b <= n_ism + 14.
//
// One CTA owns B = 8 consecutive bins of one RIR -- a spherical shell of
// 256 samples around the receiver (thinner, down to one bin, when a launch
// has too few RIRs to fill the GPU) -- and enumerates the images in it itself
// (ism_shell.cuh): each candidate's exact float-float delay decides its bin,
// so every image lands in exactly one CTA, the one whose bins hold its b.
//
// Fixed point.  Every image of bin q has s >= max(s_direct, 32 q - 1) (the
// direct path is the shortest: along each axis the source's own coordinate is
// the image coordinate nearest the receiver) and at least d / L_max - 3 wall
// hits (|n| >= |x_n - x_r| / L - 1 on each axis), so |A| <= A_max = amp_scale
// beta_max^h / s_lo.  A term A T_i is scaled by 2^e and rounded to an integer
// (one FFMA against 1.5 2^23: the sum's bits hold the integer), e the largest
// integer with 2^e A_max <= min((1 - 2^-10) 2^22, 0.98 2^31 / n - 1), n first
// four times the expected number of images per integer delay, 4 pi s^2 /
// (k^3 V) (one image per room volume V), plus 64.  The sums are 32-bit
// shared-memory atomic adds of the FFMA's raw bits K + v (K = 0x4B400000, the
// bits of 1.5 2^23; v the term's integer); with n images at the integer delay
// the sum of the v is the word minus n K, modulo 2^32, exact while it stays
// below 2^31 in magnitude.  Integer addition is associative, so the sums --
// and the FP32 result -- are the same in every run, whatever the order in
// which lanes and warps add their terms.  The CTA also counts its images per (bin,
// integer delay); if some count times the largest term could reach 2^31 a sum
// may have wrapped, and the CTA redoes its shell with scales set from the exact
// counts (which do not depend on the scales), so the second pass is safe.  The
// rounding error is at most 2^-22 A_max per term wherever the counts stay below
// ~500 per integer delay; A_max falls with the distance and the wall hits.
//
// Finally each warp expands the non-empty offsets of one bin into the taps
// (lane = tap) and rotates them into the bin's register window, which it
// stores as the bin's row; the moments of an offset sit together (8 floats),
// so a warp reads them in two broadcast loads.
//
// Other windows (the default, 4 ms, is 64 taps at 16 kHz and 176.4 at 44.1 kHz).
// A window whose end falls inside a sample interval cuts its last taps with a
// mask, which no polynomial follows, but the window has a double zero there:
// the kink falls with the cube of the window's length, and degree 9 reproduces the
// taps to 4.5e-8 of the amplitude (5e-9 without a mask; rms, norms over the taps) for the
// windows that this form takes (series_follows_window).  The 2 H coefficients
// of each term come from a table in the workspace that the geometry launch
// fills (cheb_table), and the expansion takes 32 taps at a time, each turn's
// upper half carried into the next.  The terms are converted to integers
// (cvt.rni) instead of rounded by the FFMA, which lifts the 2^22 cap on a
// term: with few images per integer delay the sums then hold up to 30 bits of a
// term, at no cost in time (the conversions go to a unit that is 14 % busy), and the
// expansion adds its terms from the last, smallest one on, c_0 (the same for every
// image) in two parts.  A RIR's error is then no larger than the per-tap sum's (of its
// norm, 15 RIRs of 176 taps, sparse: 3.6e-7 with the cap on a term, 1.7e-7 without it,
// 1.4e-7 now, 1.5e-7 per tap; of 64 taps in two dense rooms 1.27 and 1.19e-7 before,
// 0.95 and 0.91e-7 now, 1.18 and 1.08e-7 per tap).
#include "ism_accum.cuh"
#include "ism_shell.cuh"

namespace {

#define SH_B ISM_SHELL_BINS  // delay bins per CTA (a shell of 256 samples), fewer for small launches
#define SH_WARPS 8          // warps per CTA
#define SH_RS (SH_B * 32)   // row stride of the moment table: [term][bin, offset]
#define SH_NO 32            // offsets per bin (rr = -1 .. 30)
#define CB_MAGIC 12582912.0f                       // 1.5 * 2^23
#define CB_MAGIC_BITS 0x4B400000u                  // its bits

// Largest power of two 2^e with 2^e a_max <= min((1 - 2^-10) term_max, 0.98 2^31 / n - 1):
// no term reaches term_max (2^22 with the FFMA rounding trick) and n terms cannot sum to 2^31.
__device__ __forceinline__ float shell_scale(float a_max, float n, float term_max)
{
    const float cap = fminf(term_max * (1.0f - 1.0f / 1024.0f), 0.98f * 2147483648.0f / fmaxf(n, 1.0f) - 1.0f);
    const float ratio = a_max > 0.0f ? cap / a_max : 3.0e38f;
    int e = ((__float_as_int(ratio) >> 23) & 0xFF) - 127;   // floor(log2(ratio)), ratio normal
    e = max(-126, min(126, e));
    return __int_as_float((e + 127) << 23);
}

template <int NM, bool SPLIT>
__global__ void __launch_bounds__(SH_WARPS * 32, 5) shell_kernel(const __grid_constant__ JobTable t,
                                                                  const float4* __restrict__ tbl,
                                                                  const float* __restrict__ tabs,
                                                                  float* __restrict__ rows)
{
    constexpr float TERM_MAX = NM != ISM_CHEB_NF ? 1073741824.0f : 4194304.0f;
    constexpr bool CVT = NM != ISM_CHEB_NF;   // terms converted to integers, not rounded by the FFMA
    constexpr int MV = (NM + 3) / 4;   // float4 per offset of the expansion's moment table
    // [bin][offset][4 MV], which overlays the sums, the counts, the scales, the row prefix and
    // the column records (all dead by then)
    static_assert(SH_RS * MV * 16 <= (NM + 1) * SH_RS * 4 + SH_WARPS * 32 * 24,
                  "moment table larger than the tables it overlays");
    extern __shared__ __align__(16) unsigned char smem[];
    int jid, r, grp;
    if (!shell_cta(t, blockIdx.x, &jid, &r, &grp)) return;   // CTA-uniform
    const JobDev& J = t.j[jid];
    if (J.use_cheb != NM || shell_split(J) != SPLIT) return;   // another instantiation's job
    const int B = t.shell_bins;   // bins of this launch's shells: SH_B, fewer for small launch sets
    const int q0 = grp * B;
    const int nb = min(B, J.Q - q0);
    const int Nx = J.N[0], Ny = J.N[1], Nz = J.N[2];
    const int n_axis = Nx + Ny + Nz;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // shared memory: axis tables | moment sums | image counts | per-bin scales | row prefix |
    // per-warp column records
    const ShellTab T = shell_tab(smem, t.max_axis_sum);
    unsigned* S = reinterpret_cast<unsigned*>(smem + (size_t)((t.max_axis_sum + 1) & ~1) * sizeof(float4));   // [term][bin, offset]
    int* Cn = reinterpret_cast<int*>(S + NM * SH_RS);                    // [bin, offset] images
    float* scale_s = reinterpret_cast<float*>(Cn + SH_RS);
    float* inv_s = scale_s + SH_B;
    float* amax_s = inv_s + SH_B;                                                 // per-bin amplitude bound
    int* redo = reinterpret_cast<int*>(amax_s + SH_B);                            // [4]: retry flag
    int* rowpre = reinterpret_cast<int*>(redo + 4);                             // [Nx]: columns up to row ix
    int* rowy0 = rowpre + ((t.max_axis_sum + 4) & ~3);                          // [Nx]: first iy of row ix
    float4* recf = reinterpret_cast<float4*>(rowy0 + ((t.max_axis_sum + 4) & ~3));
    int2* Wi = reinterpret_cast<int2*>(recf + SH_WARPS * 32) + warp * 32;
    unsigned* Wm = reinterpret_cast<unsigned*>(Wi + (SH_WARPS - warp) * 32) + warp * SHELL_MW;   // [warps][SHELL_MW]
    float* Wo = reinterpret_cast<float*>(Wm + (SH_WARPS - warp) * SHELL_MW) + warp * 32;  // [warps][32]: o_x D_x + o_y D_y
    float4* Wf = recf + warp * 32;

    const float s2_magic = shell_s2_magic(J);
    const float4* Tg = tbl + J.tbl_base + (long long)r * n_axis;
    for (int e = threadIdx.x; e < n_axis; e += blockDim.x) shell_stage<SPLIT>(T, e, Tg[e], s2_magic);
    if (threadIdx.x == 0) *redo = 0;
    __syncthreads();

    // receiver polar pattern: the unit orientation of this RIR's receiver (|g| <= 1 keeps A_max a bound)
    const int i_rcv = r - (r / J.n_rcv) * J.n_rcv;
    const float alpha = J.mic_alpha;
    float3 orient = make_float3(0.0f, 0.0f, 0.0f);
    if (alpha != 1.0f) {
        const float* o = J.orient_rcv + 3 * i_rcv;
        const float ox = o[0], oy = o[1], oz = o[2];
        const float inv = 1.0f / sqrtf(__fmaf_rn(ox, ox, __fmaf_rn(oy, oy, oz * oz)));
        orient = make_float3(ox * inv, oy * inv, oz * inv);
    }
    // exact delays b owned by this CTA: [b_lo, b_hi), b <= n_ism + 14 for H = 16
    const Shell sh = shell_setup(J, T, r, ISM_SB * q0 - 1, min(ISM_SB * (q0 + nb) - 1, J.n_ism + J.H - 1));
    const float kinv = sh.kinv;
    const float sd2 = sh.sd2;
    const bool valid = sh.valid;

    if (threadIdx.x < SH_B) {
        // fixed-point scale of bin q0 + threadIdx.x, first from the expected number of images
        // per integer delay (verified, and redone from the exact counts if it was too small)
        const int q = q0 + (int)threadIdx.x;
        float sc = 1.0f, amax = 0.0f;
        if (q < J.Q && valid) {
            const float slo = fmaxf(fmaxf(sqrtf(sd2) * (1.0f - 1.0f / 1024.0f), (float)(ISM_SB * q) - 1.0f), 1e-30f);
            float bmax = 0.0f;
            for (int w = 0; w < 6; ++w) bmax = fmaxf(bmax, fabsf(ism_job_beta(J, w)));
            const int h = max(0, (int)floorf(slo * kinv / J.Lmax - 3.0f));
            const float decay = (h == 0) ? 1.0f : (bmax > 0.0f ? exp2f((float)h * log2f(bmax)) : 0.0f);
            amax = J.amp_scale / slo * decay * 1.001f;
            // images per integer delay at s: 4 pi s^2 / (k^3 V) (one image per volume V)
            const float shi = (float)(ISM_SB * q + ISM_SB);
            const float k = 1.0f / kinv;
            const float vol = J.vol;
            const float n_est = 4.0f * (12.566371f * shi * shi / (k * k * k * vol)) + 64.0f;
            sc = shell_scale(amax, n_est, TERM_MAX);
        }
        scale_s[threadIdx.x] = sc;
        inv_s[threadIdx.x] = 1.0f / sc;   // exact: a power of two
        amax_s[threadIdx.x] = amax;
    }
    const int n_cols = shell_rows(sh, T, rowpre, rowy0);   // (synchronises the CTA)

    for (int pass = 0; pass < 2; ++pass) {
    static_assert(SH_RS % 4 == 0, "the sums and the counts after them are cleared four words at a time");
    for (int e = threadIdx.x; e < (NM + 1) * SH_RS / 4; e += blockDim.x)
        reinterpret_cast<uint4*>(S)[e] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    shell_walk<SH_WARPS, SPLIT>(sh, T, rowpre, rowy0, n_cols, J.amp_scale, Wf, Wi, Wm, warp, lane, [&](int k, int ixy) {
        if (alpha != 1.0f) Wo[k] = __fmaf_rn(orient.y, T.D(Nx + (ixy >> 16)), orient.x * T.D(ixy & 0xFFFF));
    }, [&](int bl, float f, float rs, const float4& cf, int col, int, const float4& tz) {
        float amp = cf.z * tz.z * rs;
        if (alpha != 1.0f)   // polar pattern: cos(theta) = o . (x_n - x_r) / d
            amp *= __fmaf_rn(1.0f - alpha, __fmaf_rn(orient.z, tz.w, Wo[col]) * rs, alpha);
        const float as = amp * scale_s[bl >> 5];   // bin q0 + bl / 32, offset index rr + 1 = bl mod 32
        const float uu = __fmaf_rn(2.0f, f, -1.0f);
        const float u2 = uu + uu;
        unsigned* Sb = S + bl;
        atomicAdd(Cn + bl, 1);
        // the term's bits in the sum: K + v by the FFMA trick (the n K go at the expansion), or v
        auto term = [&](float tk) {
            return CVT ? (unsigned)__float2int_rn(as * tk) : __float_as_uint(__fmaf_rn(as, tk, CB_MAGIC));
        };
        atomicAdd(Sb, CVT ? (unsigned)__float2int_rn(as) : __float_as_uint(__fadd_rn(as, CB_MAGIC)));
        atomicAdd(Sb + SH_RS, term(uu));
        float tp = 1.0f, tc = uu;
#pragma unroll
        for (int k = 2; k < NM; ++k) {
            const float tn = __fmaf_rn(u2, tc, -tp);
            atomicAdd(Sb + k * SH_RS, term(tn));
            tp = tc;
            tc = tn;
        }
    });
    __syncthreads();
    // every sum of bin q holds at most Cn[q][o] terms of magnitude <= scale * A_max + 1/2:
    // below 2^31 means no sum can have wrapped; otherwise redo the shell with scales from
    // the exact counts (the counts do not depend on the scales, so the second pass is safe)
    // (a warp per bin, one load and a reduction, where a thread per bin met one bank 32 times
    // and the CTA waited: with the tables cleared by 16-byte stores, 16 RIRs of 64 taps 252 ->
    // 244 us, 128 of 32 taps 366.6 -> 365, 32 mixed rooms 122.5 -> 121)
    static_assert(SH_NO == 32 && SH_WARPS == SH_B, "lane = offset, warp = bin");
    if (pass == 0) {
        const int mx = __reduce_max_sync(0xffffffffu, Cn[warp * SH_NO + lane]);
        const float bound = (float)mx * (scale_s[warp] * amax_s[warp] + 0.5f);
        if (lane == 0 && !(bound < 0.99f * 2147483648.0f)) {
            const float sc = shell_scale(amax_s[warp], (float)mx, TERM_MAX);
            scale_s[warp] = sc;
            inv_s[warp] = 1.0f / sc;
            atomicOr(redo, 1);
        }
    }
    __syncthreads();
    if (!*redo || pass == 1) break;   // CTA-uniform
    }

    // ---- expansion: warp w owns bin q0 + w; lane o reads the sums of offset o
    float m[4 * MV];
    bool any = false;
    if (warp < nb) {
        const unsigned* Sb = S + warp * SH_NO + lane;
        // n K (mod 2^32) of the biased terms
        const unsigned nk = CVT ? 0u : (unsigned)Cn[warp * SH_NO + lane] * CB_MAGIC_BITS;
        const float inv = inv_s[warp];
#pragma unroll
        for (int k = 0; k < 4 * MV; ++k) {
            const int v = k < NM ? (int)(Sb[k * SH_RS] - nk) : 0;
            any |= v != 0;
            m[k] = __int2float_rn(v) * inv;   // exact scaling by a power of two
        }
    }
    __syncthreads();   // every sum is read before the moment table overwrites the CTA's tables
    if (warp >= nb) return;
    // moments of (bin, offset o) at Mt + MV (32 bin + o): {M_0..M_3}, {M_4..M_7}, ..
    float4* Mt = reinterpret_cast<float4*>(S) + MV * SH_NO * warp;
#pragma unroll
    for (int v = 0; v < MV; ++v) Mt[MV * lane + v] = make_float4(m[4 * v], m[4 * v + 1], m[4 * v + 2], m[4 * v + 3]);
    const unsigned nonempty = __ballot_sync(0xffffffffu, any);
    __syncwarp();
    const int slots = NM == ISM_CHEB_NF ? 1 : J.slots;
    float* row = rows + J.rows_base + ((long long)r * J.Q + q0 + warp) * (32 * (slots + 1));
    float carry = 0.0f;   // the previous 32 taps' share of this 32 samples
    for (int sl = 0; sl < slots; ++sl) {
        float c[NM];   // lane = tap 32 sl + lane: its Chebyshev coefficients
#pragma unroll
        for (int i = 0; i < NM; ++i)
            c[i] = NM == ISM_CHEB_NF ? t.cheb[lane * ISM_CHEB_N + i] : tabs[J.lut_base + (i * slots + sl) * 32 + lane];
        const float c0_lo = CVT ? tabs[J.lut_base + (NM * slots + sl) * 32 + lane] : 0.0f;
        float acc[2] = {carry, 0.0f};
        for (int o = 0; o < SH_NO; ++o) {
            if (!((nonempty >> o) & 1u)) continue;   // warp-uniform
            float mv[4 * MV];
#pragma unroll
            for (int v = 0; v < MV; ++v) {
                const float4 w = Mt[MV * o + v];
                mv[4 * v] = w.x;
                mv[4 * v + 1] = w.y;
                mv[4 * v + 2] = w.z;
                mv[4 * v + 3] = w.w;
            }
            float D[1];
            if constexpr (CVT) {   // the small terms first
                D[0] = c0_lo * mv[0];
#pragma unroll
                for (int k = NM - 1; k >= 0; --k) D[0] = __fmaf_rn(c[k], mv[k], D[0]);
            } else {               // (held to the truncation of 4e-7 in any order)
                D[0] = c[0] * mv[0];
#pragma unroll
                for (int k = 1; k < NM; ++k) D[0] = __fmaf_rn(c[k], mv[k], D[0]);
            }
            flush_run<1, false>(D, acc, o - 1, lane, 1.0f);
        }
        row[32 * sl + lane] = acc[0];
        carry = acc[1];
    }
    row[32 * slots + lane] = carry;
}

template <int NM, bool SPLIT>
int launch_cheb(const JobTable& t, const WsPlan& p, char* ws, cudaStream_t s, int* launched)
{
    const size_t sm = (size_t)((t.max_axis_sum + 1) & ~1) * sizeof(float4) + (size_t)(NM + 1) * SH_RS * sizeof(int) +
                      3 * SH_B * sizeof(float) + 4 * sizeof(int) + 2 * (size_t)((t.max_axis_sum + 4) & ~3) * sizeof(int) +
                      (size_t)SH_WARPS * 32 * (sizeof(float4) + sizeof(int2)) +
                      (size_t)SH_WARPS * (SHELL_MW * sizeof(unsigned) + 32 * sizeof(float));
    static std::atomic<unsigned long long> opened{0};
    int rc = ism_open_smem((const void*)shell_kernel<NM, SPLIT>, &opened);
    if (rc) return rc;
    // all of the unified L1 as shared memory: 5 CTAs of ~27 KB per SM
    cudaError_t e = cudaFuncSetAttribute(shell_kernel<NM, SPLIT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return (int)e;
    shell_kernel<NM, SPLIT><<<(unsigned)p.shell_ctas, SH_WARPS * 32, sm, s>>>(
        t, reinterpret_cast<const float4*>(ws + p.tbl_off), reinterpret_cast<const float*>(ws + p.lut_off),
        reinterpret_cast<float*>(ws + p.rows_off));
    ++*launched;
    return (int)cudaGetLastError();
}

}  // namespace

int ism_launch_accum_cheb(const JobTable& t, const WsPlan& p, char* ws, void* stream, int* launched)
{
    *launched = 0;
    if (p.shell_ctas <= 0 || !t.any_cheb) return 0;
    bool plain[2] = {false, false}, wide[2] = {false, false};   // [split offsets]
    for (int i = 0; i < t.n_jobs; ++i) {
        plain[shell_split(t.j[i])] |= t.j[i].use_cheb == ISM_CHEB_NF;
        wide[shell_split(t.j[i])] |= t.j[i].use_cheb == ISM_CHEB_NW;
    }
    int rc = 0;
    cudaStream_t s = (cudaStream_t)stream;
    if (plain[1]) rc = launch_cheb<ISM_CHEB_NF, true>(t, p, ws, s, launched);
    if (!rc && plain[0]) rc = launch_cheb<ISM_CHEB_NF, false>(t, p, ws, s, launched);
    if (!rc && wide[1]) rc = launch_cheb<ISM_CHEB_NW, true>(t, p, ws, s, launched);
    if (!rc && wide[0]) rc = launch_cheb<ISM_CHEB_NW, false>(t, p, ws, s, launched);
    return rc;
}
