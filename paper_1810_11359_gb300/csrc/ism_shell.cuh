// ism_shell.cuh -- enumeration of the images of one RIR whose delay falls in a
// spherical shell around the receiver (Section 2.1, eq. (1)-(3)), shared by the
// fused Chebyshev accumulation and the fused direct form (forward) and the fused
// Chebyshev adjoint.
//
// The image coordinates along one axis increase with the index n (eq. (1)):
// X(2m) = 2 m L + x_s and X(2m - 1) = 2 m L - x_s.  So for a grid column
// (ix, iy) the images whose distance falls in the shell [s_lo, s_hi) form at
// most two index intervals in z (below and above the receiver), found in
// closed form from the source and receiver coordinates, and the columns that
// reach the shell form one interval in iy per row ix.  A CTA's warps take the
// columns 32 at a time, compute each column's intervals and a warp prefix of
// their lengths, and process the column candidates 32 at a time (a
// candidate's column from one bit per candidate that begins a column).
// Intervals are widened by SHELL_MARGIN sample; each candidate's exact delay
// (the per-axis tables hold the squared offsets as pairs of FP32) decides
// whether it belongs to the caller's range of integer delays, so every image
// lands in exactly one shell.  Candidate j of a warp's column chunk is always
// handled by lane j % 32, so the order in which a lane sees its images is a
// function of the geometry alone.
//
// What a candidate costs in instructions and shared-memory wavefronts bounds the
// kernels that walk (the Chebyshev form: the shared-memory pipe, 79 % of its peak;
// the others: issue), so the delay arithmetic and the column lookup are kept short.
// Binary search, two-sums and one 16-byte record of everything -> start bits, split
// offsets (ShellTab) and 24 bytes a candidate: accumulation of 128 RIRs (6 x 5 x 3 m,
// T60 0.6 s, 16 kHz) 413 -> 369 us, of 64 in FP16X2 596 -> 555 us, of 512 at 48 kHz
// 223 -> 215 us, the adjoint of 256 rooms 291 -> 255 us.
#pragma once

#include "ism_device.cuh"

#define SHELL_MARGIN 0.05f   // candidate margin (samples)

// Smallest image index n of an axis with coordinate X(n) >= Z.
__device__ __forceinline__ int ax_first(float Z, float xs, float inv2L)
{
    Z = fminf(fmaxf(Z, -1e7f), 1e7f);
    const int me = (int)ceilf((Z - xs) * inv2L);
    const int mo = (int)ceilf((Z + xs) * inv2L);
    return min(2 * me, 2 * mo - 1);
}

struct ShellAxis {
    float xs, xr, inv2L;   // source, receiver coordinate; 1 / (2 L)
    int nlo, N;
};

// Index interval [i0, i1) (0-based, clamped to the grid) of the images of an
// axis with X(n) - x_r in [D_lo, D_hi) (metres).
__device__ __forceinline__ void ax_range(const ShellAxis& a, float Dlo, float Dhi, int* i0, int* i1)
{
    const int n0 = ax_first(a.xr + Dlo, a.xs, a.inv2L);
    const int n1 = ax_first(a.xr + Dhi, a.xs, a.inv2L);
    *i0 = min(max(n0 - a.nlo, 0), a.N);
    *i1 = min(max(n1 - a.nlo, 0), a.N);
}

// CTA g of a fused launch -> (job, RIR, shell).  When the jobs' shell counts
// are alike the CTAs are ordered by the shell's rank from the outside over all
// fused RIRs of the launch set: every RIR's outermost (densest, since the
// images per delay grow as s^2) shell first, so the lightest shells fill the
// end of the launch; false for a CTA past its job's shells.  Otherwise they go
// job by job, RIR by RIR, densest shell first.
__device__ __forceinline__ bool shell_cta(const JobTable& t, long long g, int* jid, int* r, int* grp)
{
    if (!t.shell_rank_major) {
        const int j = ism_find_job(t, g, [](const JobDev& d) { return d.shell_cta_base; });
        const long long local = g - t.j[j].shell_cta_base;
        *jid = j;
        *r = (int)(local / t.j[j].shell_groups);
        *grp = t.j[j].shell_groups - 1 - (int)(local % t.j[j].shell_groups);
        return true;
    }
    const long long k = g / t.shell_rirs;   // rank from the outside
    const long long rr = g - k * t.shell_rirs;
    const int j = ism_find_job(t, rr, [](const JobDev& d) { return d.shell_rir_base; });
    *jid = j;
    *r = (int)(rr - t.j[j].shell_rir_base);
    *grp = t.j[j].shell_groups - 1 - (int)k;
    return *grp >= 0;
}

// What a CTA needs to walk the shell [b_lo, b_hi) of integer delays of RIR r.
struct Shell {
    ShellAxis ax[3];
    float kinv;            // c / f_s: metres per sample
    float s_lo2, s_hi2;    // squared shell bounds (samples^2), widened by the margin
    int b_lo;              // integer delays owned: [b_lo, b_lo + span)
    unsigned span;
    float sd2;             // squared delay of the direct path (samples^2)
    int Nx, Ny;
    bool valid;            // false: the pair lies outside the room (+inf tables)
};

// The axis tables of an RIR as the fused kernels stage them in shared memory, three
// arrays over x, y, z indices: squared offsets, reflection products and signed
// offsets apart, so that a candidate loads 12 bytes of its z entry (3 conflict-free
// wavefronts a warp) and the signed offset only where a polar pattern or a gradient
// needs it.
//
// The squared offset is split as hi + lo with hi a multiple of G instead of an FP32
// value and its rounding error.  G is a power of two with 2^24 G above every squared
// delay of the RIR that a candidate can have (shell_s2_magic = 1.5 2^23 G), so the hi
// parts of the three axes add without rounding and a sum of two entries is two FADDs
// instead of a two-sum (ff_add: 10 operations).  Both subtractions are exact; what is lost
// are the low words of the lo parts, |lo| <= G / 2: a few 2^-25 G samples^2, or up to
// 2^-24 G / s samples of a delay s, at most 2^-24 sqrt(G) near s = sqrt(G); relative to the
// 2^-25 that f is rounded to it matters for the direct path of a long RIR.  Root mean squares
// over directions, samples, 0.2 to 0.4 m from the source at 16 / 48 kHz (rounding alone:
// 1.3e-8): G = 8 (11,300 samples) 1.5e-8 / 1.3e-8, 16 (16,000) 1.9e-8 / 1.4e-8, 32 (22,600)
// 3.1e-8 / 1.6e-8, 256 (64,000) 2.1e-7 / 7.6e-8, the largest 1.5e-7, 2.7e-7 and 1.3e-6 of G =
// 16, 32 and 256.  So jobs of more than ISM_SPLIT_SAMPLES samples (G > 16) keep the two-sum on
// the table as it is (SPLIT = false; by job, since two shells must find the same integer delay
// for an image at their border), 1 to 4 % slower (8 RIRs of 23,200 samples, 32 taps: 333 and
// 337 us, their adjoint 479 and 500; 64 of 24,000 at 48 kHz 175 and 178).
// The reduced tap arithmetics keep it at every length: a
// change in the fraction's last bit can move a 16-bit tap by its own, far larger,
// last bit.
struct ShellTab {
    float2* s2_;   // hi, lo
    float* F_;     // product of the reflection coefficients
    float* D_;     // signed offset, samples
    __device__ __forceinline__ float2 s2(int e) const { return s2_[e]; }
    __device__ __forceinline__ float F(int e) const { return F_[e]; }
    __device__ __forceinline__ float D(int e) const { return D_[e]; }
    __device__ __forceinline__ float4 all(int e) const { return make_float4(s2_[e].x, s2_[e].y, F_[e], D_[e]); }
    __device__ __forceinline__ void put(int e, float4 v) const { s2_[e] = make_float2(v.x, v.y); F_[e] = v.z; D_[e] = v.w; }
};

__device__ __forceinline__ ShellTab shell_tab(unsigned char* smem, int max_axis_sum)
{
    const int n = (max_axis_sum + 1) & ~1;
    float2* s2 = reinterpret_cast<float2*>(smem);
    float* F = reinterpret_cast<float*>(s2 + n);
    return {s2, F, F + n};
}

// (of FP32 forms)
__host__ __device__ inline bool shell_split(const JobDev& J) { return J.n_ism + J.H <= ISM_SPLIT_SAMPLES; }

__device__ __forceinline__ float shell_s2_magic(const JobDev& J)
{
    const float s = (float)(J.n_ism + J.H + 2);
    const int e = (__float_as_int(1.05f * s * s) >> 23) - 127 + 1;   // 2^e > 1.05 s^2
    return 12582912.0f * __int_as_float((e - 24 + 127) << 23);
}

template <bool SPLIT>
__device__ __forceinline__ void shell_stage(const ShellTab& T, int e, float4 v, float s2_magic)
{
    const float hi = __fsub_rn(__fadd_rn(v.x, s2_magic), s2_magic);
    T.put(e, SPLIT ? make_float4(hi, __fadd_rn(__fsub_rn(v.x, hi), v.y), v.z, v.w) : v);
}

__device__ __forceinline__ Shell shell_setup(const JobDev& J, const ShellTab& T, int r, int b_lo, int b_hi)
{
    Shell sh;
    const int i_src = r / J.n_rcv, i_rcv = r - (r / J.n_rcv) * J.n_rcv;
    sh.kinv = J.kinv;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        sh.ax[a].xs = J.pos_src[3 * i_src + a];
        sh.ax[a].xr = J.pos_rcv[3 * i_rcv + a];
        sh.ax[a].inv2L = J.inv2L[a];
        sh.ax[a].nlo = J.nlo[a];
        sh.ax[a].N = J.N[a];
    }
    sh.Nx = J.N[0];
    sh.Ny = J.N[1];
    const float2 dx = T.s2(-J.nlo[0]), dy = T.s2(J.N[0] - J.nlo[1]), dz = T.s2(J.N[0] + J.N[1] - J.nlo[2]);
    sh.sd2 = (dx.x + dy.x + dz.x) + (dx.y + dy.y + dz.y);
    sh.valid = sh.sd2 < 3.0e38f;   // +inf tables (NaN here): a pair outside the room (flagged by the geometry kernel)
    sh.b_lo = b_lo;
    sh.span = (unsigned)max(b_hi - b_lo, 0);
    const float s_lo = fmaxf((float)b_lo - SHELL_MARGIN, 0.0f);
    const float s_hi = (float)b_hi + SHELL_MARGIN;
    sh.s_lo2 = s_lo * s_lo;
    sh.s_hi2 = s_hi * s_hi;
    return sh;
}

// Columns that reach the shell: row ix takes the iy with |y - y_r| < D_y.
// rowpre[ix] = columns in rows 0 .. ix (inclusive prefix), rowy0[ix] = first
// iy of row ix.  Every thread of the CTA calls it; returns the column count.
__device__ __forceinline__ int shell_rows(const Shell& sh, const ShellTab& T, int* rowpre, int* rowy0)
{
    const int Nx = sh.Nx;
    for (int ix = threadIdx.x; ix < Nx; ix += blockDim.x) {
        int w = 0, y0 = 0;
        if (sh.valid) {
            const float rem = __fsub_rn(sh.s_hi2, __fadd_rn(T.s2(ix).x, T.s2(ix).y));
            if (rem > 0.0f) {
                const float Dy = __fadd_rn(__fmul_rn(sqrtf(rem), sh.kinv), 1e-3f);
                int y1;
                ax_range(sh.ax[1], -Dy, Dy, &y0, &y1);
                w = max(y1 - y0, 0);
            }
        }
        rowpre[ix] = w;
        rowy0[ix] = y0;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int carry = 0;
        for (int base = 0; base < Nx; base += 32) {
            const int i = base + lane;
            int v = i < Nx ? rowpre[i] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += n;
            }
            if (i < Nx) rowpre[i] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    return Nx > 0 ? rowpre[Nx - 1] : 0;
}

// Column cl of the shell (cl < n_cols): its candidate intervals in z and its
// record.  Returns the number of candidates; rec = {S_xy hi, S_xy lo, col_scale F_x
// F_y, 0}; zi = {first z index below, count below, first z index above, ix | iy << 16}.
template <bool SPLIT>
__device__ __forceinline__ int shell_column(const Shell& sh, const ShellTab& T, const int* rowpre, const int* rowy0,
                                            int cl, float col_scale, float4* rec, int4* zi)
{
    const int Nx = sh.Nx, Ny = sh.Ny;
    int lo = 0, hi = Nx - 1;   // row: first ix with rowpre[ix] > cl
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (rowpre[mid] > cl) hi = mid;
        else lo = mid + 1;
    }
    const int ix = lo;
    const int before = ix > 0 ? rowpre[ix - 1] : 0;
    const float4 tx = T.all(ix);
    const int iy = min(rowy0[ix] + (cl - before), Ny - 1);
    const float4 ty = T.all(Nx + iy);
    const float s_hi = __fadd_rn(tx.x, ty.x), s_lo = __fadd_rn(tx.y, ty.y);   // the first exact (ShellTab)
    const ff sxy = SPLIT ? ff{s_hi, s_lo} : ff_add(ff{tx.x, tx.y}, ff{ty.x, ty.y});
    const float sxy_p = SPLIT ? __fadd_rn(s_hi, s_lo) : s_hi;
    const float D1 =
        fmaxf(__fsub_rn(__fmul_rn(sqrtf(fmaxf(__fsub_rn(sh.s_lo2, sxy_p), 0.0f)), sh.kinv), 1e-3f), 0.0f);
    const float D2 = __fadd_rn(__fmul_rn(sqrtf(fmaxf(__fsub_rn(sh.s_hi2, sxy_p), 0.0f)), sh.kinv), 1e-3f);
    int d0 = 0, d1 = 0, u0 = 0, u1 = 0;
    if (sh.s_hi2 > sxy_p) {
        ax_range(sh.ax[2], -D2, -D1, &d0, &d1);   // below the receiver (closed-open in n)
        ax_range(sh.ax[2], D1, D2, &u0, &u1);     // above
        d1 = min(d1, u0);                         // disjoint, whatever the rounding
    }
    const int nd = max(d1 - d0, 0), nu = max(u1 - u0, 0);
    *rec = make_float4(sxy.hi, sxy.lo, tx.z * ty.z * col_scale, 0.0f);
    *zi = make_int4(d0, nd, max(u0, d0 + nd), ix | (iy << 16));
    return nd + nu;
}

// Candidates of a warp's chunk of columns are numbered column by column, at most
// SHELL_MAX at a time.  The column of a candidate comes from one bit per candidate, set
// at the first of every column: a population count instead of a binary search over the
// prefix of the counts (5 dependent shared loads and ~20 instructions a candidate).
#define SHELL_MW 32                       // words of column-start bits per warp
#define SHELL_MAX (32 * SHELL_MW - 1)     // ISM_MAX_AXIS fits: a column is never cut
static_assert(ISM_MAX_AXIS <= SHELL_MAX, "a column's candidates fit one pass");

// Candidate j of a pass, in the column of record cf: its delay; true if its integer
// delay b lies in the shell, with bl = b - b_lo, f = the fractional part in [0, 1],
// rs = 1 / s, ez = the index of its z entry in the tables.  ci = {the column's first
// candidate above the receiver, z entry of candidate 0 below it}, cf.w = the z indices
// skipped between the two intervals.
//
// s^2 = hi + lo (ShellTab); r = s^2 rsqrt(s^2) is s to a few ulp, and one Newton
// correction from the exact residual hi - r^2 (FMA) + lo gives s = r + corr to ~2^-44
// relative.  b is floor(r) moved by the floor of the corrected fraction; both floors
// are additions of 1.5 2^23 rounded down, whose bits hold the integer (no conversion
// unit).  b and f depend on the image and its job's length, never on the shell, so every
// image lands in exactly one shell.
template <bool SPLIT>
__device__ __forceinline__ bool shell_delay(const Shell& sh, const ShellTab& T, const float4& cf, int2 ci, int j,
                                            int* bl_out, float* f_out, float* rs_out, int* ez_out, float4* tz_out)
{
    const float M = 12582912.0f;   // 1.5 2^23
    const int ez = j + ci.y + (j < ci.x ? 0 : __float_as_int(cf.w));
    const float4 tz = T.all(ez);
    *ez_out = ez;
    *tz_out = tz;
    if (!SPLIT) {
        const ff sq = ff_sqrt(ff_add(ff{cf.x, cf.y}, ff{tz.x, tz.y}));
        float bf = floorf(sq.hi);
        float f = __fadd_rn(__fsub_rn(sq.hi, bf), sq.lo);
        const bool neg = f < 0.0f;   // bring f into [0, 1) (see ism_delay)
        f = neg ? __fadd_rn(f, 1.0f) : f;
        bf = neg ? bf - 1.0f : bf;
        const bool one = f >= 1.0f;
        *f_out = one ? __fsub_rn(f, 1.0f) : f;
        *rs_out = ism_rcp(sq.hi);
        *bl_out = ism_int_of_integral(one ? bf + 1.0f : bf) - sh.b_lo;
        return (unsigned)*bl_out < sh.span;
    }
    const float hi = __fadd_rn(cf.x, tz.x), lo = __fadd_rn(cf.y, tz.y);
    const float s2 = __fadd_rn(hi, lo);
    const float rs = ism_rsqrt(s2);
    const float r = __fmul_rn(s2, rs);
    const float res = __fadd_rn(__fmaf_rn(-r, r, hi), lo);
    const float t = __fadd_rd(r, M);
    const float f0 = __fmaf_rn(__fmul_rn(res, 0.5f), rs, __fsub_rn(r, __fsub_rn(t, M)));
    const float t1 = __fadd_rd(f0, M);   // 1.5 2^23 - 1, + 0 or + 1
    const int bl = (__float_as_int(t) - 0x4B400000) + (__float_as_int(t1) - 0x4B400000) - sh.b_lo;
    *bl_out = bl;
    *f_out = __fsub_rn(f0, __fsub_rn(t1, M));
    *rs_out = rs;
    return (unsigned)bl < sh.span;
}

// The pass over the columns c0 .. c0 + 31 of a warp that begins at candidate `base` of
// theirs (0 but for very flat rooms, whose columns are found again for every pass rather
// than kept in registers): writes the records of its columns (Wf, Wi; extra(k, ixy)
// writes what else the caller keeps of the k-th of them) and their start bits (Wm).
// Returns its candidates and *total, those of all 32 columns; *start, *cnt, *k: the
// lane's column in the pass (cnt = 0: none).
template <bool SPLIT, class X>
__device__ __forceinline__ int shell_pass(const Shell& sh, const ShellTab& T, const int* rowpre, const int* rowy0,
                                          int n_cols, int c0, int base, float col_scale, float4* Wf, int2* Wi,
                                          unsigned* Wm, int lane, int* total, int* start, int* cnt, int* k_out,
                                          X&& extra)
{
    float4 rec = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int4 zi = make_int4(0, 0, 0, 0);
    const int cl = c0 + lane;
    int n = cl < n_cols ? shell_column<SPLIT>(sh, T, rowpre, rowy0, cl, col_scale, &rec, &zi) : 0;
    int inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    *total = __shfl_sync(0xffffffffu, inc, 31);
    const int s = inc - n - base;
    const bool in = n > 0 && s >= 0 && inc - base <= SHELL_MAX;
    const unsigned held = __ballot_sync(0xffffffffu, in);   // (a run of columns, in order)
    const int k = __popc(held & ((1u << lane) - 1u));
    Wm[lane] = 0;
    if (in) {
        Wf[k] = make_float4(rec.x, rec.y, rec.z, __int_as_float(zi.z - zi.x - zi.y));
        Wi[k] = make_int2(s + zi.y, sh.Nx + sh.Ny + zi.x - s);
        extra(k, zi.w);
    }
    __syncwarp();
    if (in) atomicOr(Wm + (s >> 5), 1u << (s & 31));
    *start = s;
    *cnt = in ? n : 0;
    *k_out = k;
    return *total <= SHELL_MAX ? *total - base : held ? __shfl_sync(0xffffffffu, inc, 31 - __clz(held)) - base : 0;
}

// The images of the shell, for the calling warp's share of the columns
// (chunks c0 = warp * 32 + k * 32 WARPS).  For each image with integer delay
// b_lo + bl in the shell lane calls
//   on_image(bl, f, rs, cf, o, ez, tz)
// with f = the fractional part of its delay s in [0, 1], rs = 1 / s, cf = its
// column's record (cf.z = col_scale F_x F_y), o = the record's place, where
// extra(o, ix | iy << 16) was called before, ez, tz = its z entry in the tables.  Wf, Wi:
// the warp's 32-entry scratch in shared memory; Wm: its SHELL_MW words.
template <int WARPS, bool SPLIT, class X, class F>
__device__ __forceinline__ void shell_walk(const Shell& sh, const ShellTab& T, const int* rowpre, const int* rowy0,
                                           int n_cols, float col_scale, float4* Wf, int2* Wi, unsigned* Wm, int warp, int lane,
                                           X&& extra, F&& on_image)
{
    const unsigned le = 0xffffffffu >> (31 - lane);
    for (int c0 = warp * 32; c0 < n_cols; c0 += WARPS * 32) {
        int total, base = 0;
        do {   // (one pass but for very flat rooms)
            int start, cnt, k;
            const int n = shell_pass<SPLIT>(sh, T, rowpre, rowy0, n_cols, c0, base, col_scale, Wf, Wi, Wm, lane, &total,
                                           &start, &cnt, &k, extra);
            __syncwarp();
            int cols = -1;   // last column begun before the batch
            for (int j0 = 0; j0 < n; j0 += 32) {
                const int j = j0 + lane;
                const unsigned m = Wm[j0 >> 5];
                const int o = cols + __popc(m & le);
                cols += __popc(m);
                if (j < n) {
                    const float4 cf = Wf[o];
                    int bl, ez;
                    float f, rs;
                    float4 tz;
                    if (shell_delay<SPLIT>(sh, T, cf, Wi[o], j, &bl, &f, &rs, &ez, &tz))
                        on_image(bl, f, rs, cf, o, ez, tz);
                }
            }
            __syncwarp();   // the records are read before the next pass overwrites them
            base += n;
        } while (base < total);
    }
}

// The images of the shell for the whole CTA.  The candidates of every chunk of
// WARPS x 32 columns form batches of 32 (candidate c by lane c mod 32), and
// warp w takes the chunk's batches w, w + WARPS, ..: the warps differ by at
// most one batch per chunk, and only the chunk's last batch is partial.  For
// every batch the warp's 32 lanes call, converged,
//   on_lane(has, bl, f, rs, cf, o, ez, tz)
// has = the lane's candidate is an image of the shell (the other arguments are
// unspecified when it is not); the arguments and extra(o, ixy) are those of
// shell_walk, o counted over the CTA.  Which warp and lane meet an image, and in
// which order, is a function of the geometry alone.  Every thread of the CTA
// calls it.  Wf, Wi: [WARPS x 32] column records; Wm: [WARPS][SHELL_MW] column starts, Wb:
// the same shape, the column that holds each word's first candidate; wtot: [WARPS].
template <int WARPS, bool SPLIT, class X, class F>
__device__ __forceinline__ void shell_walk_cta(const Shell& sh, const ShellTab& T, const int* rowpre, const int* rowy0,
                                               int n_cols, float col_scale, float4* Wf, int2* Wi, unsigned* Wm,
                                               unsigned char* Wb, int* wtot, int warp, int lane, X&& extra,
                                               F&& on_lane)
{
    unsigned char* wb = Wb + warp * SHELL_MW;
    for (int c0 = 0; c0 < n_cols; c0 += WARPS * 32) {
        int base = 0;
        bool more = true;
        while (more) {   // (one pass but for very flat rooms)
            int total, start, cnt, k;
            const int n = shell_pass<SPLIT>(sh, T, rowpre, rowy0, n_cols, c0 + warp * 32, base, col_scale,
                                            Wf + warp * 32, Wi + warp * 32, Wm + warp * SHELL_MW, lane, &total, &start,
                                            &cnt, &k, [&](int kk, int ixy) { extra(warp * 32 + kk, ixy); });
            if (cnt > 0)
                for (int w = (start + 31) >> 5; 32 * w < start + cnt; ++w) wb[w] = (unsigned char)k;
            base += n;
            if (lane == 0) wtot[warp] = n | (base < total ? 0x10000 : 0);
            __syncthreads();
            int off[WARPS + 1];   // exclusive prefix of the warps' candidates in the pass
            off[0] = 0;
            more = false;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                const int v = wtot[w];
                off[w + 1] = off[w] + (v & 0xffff);
                more |= v > 0xffff;
            }
            const int n_batches = (off[WARPS] + 31) >> 5;
            for (int bt = warp; bt < n_batches; bt += WARPS) {   // warp-uniform
                const int cc = bt * 32 + lane;
                bool has = false;
                int bl = 0, o = 0, ez = 0;
                float f = 0.0f, rs = 1.0f;
                float4 cf = make_float4(0.0f, 0.0f, 0.0f, 0.0f), tz = cf;
                if (cc < off[WARPS]) {
                    int wbk = 0, wo = 0;   // the warp whose columns hold candidate cc: the last w with off[w] <= cc
#pragma unroll
                    for (int w = 1; w < WARPS; ++w)   // (never an empty block: off[wbk + 1] > cc)
                        if (off[w] <= cc) {
                            wbk = w;
                            wo = off[w];
                        }
                    const int j = cc - wo, wd = wbk * SHELL_MW + (j >> 5);
                    o = wbk * 32 + Wb[wd] + __popc(Wm[wd] & 0xfffffffeu & (0xffffffffu >> (31 - (j & 31))));
                    cf = Wf[o];
                    has = shell_delay<SPLIT>(sh, T, cf, Wi[o], j, &bl, &f, &rs, &ez, &tz);
                }
                on_lane(has, bl, f, rs, cf, o, ez, tz);
            }
            __syncthreads();   // the records are read before the next pass overwrites them
        }
    }
}
