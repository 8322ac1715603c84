// ism_auralize_ols.cu -- moving sources (Section 4) through the frequency
// domain with one short DFT length: overlap-save over blocks of the output.
//
// The four-step form (ism_auralize_fft.cu) transforms every RIR at a length of
// 2^ceil(log2(n_x + n_S - 1)): more than twice the RIR's own length, in two
// passes over device memory, and its shared-memory stages are bound by issue.
// Where the segments of the signal are short -- many trajectory points -- a block
// of V output samples needs, of segment x_p (at most Lb samples from sample s0),
// only the RIR samples h[T0 - s0 - (Lb - 1) .. T0 - s0 + V - 1], so with
// V + Lb - 1 = N = 4096
//   y_m[T0 + v] = sum_p IDFT(X_p . DFT(h_{p,m}[T0 - s0 - (Lb - 1) + i], i < N))[v + Lb - 1],
// X_p the spectrum of the segment's samples at 0 .. len - 1: no wrapped product
// reaches the V samples kept.  The products are summed over the segments in the
// frequency domain, so a block costs one forward DFT per segment that reaches
// it and microphone pair, and one inverse DFT per pair.  N = 4096 sits in the
// registers of one CTA (256 threads x 16 points) and no intermediate goes to
// device memory: an RIR is read once (its blocks' overlap, Lb / V, from L2).
// The 48 kHz array (64 segments of 900 samples, 8 microphones, RIRs of 57,600):
// 5.1 k DFTs of 4096 points instead of 324 of 131,072, 94 us instead of 367.  Its sums
// (80 us) wait for L2 and shared memory with 16 warps per SM at 45 % of the issue slots;
// samples of the next piece fetched into registers (spills: 112 us) or by cp.async (a second
// barrier and 32 more shared loads a thread: 105 us) cost more than the waits.
//
// Two microphones share a complex sequence, as in the four-step form.  Segments
// longer than Lb are cut into pieces.  A uniform cut's segments have equally many
// (cuts: slot cuts p + j); with given starts piece j of segment p has the slot
// p + floor(a_p / Lb) + j, which no other piece has (starts are non-decreasing),
// so the slots need no prefix sum over the points.  A CTA takes the pieces of
// one group (of every G-th that reach its block) and leaves their summed
// products in the workspace; the groups are added in order by the inverse
// kernel.  Every sum has a fixed order.
//
// The DFT: n = a + 16 b + 256 j, k = k0 + 16 k1 + 256 k2,
//   thread (a, b): DFT16 over j -> k0, times W_4096^((a + 16 b) k0);
//   exchange b <-> k0 (across the CTA), thread (a, k0): DFT16 over b -> k1, times W_256^(a k1);
//   exchange a <-> k1 (within 16 lanes), thread (k1, k0): DFT16 over a -> k2.
// The spectrum stays where it lands (thread k1 + 16 k0 holds k2 = 0 .. 15): the
// products need only that X and H agree, and the inverse undoes the steps in
// reverse.  The exchanges are conflict-free: rows of 272 points per k0, 17 per k1.
#include "ism_device.cuh"

namespace {

#define AO_N 4096
#define AO_T 256
#define AO_ROW 272                    // points per k0 row of an exchange buffer
#define AO_BUF (16 * AO_ROW)
#define AO_XT 144                     // threads whose k0 <= 8: a piece's spectrum is Hermitian, the others' is theirs
#define AO_XN (16 * AO_XT)            // points kept of it

__device__ __forceinline__ float2 ao_cmul(float2 a, float2 b)
{
    return make_float2(__fmaf_rn(a.x, b.x, -a.y * b.y), __fmaf_rn(a.x, b.y, a.y * b.x));
}
// a conj(b)
__device__ __forceinline__ float2 ao_cmulc(float2 a, float2 b)
{
    return make_float2(__fmaf_rn(a.x, b.x, a.y * b.y), __fmaf_rn(-a.x, b.y, a.y * b.x));
}
template <bool INV>
__device__ __forceinline__ float2 ao_tw(float2 a, float2 w)
{
    return INV ? ao_cmulc(a, w) : ao_cmul(a, w);
}
__device__ __forceinline__ float2 ao_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 ao_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// exp(-2 pi i t / L), L = 2^logL, 0 <= t < L: the argument is exact
__device__ __forceinline__ float2 ao_root(int t, int logL)
{
    float s, c;
    sincospif(-__int2float_rn(2 * t) * __int_as_float((127 - logL) << 23), &s, &c);
    return make_float2(c, s);
}

// 4-point DFT in place (forward: W_4 = -i)
template <bool INV>
__device__ __forceinline__ void ao_dft4(float2& x0, float2& x1, float2& x2, float2& x3)
{
    const float2 a = ao_add(x0, x2), b = ao_sub(x0, x2), c = ao_add(x1, x3), d = ao_sub(x1, x3);
    x0 = ao_add(a, c);
    x2 = ao_sub(a, c);
    x1 = INV ? make_float2(b.x - d.y, b.y + d.x) : make_float2(b.x + d.y, b.y - d.x);
    x3 = INV ? make_float2(b.x + d.y, b.y - d.x) : make_float2(b.x - d.y, b.y + d.x);
}

// 16-point DFT: n = 4 n1 + n2, k = k1 + 4 k2; v[k] on return
template <bool INV>
__device__ __forceinline__ void ao_dft16(float2 (&v)[16])
{
    const float h = 0.70710678118654752440f, c = 0.92387953251128675613f, s = 0.38268343236508977173f;
    // cos, -sin of 2 pi m / 16, m = n2 k1
    const float2 w1 = make_float2(c, -s), w2 = make_float2(h, -h), w3 = make_float2(s, -c), w6 = make_float2(-h, -h),
                 w9 = make_float2(-c, s);
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) ao_dft4<INV>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);   // v[4 k1 + n2]
    v[4 + 1] = ao_tw<INV>(v[4 + 1], w1);
    v[4 + 2] = ao_tw<INV>(v[4 + 2], w2);
    v[4 + 3] = ao_tw<INV>(v[4 + 3], w3);
    v[8 + 1] = ao_tw<INV>(v[8 + 1], w2);
    v[8 + 2] = INV ? make_float2(-v[8 + 2].y, v[8 + 2].x) : make_float2(v[8 + 2].y, -v[8 + 2].x);   // W_16^4 = -i
    v[8 + 3] = ao_tw<INV>(v[8 + 3], w6);
    v[12 + 1] = ao_tw<INV>(v[12 + 1], w3);
    v[12 + 2] = ao_tw<INV>(v[12 + 2], w6);
    v[12 + 3] = ao_tw<INV>(v[12 + 3], w9);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) ao_dft4<INV>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);   // v[4 k1 + k2]
    float2 u[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) u[k1 + 4 * k2] = v[4 * k1 + k2];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = u[i];
}

// Forward DFT of the CTA's 4096 points: v[j] = z[tid + 256 j] on entry, v[k2] =
// Z[k0 + 16 k1 + 256 k2] for tid = k1 + 16 k0 on return.  t1 = W_4096^(tid k0) at
// [256 k0 + tid], t2 = W_256^(a k1) at [16 k1 + a].  buf must not be the buffer of the
// call before (whose rows slower warps may still read); one CTA barrier.
__device__ __forceinline__ void ao_forward(float2 (&v)[16], float2* buf, const float2* t1, const float2* t2)
{
    const int tid = threadIdx.x, a = tid & 15, hi = tid >> 4;
    ao_dft16<false>(v);
    buf[tid] = v[0];
#pragma unroll
    for (int k0 = 1; k0 < 16; ++k0) buf[AO_ROW * k0 + tid] = ao_cmul(v[k0], t1[256 * k0 + tid]);
    __syncthreads();
    float2* row = buf + AO_ROW * hi;   // thread (a, k0 = hi): the row is this warp's alone from here on
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = row[a + 16 * b];
    ao_dft16<false>(v);
    __syncwarp();
    row[a] = v[0];
#pragma unroll
    for (int k1 = 1; k1 < 16; ++k1) row[17 * k1 + a] = ao_cmul(v[k1], t2[16 * k1 + a]);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = row[17 * a + i];   // thread (k1 = a, k0)
    ao_dft16<false>(v);
}

// Its inverse (unscaled), the same layouts the other way round.
__device__ __forceinline__ void ao_inverse(float2 (&v)[16], float2* buf, const float2* t1, const float2* t2)
{
    const int tid = threadIdx.x, a = tid & 15, hi = tid >> 4;
    float2* row = buf + AO_ROW * hi;
    ao_dft16<true>(v);   // over k2 -> a
#pragma unroll
    for (int i = 0; i < 16; ++i) row[17 * a + i] = v[i];
    __syncwarp();
#pragma unroll
    for (int k1 = 0; k1 < 16; ++k1) v[k1] = k1 ? ao_cmulc(row[17 * k1 + a], t2[16 * k1 + a]) : row[a];
    ao_dft16<true>(v);   // over k1 -> b
    __syncwarp();
#pragma unroll
    for (int b = 0; b < 16; ++b) row[a + 16 * b] = v[b];   // [k0][a + 16 b]
    __syncthreads();
#pragma unroll
    for (int k0 = 0; k0 < 16; ++k0) v[k0] = k0 ? ao_cmulc(buf[AO_ROW * k0 + tid], t1[256 * k0 + tid]) : buf[tid];
    ao_dft16<true>(v);   // over k0 -> j
}

__device__ __forceinline__ int ao_start(int p, int n_x, int P, const int* starts)
{
    if (p >= P) return n_x;
    if (!starts) return (int)(((long long)p * n_x) / P);
    return min(max(starts[p], 0), n_x);
}

// t2, and t1 from the table that the piece kernel left in the workspace (t1g NULL: computed)
__device__ __forceinline__ void ao_tables(float2* t1, float2* t2, const float2* t1g)
{
    for (int e = threadIdx.x; e < AO_N; e += AO_T) t1[e] = t1g ? t1g[e] : ao_root((e >> 8) * (e & 255), 12);
    t2[threadIdx.x] = ao_root((threadIdx.x >> 4) * (threadIdx.x & 15), 8);
}

// One CTA per slot: finds its piece {p, s0, len} (len 0: none), writes it and its
// spectrum / N.  The first CTA also writes the twiddle table.
__global__ void __launch_bounds__(AO_T) ao_piece_kernel(AoPlan pl, const float* __restrict__ x,
                                                        const int* __restrict__ starts, int4* __restrict__ desc,
                                                        float2* __restrict__ t1g, float2* __restrict__ X)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float2* buf = reinterpret_cast<float2*>(smem);
    float2* t1 = buf + AO_BUF;
    float2* t2 = t1 + AO_N;
    const int c = blockIdx.x;
    ao_tables(t1, t2, nullptr);
    int lo = 0, hi = pl.P - 1;
    if (pl.cuts) lo = c / pl.cuts;
    else
        while (lo < hi) {   // the last point whose first slot is <= c
            const int mid = (lo + hi + 1) >> 1;
            if (mid + ao_start(mid, pl.n_x, pl.P, starts) / pl.Lb <= c) lo = mid;
            else hi = mid - 1;
        }
    const int a = ao_start(lo, pl.n_x, pl.P, starts), b = ao_start(lo + 1, pl.n_x, pl.P, starts);
    const long long s0 = (long long)a + (long long)(c - (pl.cuts ? lo * pl.cuts : lo + a / pl.Lb)) * pl.Lb;
    const int len = s0 >= a && s0 < b ? (int)min((long long)pl.Lb, b - s0) : 0;
    if (threadIdx.x == 0) desc[c] = make_int4(lo, (int)min(s0, (long long)pl.n_x), len, 0);
    __syncthreads();
    if (c == 0)
        for (int e = threadIdx.x; e < AO_N; e += AO_T) t1g[e] = t1[e];
    if (len == 0) return;   // CTA-uniform
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int n = (int)threadIdx.x + AO_T * j;
        v[j] = make_float2(n < len ? x[s0 + n] * (1.0f / AO_N) : 0.0f, 0.0f);
    }
    ao_forward(v, buf, t1, t2);
    if (threadIdx.x >= AO_XT) return;
    float2* Xc = X + (long long)c * AO_XN;
#pragma unroll
    for (int k = 0; k < 16; ++k) Xc[AO_XT * k + threadIdx.x] = v[k];
}

// One CTA per (block of outputs, group of pieces, microphone pair), the blocks that the
// most pieces reach (the middle ones) first.
__device__ __forceinline__ int ao_block(int i, int NB)
{
    const int mid = (NB - 1) / 2, d = (i + 1) / 2;
    return (i & 1) ? mid + d : mid - d;
}

// The RIR samples k0 + 256 j, j < 16, of microphone 2 q and, in the imaginary parts, 2 q + 1;
// 0 outside [0, n_S).  all: none of the CTA's is outside, and the pair has both.
__device__ __forceinline__ void ao_load(float2 (&v)[16], const float* h0, int n_S, long long k0, bool two, bool all)
{
    if (all) {
        const float* a = h0 + k0;
        const float* b = a + n_S;
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = make_float2(a[AO_T * j], b[AO_T * j]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const long long k = k0 + AO_T * j;
            const bool ok = k >= 0 && k < n_S;
            v[j] = make_float2(ok ? h0[k] : 0.0f, ok && two ? h0[n_S + k] : 0.0f);
        }
    }
}

__global__ void __launch_bounds__(AO_T, 2) ao_sum_kernel(AoPlan pl, const float* __restrict__ h,
                                                         const int4* __restrict__ desc,
                                                         const float2* __restrict__ t1g, const float2* __restrict__ X,
                                                         float2* __restrict__ Y)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float2* buf = reinterpret_cast<float2*>(smem);   // two exchange buffers, in turn
    float2* t1 = buf + 2 * AO_BUF;
    float2* t2 = t1 + AO_N;
    int* list = reinterpret_cast<int*>(t2 + 256);    // [256] slots of the scan's stretch that reach the block
    __shared__ int warp_n[AO_T / 32];
    const int tid = threadIdx.x;
    const int q = blockIdx.x % pl.n_pairs, bg = blockIdx.x / pl.n_pairs;
    const int bi = bg / pl.G, g = bg - bi * pl.G;
    const long long T0 = (long long)ao_block(bi, pl.NB) * pl.V;
    const bool two = 2 * q + 1 < pl.M;
    ao_tables(t1, t2, t1g);
    // where the piece spectra hold the values of this thread's k: its own, or for k0 > 8 the
    // conjugate at N - k = (16 - k0) + 16 (15 - k1) + 256 (15 - k2)
    const bool mirror = tid >= AO_XT;
    const int x0 = mirror ? 15 * AO_XT + (15 - (tid & 15)) + 16 * (16 - (tid >> 4)) : tid;
    const int xstep = mirror ? -AO_XT : AO_XT;
    const float xsign = mirror ? -1.0f : 1.0f;
    float2 acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = make_float2(0.0f, 0.0f);
    int turn = 0;
    int seen = 0;   // pieces that reach the block before this stretch
    for (int c0 = 0; c0 < pl.slots; c0 += AO_T) {
        // the stretch's pieces that reach the block, in order, every G-th of them this CTA's
        __syncthreads();
        const int c = c0 + tid;
        bool in = false;
        if (c < pl.slots) {
            const int4 d = desc[c];
            in = d.z > 0 && d.y < T0 + pl.V && (long long)d.y + d.z + pl.n_S - 1 > T0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if ((tid & 31) == 0) warp_n[tid >> 5] = __popc(m);
        __syncthreads();
        int before = 0, n = 0;
#pragma unroll
        for (int w = 0; w < AO_T / 32; ++w) {
            before += w < (tid >> 5) ? warp_n[w] : 0;
            n += warp_n[w];
        }
        if (in) list[before + __popc(m & ((1u << (tid & 31)) - 1u))] = c;
        __syncthreads();
        for (int i = ((g - seen) % pl.G + pl.G) % pl.G; i < n; i += pl.G) {
            const int cs = list[i];
            const int4 d = desc[cs];
            // h'[i] = h[T0 - s0 - (Lb - 1) + i]
            const long long o = T0 - d.y - (pl.Lb - 1);
            float2 v[16];
            ao_load(v, h + ((long long)d.x * pl.M + 2 * q) * pl.n_S, pl.n_S, o + tid, two,
                    two && o >= 0 && o + AO_N <= pl.n_S);
            if (i + pl.G < n) {   // the next piece's samples on their way to L2: 256 lines of 128 bytes, one a thread
                const int4 dn = desc[list[i + pl.G]];
                const long long k = T0 - dn.y - (pl.Lb - 1) + 32 * (tid & 127);
                if (k >= 0 && k < pl.n_S && (tid < 128 || two))
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(
                        h + ((long long)dn.x * pl.M + 2 * q + (tid >> 7)) * pl.n_S + k));
            }
            ao_forward(v, buf + turn * AO_BUF, t1, t2);
            turn ^= 1;
            const float2* Xc = X + (long long)cs * AO_XN + x0;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float2 xk = Xc[xstep * k];
                const float xi = xk.y * xsign;
                acc[k].x = __fmaf_rn(xk.x, v[k].x, __fmaf_rn(-xi, v[k].y, acc[k].x));
                acc[k].y = __fmaf_rn(xk.x, v[k].y, __fmaf_rn(xi, v[k].x, acc[k].y));
            }
        }
        seen += n;
    }
    float2* Yo = Y + (((long long)q * pl.NB + bi) * pl.G + g) * AO_N + tid;
#pragma unroll
    for (int k = 0; k < 16; ++k) Yo[AO_T * k] = acc[k];
}

__global__ void __launch_bounds__(AO_T, 2) ao_out_kernel(AoPlan pl, const float2* __restrict__ t1g,
                                                         const float2* __restrict__ Y, float* __restrict__ y)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float2* buf = reinterpret_cast<float2*>(smem);
    float2* t1 = buf + AO_BUF;
    float2* t2 = t1 + AO_N;
    const int tid = threadIdx.x;
    const int bi = blockIdx.x, q = blockIdx.y;
    const long long T0 = (long long)ao_block(bi, pl.NB) * pl.V;
    const float2* Yo = Y + ((long long)q * pl.NB + bi) * pl.G * AO_N + tid;
    float2 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = Yo[AO_T * k];
#pragma unroll 2
    for (int g = 1; g < pl.G; ++g)
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = ao_add(v[k], Yo[(long long)g * AO_N + AO_T * k]);
    ao_tables(t1, t2, t1g);
    __syncthreads();
    ao_inverse(v, buf, t1, t2);
    float* y0 = y + (long long)(2 * q) * pl.n_out + T0;
    const bool two = 2 * q + 1 < pl.M;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int o = tid + AO_T * j - (pl.Lb - 1);   // output of the block
        if (o >= 0 && o < pl.V && T0 + o < pl.n_out) {
            y0[o] = v[j].x;
            if (two) y0[pl.n_out + o] = v[j].y;
        }
    }
}

}  // namespace

// Operations of the overlap-save form's DFTs, 5 n log2 n each: one per (piece, block that
// it reaches, pair), per (block, pair) and per piece.
static double ao_flops(const AoPlan& pl, double pieces)
{
    const double reach = ((double)pl.n_S + pl.Lb) / pl.V + 1.0;   // blocks that a piece reaches
    return 5.0 * AO_N * 12 * ((pieces * std::min(reach, (double)pl.NB) + pl.NB) * pl.n_pairs + pieces);
}

// Sizes that do not depend on a workspace; false if the form cannot take the filtering.
static bool ao_sizes(int n_x, int P, int M, int n_S, bool uniform, AoPlan& pl, double* flops)
{
    pl = AoPlan{};
    pl.n_x = n_x;
    pl.P = P;
    pl.M = M;
    pl.n_S = n_S;
    pl.n_out = n_x + n_S - 1;
    pl.n_pairs = (M + 1) / 2;
    // pieces of at most Lb samples: a uniform cut's segments whole, up to half the DFT
    // length; segments of unknown lengths up to twice their mean
    const int seg = (n_x + P - 1) / P;
    const int cap = AO_N / 2;
    const int cuts = (seg + cap - 1) / cap;
    pl.Lb = uniform ? (seg + cuts - 1) / cuts : std::min(cap, 2 * seg);
    pl.V = AO_N - pl.Lb + 1;
    pl.NB = (pl.n_out + pl.V - 1) / pl.V;
    pl.cuts = uniform ? (seg + pl.Lb - 1) / pl.Lb : 0;
    const long long slots = uniform ? (long long)P * pl.cuts : (long long)P + n_x / pl.Lb + 1;
    if (slots > 65535 || (long long)pl.NB * 8 * pl.n_pairs > 0x7FFFFFFFll || pl.n_pairs > 65535) return false;
    pl.slots = (int)slots;
    *flops = ao_flops(pl, uniform ? (double)P * pl.cuts : 1.3 * P);
    return true;
}

// Seconds of the four-step form, roughly: its launches, and per length-N DFT (one per segment,
// one per microphone pair and point, one inverse per pair) 4 N log2 N lane operations and 4 N
// per product of spectra, at 6 T/s.
double ism_auralize_four_step_seconds(int logN, int P, int pairs)
{
    const double N = (double)(1ll << logN);
    return 2.4e-5 + (((double)P * (1.0 + pairs) + pairs) * 4.0 * N * logN + (double)P * pairs * 4.0 * N) / 6.0e12;
}

// Whether the overlap-save form takes a filtering, and its plan.  It does where its DFTs'
// operations are below 1.3 times the four-step form's (one DFT of 2^logN per segment and
// per (point, pair)), which passes over device memory twice.  Measured at a ratio of 0.35
// (64 points x 8 microphones, 57,600 samples): 97 against 367 us; 0.97 (16 points) 75 and
// 107; 1.48 (10 points, 144,000 samples, 4 microphones) 86 and 111; 1.84 (8 points) 75 and
// 69; 3.4 (4 points) 73 and 53.
// ws_min: the workspace that the four-step form needs at least (every workspace that
// the caller may pass holds that; this form takes no more).
// out->seconds: the time that the form takes, within 10 % (rms of 410 sizes), for the choice
// between it and the direct form: three launches, 26 us, and the DFTs, at 14 T operations/s
// where they fill the GPU and 2 us for each piece of a CTA's, one after another, where a
// few blocks in a small workspace leave few CTAs (270 samples in 99 segments, RIRs of
// 16,285, 2 microphones: 99 pieces in each of 5 CTAs, 255 us); out->total: the workspace it takes.
bool ism_auralize_ols_plan(int n_x, int P, int M, int n_S, bool uniform, int logN, size_t ws_min, AoPlan* out)
{
    AoPlan pl;
    double flops = 0.0;
    if (!ao_sizes(n_x, P, M, n_S, uniform, pl, &flops)) return false;
    const double N = (double)(1ll << logN);
    if (flops > 1.3 * 5.0 * N * logN * ((double)P * (1.0 + pl.n_pairs) + pl.n_pairs)) return false;
    // groups of pieces: the least that give 1.85 CTAs per slot of the launch (2 per SM); more
    // only add products to write and sum.  Groups 1 to 5, us: 148 (block, pair)s, 185 121 95
    // 94 97; 204, 101 73 73 77; 208, 70 64 60 64 66; 246, 92 70 64 68; 32, 178 101 76 64 64
    const long long units = (long long)pl.NB * pl.n_pairs;
    pl.G = (int)std::max(1LL, std::min(8LL, (562 + units - 1) / units));
    for (;; --pl.G) {
        size_t off = 0;
        auto take = [&](size_t bytes) {
            const size_t o = off;
            off = (off + bytes + 255) & ~(size_t)255;
            return o;
        };
        pl.desc_off = take((size_t)pl.slots * sizeof(int4));
        pl.t1_off = take((size_t)AO_N * sizeof(float2));
        pl.x_off = take((size_t)pl.slots * AO_XN * sizeof(float2));
        pl.y_off = take((size_t)units * pl.G * AO_N * sizeof(float2));
        pl.total = off;
        if (off <= ws_min) break;
        if (pl.G == 1) return false;
    }
    const double pieces = (uniform ? (double)P * pl.cuts : std::min(1.3 * P, (double)n_x)) *
                          std::min(1.0, ((double)n_S + pl.V) / n_x);
    const double ctas = (double)units * pl.G;
    pl.seconds = 2.6e-5 + std::max(flops / 1.4e13, std::ceil(pieces / pl.G) * 2.0e-6 * std::max(1.0, ctas / 304.0));
    // (nor where a chain of pieces makes it longer than the four-step form: 44 segments of 7
    // samples x 3 microphones, RIRs of 6720, 136 and 38 us)
    if (pl.seconds > 1.15 * ism_auralize_four_step_seconds(logN, P, pl.n_pairs)) return false;
    *out = pl;
    return true;
}

int ism_launch_auralize_ols(const float* x, const float* h, const int* starts, float* y, const AoPlan& pl, char* ws,
                            void* stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    int4* desc = reinterpret_cast<int4*>(ws + pl.desc_off);
    float2* t1 = reinterpret_cast<float2*>(ws + pl.t1_off);
    float2* X = reinterpret_cast<float2*>(ws + pl.x_off);
    float2* Y = reinterpret_cast<float2*>(ws + pl.y_off);
    const size_t one = (size_t)(AO_BUF + AO_N + 256) * sizeof(float2);
    const size_t sum = one + (size_t)AO_BUF * sizeof(float2) + AO_T * sizeof(int);
    static std::atomic<unsigned long long> o1{0}, o2{0}, o3{0};
    int rc;
    if ((rc = ism_open_smem((const void*)ao_piece_kernel, &o1))) return rc;
    if ((rc = ism_open_smem((const void*)ao_sum_kernel, &o2))) return rc;
    if ((rc = ism_open_smem((const void*)ao_out_kernel, &o3))) return rc;
    ao_piece_kernel<<<(unsigned)pl.slots, AO_T, one, s>>>(pl, x, starts, desc, t1, X);
    if ((rc = (int)cudaGetLastError())) return rc;
    ao_sum_kernel<<<(unsigned)(pl.NB * pl.G * pl.n_pairs), AO_T, sum, s>>>(pl, h, desc, t1, X, Y);
    if ((rc = (int)cudaGetLastError())) return rc;
    ao_out_kernel<<<dim3((unsigned)pl.NB, (unsigned)pl.n_pairs), AO_T, one, s>>>(pl, t1, Y, y);
    return (int)cudaGetLastError();
}
