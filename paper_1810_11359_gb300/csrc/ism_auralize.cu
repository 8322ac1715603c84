// ism_auralize.cu -- moving sources (Section 4): the source signal is cut into
// one segment per trajectory point, each segment is filtered by the RIRs of its
// point (one per microphone) and the filtered segments are overlap-added:
//   y[m][t] = sum_p sum_{s in [a_p, a_(p+1))} x[s] h[p][m][t - s].
// The paper does this with batched FFTs; here it is a direct FP32 convolution
// on the FMA pipe (the RIRs are long, the signal is short, and the sum has a
// fixed order).
//
// One CTA owns 128 consecutive output samples and up to 8 microphones (1, 2, 4 or
// 8, the least that holds the call's).  Lane l of a warp owns the outputs
// T0 + 4 l + r, r = 0 .. 3, for the microphones (32 accumulators for 8).  For one
// segment the taps k that connect it to the tile are walked in chunks of 128;
// the chunks of all segments are dealt to the CTA's warps in turn, which add
// their partial sums in warp order at the end.  A segment's chunks are of one size where their
// number is a power of two (142 taps as 72 + 70, not 128 + 14, of which every other warp
// would take the short ones: 18 segments of 14 samples, RIRs of 27,800, 9 microphones 103 ->
// 62 us).  (16 points x 1 microphone, RIRs
// of 9600 samples, a signal of 57,600: 337 us with 8 microphones' sums always
// and whole segments dealt to 4 warps, 49 us now; 30 x 5, 16,000, 48,000: 340 ->
// 282; the 48 kHz array 1285 -> 1193.)
// The chunk's taps of the microphones and the signal window it needs (the
// samples outside the segment zeroed) are staged in the warp's shared memory,
// the taps as [microphone][k] rows copied with 128-bit loads when every RIR
// row starts on a 16-byte boundary (n_S a multiple of 4; the chunk's first
// tap rounded down to a multiple of 4 -- the extra taps meet zeroed signal
// samples), else one float at a time.  The taps go in groups of 4: for taps
// k .. k + 3 the lane's 16 products need the 7 signal values
// x[T0 + 4 l - k - 3 .. T0 + 4 l - k + 3], two aligned float4 of the window of
// which the later one is the previous group's earlier one, so a group costs
// one 128-bit signal load (the 32 lanes read 512 contiguous bytes) and eight
// broadcast 128-bit tap loads (taps k .. k + 3 of each microphone) for 128
// FFMA; every shared address is the lane's base plus a constant.  (8 outputs per lane: fewer CTAs than SM
// slots, 13 % of the warps active, measured 10 % slower.)
#include "ism_device.cuh"

namespace {

#define AU_R 4                       // outputs per lane
#define AU_KC 128                    // taps per staged chunk
#define AU_TILE (32 * AU_R)          // outputs per CTA
#define AU_XN (AU_TILE + AU_KC)      // signal samples per chunk (the last one is never used)

static_assert(AU_R == 4 && AU_KC % 4 == 0, "the signal window is read as float4 groups of 4 taps");

template <int AU_M>
struct AuWarp {
    float4 h[AU_M][AU_KC / 4];       // taps of the chunk: [microphone][k / 4]
    float4 x[AU_XN / 4];             // signal window
};

// Segment of sample s (the largest p with a_p <= s): uniform cut when starts
// is NULL, else a binary search over the caller's start array.
__device__ __forceinline__ int au_segment(long long s, int n_x, int n_points, const int* starts)
{
    if (!starts) return (int)min((long long)n_points - 1, ((s + 1) * n_points - 1) / n_x);
    int lo = 0, hi = n_points - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long long)starts[mid] <= s) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int au_start(int p, int n_x, int n_points, const int* starts)
{
    if (!starts) return (int)(((long long)p * n_x) / n_points);
    return min(max(starts[p], 0), n_x);
}

// VEC: 128-bit tap staging (16-byte aligned RIR rows); AU_M: microphones per CTA
template <bool VEC, int AU_M, int AU_WARPS>
__global__ void __launch_bounds__(AU_WARPS * 32, AU_WARPS > 4 ? 1 : AU_M == 8 ? 5 : 6)   // (8 in 80 registers: spills)
    auralize_kernel(const float* __restrict__ x, int n_x, const float* __restrict__ h, int n_points, int n_mics, int n_s,
                    const int* __restrict__ starts, float* __restrict__ y, int n_out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    AuWarp<AU_M>& W = reinterpret_cast<AuWarp<AU_M>*>(smem)[warp];
    const long long T0 = (long long)blockIdx.x * AU_TILE;
    const int m0 = blockIdx.y * AU_M;

    float acc[AU_R][AU_M];
#pragma unroll
    for (int r = 0; r < AU_R; ++r)
#pragma unroll
        for (int m = 0; m < AU_M; ++m) acc[r][m] = 0.0f;

    // samples that reach the tile: s in [T0 - n_s + 1, T0 + TILE - 1]
    const long long s_lo = max(T0 - n_s + 1, 0ll);
    const long long s_hi = min(T0 + AU_TILE - 1, (long long)n_x - 1);
    if (s_lo <= s_hi) {
        const int p_lo = au_segment(s_lo, n_x, n_points, starts);
        const int p_hi = au_segment(s_hi, n_x, n_points, starts);
        int turn = 0;   // chunks of the segments so far, modulo the warps
        for (int p0 = p_lo; p0 <= p_hi; p0 += 32) {
          // the bounds of 32 segments at once, a lane each
          int a_l = 0, b_l = 0;
          if (p0 + lane <= p_hi) {
              a_l = au_start(p0 + lane, n_x, n_points, starts);
              b_l = max(a_l, p0 + lane + 1 < n_points ? au_start(p0 + lane + 1, n_x, n_points, starts) : n_x);
          }
          for (int pp = 0; pp < min(32, p_hi - p0 + 1); ++pp) {
            const int p = p0 + pp;
            const int a = __shfl_sync(0xffffffffu, a_l, pp), b = __shfl_sync(0xffffffffu, b_l, pp);
            if (b <= a) continue;
            // taps linking [a, b) to the tile (the vector form starts on a multiple of 4)
            const long long k_lo = VEC ? (max(T0 - b + 1, 0ll) & ~3ll) : max(T0 - b + 1, 0ll);
            const long long k_hi = min(T0 + AU_TILE - 1 - a, (long long)n_s - 1);
            if (k_hi < k_lo) continue;
            const float* hp = h + (long long)p * n_mics * n_s;
            const int n_k = (int)(k_hi - k_lo);
            const int n_ch = n_k / AU_KC + 1;
            // taps of a chunk: as even as whole groups allow where the number of chunks shares
            // the warps' (a power of two), else 128 and a remnant that goes round all warps
            const int kc = n_ch & (n_ch - 1) ? AU_KC : ((n_k >> (31 - __clz(n_ch))) + 4) & ~3;
            const int first = (warp - turn + AU_WARPS) % AU_WARPS;   // the warp's first chunk of this segment
            turn = (turn + n_ch) % AU_WARPS;
            for (long long k0 = k_lo + (long long)first * kc; k0 <= k_hi; k0 += AU_WARPS * kc) {
                __syncwarp();
                // taps k0 .. k0 + KC - 1 of the microphones (0 past k_hi or past the array; those
                // past k0 + kc - 1 are not used)
                if (VEC) {
                    for (int e = lane; e < AU_M * AU_KC / 4; e += 32) {   // 32 lanes: 512 contiguous bytes
                        const int m = e / (AU_KC / 4), kq = e % (AU_KC / 4);
                        const long long k = k0 + 4 * kq;   // k0 % 4 == 0 and n_s % 4 == 0: k .. k + 3 < n_s
                        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (k <= k_hi && m0 + m < n_mics)
                            v = *reinterpret_cast<const float4*>(hp + (long long)(m0 + m) * n_s + k);
                        W.h[m][kq] = v;
                    }
                } else {
                    for (int e = lane; e < AU_KC * AU_M; e += 32) {   // coalesced along the taps
                        const int m = e / AU_KC, kk = e % AU_KC;
                        const long long k = k0 + kk;
                        float v = 0.0f;
                        if (k <= k_hi && m0 + m < n_mics) v = hp[(long long)(m0 + m) * n_s + k];
                        reinterpret_cast<float*>(&W.h[m][0])[kk] = v;
                    }
                }
                // signal window: x[T0 - k0 - KC + 1 + j], zero outside [a, b)
                const long long xb = T0 - k0 - AU_KC + 1;
                float* xw = reinterpret_cast<float*>(W.x);
                for (int j = lane; j < AU_XN; j += 32) {
                    const long long s = xb + j;
                    xw[j] = (s >= a && s < b) ? x[s] : 0.0f;
                }
                __syncwarp();
                // output r of the lane at tap kk reads window index 4 l + r + KC - 1 - kk; for the
                // group kk = 4 g + u that is element 3 + r - u of {xa, xb4}, xa = float4 at
                // 4 l + KC - 4 - 4 g, xb4 = the next float4 (the previous group's xa)
                const float4* xl = W.x + lane + (AU_KC - 4) / 4;
                float4 xb4 = xl[1];
                // the groups that hold taps of the chunk
                const int ng = (int)min((long long)(kc / 4), (k_hi - k0) / 4 + 1);
#pragma unroll 2
                for (int g = 0; g < ng; ++g) {
                    const float4 xa = xl[-g];
                    const float v[8] = {xa.x, xa.y, xa.z, xa.w, xb4.x, xb4.y, xb4.z, xb4.w};
                    float hv[AU_M][4];   // taps 4 g .. 4 g + 3 of each microphone
#pragma unroll
                    for (int m = 0; m < AU_M; ++m) {
                        const float4 hm = W.h[m][g];
                        hv[m][0] = hm.x;
                        hv[m][1] = hm.y;
                        hv[m][2] = hm.z;
                        hv[m][3] = hm.w;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int r = 0; r < AU_R; ++r)
#pragma unroll
                            for (int m = 0; m < AU_M; ++m)
                                acc[r][m] = __fmaf_rn(v[3 + r - u], hv[m][u], acc[r][m]);
                    xb4 = xa;
                }
            }
          }
        }
    }

    // partial sums of the warps, added in warp order
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);   // [warps][R][M][32]
#pragma unroll
    for (int r = 0; r < AU_R; ++r)
#pragma unroll
        for (int m = 0; m < AU_M; ++m) red[((warp * AU_R + r) * AU_M + m) * 32 + lane] = acc[r][m];
    __syncthreads();
    // thread e writes output (t, m) pairs; consecutive threads take consecutive t
    for (int e = threadIdx.x; e < AU_TILE * AU_M; e += blockDim.x) {
        const int m = e / AU_TILE, i = e % AU_TILE;   // i = 4 l + r
        const int l = i / AU_R, r = i % AU_R;
        float v = red[((0 * AU_R + r) * AU_M + m) * 32 + l];
#pragma unroll
        for (int w = 1; w < AU_WARPS; ++w) v += red[((w * AU_R + r) * AU_M + m) * 32 + l];
        const long long t = T0 + i;
        if (t < n_out && m0 + m < n_mics) y[(long long)(m0 + m) * n_out + t] = v;
    }
}

template <bool VEC, int AU_M, int AU_WARPS>
int launch_au(const float* x, int n_x, const float* h, int n_points, int n_mics, int n_s, const int* starts, float* y,
              cudaStream_t s)
{
    const long long n_out = (long long)n_x + n_s - 1;
    const dim3 grid((unsigned)((n_out + AU_TILE - 1) / AU_TILE), (unsigned)((n_mics + AU_M - 1) / AU_M));
    const size_t sm = std::max(AU_WARPS * sizeof(AuWarp<AU_M>), (size_t)AU_WARPS * AU_R * AU_M * 32 * sizeof(float));
    static std::atomic<unsigned long long> opened{0};
    const int rc = ism_open_smem((const void*)auralize_kernel<VEC, AU_M, AU_WARPS>, &opened);
    if (rc) return rc;
    auralize_kernel<VEC, AU_M, AU_WARPS><<<grid, AU_WARPS * 32, sm, s>>>(x, n_x, h, n_points, n_mics, n_s, starts, y,
                                                                       (int)n_out);
    return (int)cudaGetLastError();
}

template <bool VEC, int AU_M>
int launch_au_m(const float* x, int n_x, const float* h, int n_points, int n_mics, int n_s, const int* starts, float* y,
                cudaStream_t s)
{
    // 16 warps share a tile where it has chunks for them; 4 where a tile has few (RIRs or segments
    // of a chunk or two) and there are tiles to fill the GPU all the same.  By the turns that the
    // fullest warp takes, an SM running 16 warps as fast as one: a turn is a chunk, 1.5 or 2 more
    // begin and end the tile, and every warp looks at all the tile's segments, a fifth of a
    // turn each for one microphone.  Long tiles (64 chunks or more of whole segments) in fewer
    // than 1024 end the launch better in 16 warps.  1000 sizes from 200 x 50 to 250,000 x
    // 80,000 samples: 0.6 % above the better of the two on average, 37 % at most.  us, 4 warps
    // and 16: 241,000 samples, RIRs of 51, 11 microphones 36 and 140; 3000 segments of 16
    // samples, RIRs of 8960 527 and 688; 10 points x 2, 12,001, 4801 25 and 17; the 48 kHz
    // array 1326 and 1192.
    const long long tiles = (((long long)n_x + n_s - 1 + AU_TILE - 1) / AU_TILE) * ((n_mics + AU_M - 1) / AU_M);
    const int seg = std::max(1, n_x / n_points);
    const long long segs = std::min<long long>(n_points, std::min<long long>(n_x, n_s + AU_TILE - 1ll) / seg + 1);
    const long long chunks = segs * ((std::min<long long>(n_s, seg + AU_TILE - 1ll) + AU_KC - 1) / AU_KC);
    const auto turns = [&](int warps, double ends) {
        return std::max(1.0, (double)tiles * warps / (152.0 * 16.0)) *
               ((double)((chunks + warps - 1) / warps) + ends + 0.2 * (double)segs / AU_M);
    };
    const bool few_long = seg >= AU_KC && chunks >= 64 && tiles < 1024;
    return turns(4, 1.5) * (few_long ? 1.3 : 1.0) <= turns(16, 2.0)
               ? launch_au<VEC, AU_M, 4>(x, n_x, h, n_points, n_mics, n_s, starts, y, s)
               : launch_au<VEC, AU_M, 16>(x, n_x, h, n_points, n_mics, n_s, starts, y, s);
}

}  // namespace

int ism_launch_auralize(const float* x, int n_x, const float* h, int n_points, int n_mics, int n_s,
                        const int* starts, float* y, void* stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    // 128-bit tap rows when every row starts on a 16-byte boundary
    const bool vec = (n_s % 4 == 0) && (((uintptr_t)h & 15u) == 0);
#define AU_L(M)                                                                      \
    return vec ? launch_au_m<true, M>(x, n_x, h, n_points, n_mics, n_s, starts, y, s) \
               : launch_au_m<false, M>(x, n_x, h, n_points, n_mics, n_s, starts, y, s)
    if (n_mics == 1) AU_L(1);
    if (n_mics == 2) AU_L(2);
    if (n_mics <= 4) AU_L(4);
    AU_L(8);
#undef AU_L
}
