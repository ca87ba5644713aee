// Measurements (Sec. 2.4, "Measurements": sampling the final state and the
// outcome probabilities of a group of qubits traced over the others; Sec. 3.3
// times the sampling):
//   * marginal_partial_kernel / marginal_finalize_kernel: per-block histograms
//     of |psi|^2 over the group's outcome in shared memory (each thread adds
//     the sum of a run of amplitudes with one outcome), then a fixed-order sum
//     of the blocks' histograms (FP64);
//     (a group that leaves 4 index bits above the low 8 free: those are a
//     thread's registers, so a thread's outcome stays the same over its walk);
//   * block_sums_kernel, scan kernels, sample_kernel: |psi|^2 summed over
//     blocks of kSampleBlock amplitudes, their exclusive prefix sums in FP64
//     (a two-level scan), the cumulative sums at 32 points inside each block
//     (segment_kernel), and one warp per shot: a binary search over the block
//     prefixes, one look at the block's points, then a warp scan up to the
//     first amplitude whose cumulative probability exceeds the shot's target.
#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "float_sum.cuh"
#include "internal.h"
#include "prof.h"

namespace qsim {

static int sms_of(int device) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || v <= 0) v = 148;
    return v;
}

// ------------------------------------------------------------------ marginals
struct MargP {
    int pos[kMarginalMaxQubits];  // index bit of the group's qubit j (outcome bit m-1-j)
    int m;
    int ms;        // member shift
    uint64_t per;  // amplitudes per member
};

// Each block takes a contiguous range of the member's amplitudes (a multiple
// of 256 long); thread tid reads x = start + tid + 256 i (coalesced), so its
// index bits 0..7 are fixed and its outcome y changes only where x crosses a
// multiple of 2^pmin, pmin the lowest group bit above bit 7. The thread walks
// those runs: y is formed once per run, the run's |psi|^2 is summed (runs of
// 64 in the state's precision, then FP64; 8 loads in flight) and added to the
// block's shared histogram.
template <typename R>
__global__ void __launch_bounds__(256) marginal_partial_kernel(const V<R> *__restrict__ psi, const MargP p,
                                                               double *__restrict__ part) {
    __shared__ double h[1 << kMarginalMaxQubits];
    const int bins = 1 << p.m;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) h[i] = 0.0;
    __syncthreads();
    const V<R> *q = psi + ((uint64_t)blockIdx.y << p.ms);
    const uint64_t span = ((p.per + gridDim.x - 1) / gridDim.x + 255) & ~255ull;
    const uint64_t start = (uint64_t)blockIdx.x * span;
    const uint64_t end = start + span < p.per ? start + span : p.per;
    int pmin = 63;
    for (int j = 0; j < p.m; ++j)
        if (p.pos[j] >= 8 && p.pos[j] < pmin) pmin = p.pos[j];
    constexpr int U = 8;  // loads in flight per thread
    for (uint64_t x0 = start + threadIdx.x; x0 < end;) {
        uint32_t y = 0;
        for (int j = 0; j < p.m; ++j) y |= (uint32_t)((x0 >> p.pos[j]) & 1ull) << (p.m - 1 - j);
        // the run ends at the next multiple of 2^pmin (or the range's end)
        const uint64_t bound = ((x0 >> pmin) + 1) << pmin;
        const uint64_t rend = bound < end ? bound : end;
        double accd = 0.0;
        R accf = 0;
        int run = 0;
        uint64_t x = x0;
        for (; x < rend; x += (uint64_t)U * blockDim.x) {
            R pr[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint64_t xk = x + (uint64_t)k * blockDim.x;
                pr[k] = 0;
                if (xk < rend) {
                    const V<R> a = q[xk];
                    pr[k] = a.x * a.x + a.y * a.y;
                }
            }
#pragma unroll
            for (int k = 0; k < U; ++k) accf += pr[k];
            run += U;
            if (run >= 64) {
                accd += (double)accf;
                accf = 0;
                run = 0;
            }
        }
        atomicAdd(&h[y], accd + (double)accf);
        x0 = rend + threadIdx.x;  // rend is a multiple of 256 unless it is the range's end
    }
    __syncthreads();
    double *out = part + ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * bins;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) out[i] = h[i];
}

// The same where at least 4 index bits above the low 8 are not the group's. A
// thread holds 16 amplitudes that differ in the lowest 4 of those (16 loads in
// flight), its low 8 index bits are its own, and the block walks the other free
// bits with the group's high bits fixed: one outcome per thread until the high
// outcome changes, one FP64 sum, and a shuffle over the lanes that share an
// outcome before the histogram. FP64 takes the sums of 2^LV products (in pairs,
// fours, ...): 16, or as many as the runs of marginal_partial_kernel hold where
// the group's lowest bit above 8 leaves them shorter (bit 8: every product).
// Bound by memory, with a thread's 16 loads in flight together: 4 CTAs per SM
// have the 60 registers a thread that takes; left to itself the compiler kept to
// 40 and issued the loads in parts (n = 32 complex64: 5.9 ms, so 4.9).
struct MargWalkP {
    int pos[kMarginalMaxQubits];
    int m;
    int ms;
    int reg[4];         // the register bits
    uint64_t rest;      // walked bits: above 8, neither the group's nor register bits
    uint64_t high;      // the group's bits above 8
    int nrest;          // bits of rest
    uint32_t lanes;     // lane bits the group has
    int lv;             // products summed in the state's precision: 2^lv
    uint64_t chunks;    // per member: 2^(n - 12)
};

template <typename R, int LV>
__global__ void __launch_bounds__(256, 4) marginal_walk_kernel(const V<R> *__restrict__ psi, const MargWalkP p,
                                                            double *__restrict__ part) {
    __shared__ double h[1 << kMarginalMaxQubits];
    const int bins = 1 << p.m;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) h[i] = 0.0;
    __syncthreads();
    const V<R> *q = psi + ((uint64_t)blockIdx.y << p.ms) + threadIdx.x;
    // chunk k: the low nrest bits walk `rest`, the others `high`
    const uint64_t k0 = p.chunks * blockIdx.x / gridDim.x, k1 = p.chunks * (blockIdx.x + 1) / gridDim.x;
    auto deposit = [](uint64_t v, uint64_t mask) {
        uint64_t x = 0;
        for (; mask; mask &= mask - 1, v >>= 1)
            if (v & 1ull) x |= mask & (0ull - mask);
        return x;
    };
    uint64_t xr = deposit(k0 & ((1ull << p.nrest) - 1ull), p.rest), xh = deposit(k0 >> p.nrest, p.high);
    uint64_t off[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) off[j] = 1ull << p.reg[j];
    // more than 2 FP64 sums per chunk go through FloatSum
    constexpr bool kFloats = sizeof(R) == 4 && LV <= 2;
    double acc = 0.0;
    FloatSum fs;
    for (uint64_t k = k0; k < k1;) {
        bool done;  // the high outcome ends here, or the block's range
#pragma unroll 1
        for (int i = 0; i < 8; ++i) {
            const V<R> *b = q + (xr | xh);
            V<R> a[16];
#pragma unroll
            for (int c = 0; c < 16; ++c)
                a[c] = b[((c & 1) ? off[0] : 0ull) | ((c & 2) ? off[1] : 0ull) | ((c & 4) ? off[2] : 0ull) |
                         ((c & 8) ? off[3] : 0ull)];
            R pr[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) pr[c] = a[c].x * a[c].x + a[c].y * a[c].y;
#pragma unroll
            for (int l = 0; l < LV; ++l)
#pragma unroll
                for (int j = 0; j < (16 >> (l + 1)); ++j) pr[j] = pr[2 * j] + pr[2 * j + 1];
            if constexpr (kFloats) {
#pragma unroll
                for (int j = 0; j < (16 >> LV); j += 4) fs.add(pr + j);
            } else {
#pragma unroll
                for (int j = 0; j < (16 >> LV); ++j) acc += (double)pr[j];
            }
            xr = (xr - p.rest) & p.rest;
            done = ++k == k1 || xr == 0;
            if (done) break;
        }
        if constexpr (kFloats) {
            fs.flush();
            acc += fs.sum;
            fs.sum = 0.0;
        }
        if (done) {
            const uint64_t x = xh | threadIdx.x;
            uint32_t y = 0;
            for (int j = 0; j < p.m; ++j) y |= (uint32_t)((x >> p.pos[j]) & 1ull) << (p.m - 1 - j);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
                if (!(p.lanes & o)) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if ((threadIdx.x & 31u & ~p.lanes) == 0) atomicAdd(&h[y], acc);
            acc = 0.0;
            xh = (xh - p.high) & p.high;
        }
    }
    __syncthreads();
    double *out = part + ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * bins;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) out[i] = h[i];
}

// 32 bins per CTA, the parts in 8 slices, the slices in a fixed order
__global__ void __launch_bounds__(256) marginal_finalize_kernel(const double *__restrict__ part, int parts,
                                                                int bins, double *__restrict__ out) {
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int y = blockIdx.x * 32 + lane;
    const double *pp = part + (uint64_t)blockIdx.y * parts * bins + y;
    double acc = 0.0;
    if (y < bins)
        for (int b = slice; b < parts; b += 8) acc += pp[(uint64_t)b * bins];
    sh[slice][lane] = acc;
    __syncthreads();
    if (slice == 0 && y < bins) {
        for (int w = 1; w < 8; ++w) acc += sh[w][lane];
        out[(uint64_t)blockIdx.y * bins + y] = acc;
    }
}

// Whether the walk takes the group (its 4 register bits exist), and its
// parameters. It is the faster one wherever it applies. Microseconds, complex64,
// against marginal_partial_kernel, whose runs are short where the group has a low
// bit above 8: n = 27, one qubit at bit 11 / 16 / 23: 184 / 184 / 184 against
// 3825 / 267 / 245, 8 lane and warp bits 183 against 207; n = 32, bit 16 / 23:
// 4964 / 4942 against 5810 / 5604, 12 qubits from the top 4984 against 5617; n =
// 25, 8 lane and warp bits: 67 against 73. Below n = 19 both take 16 to 20.
static bool marginal_walk(const qs_state *s, const MargP &p, MargWalkP *w) {
    std::memset(w, 0, sizeof(*w));
    uint64_t group = 0;
    for (int j = 0; j < p.m; ++j) {
        w->pos[j] = p.pos[j];
        group |= 1ull << p.pos[j];
    }
    w->m = p.m;
    w->ms = p.ms;
    w->lanes = (uint32_t)(group & 31u);
    int regs = 0;
    for (int b = 8; b < s->n; ++b) {
        if ((group >> b) & 1ull) w->high |= 1ull << b;
        else if (regs < 4) w->reg[regs++] = b;
        else w->rest |= 1ull << b, ++w->nrest;
    }
    w->lv = w->high ? std::min(4, __builtin_ctzll(w->high) - 8) : 4;
    w->chunks = s->n >= 12 ? 1ull << (s->n - 12) : 0;
    return regs == 4;
}

qs_status k_marginal(qs_state *s, const int *bitpos, int m, double *out_dev) {
    MargP p;
    std::memset(&p, 0, sizeof(p));
    for (int j = 0; j < m; ++j) p.pos[j] = bitpos[j];
    p.m = m;
    p.ms = s->ms;
    p.per = 1ull << s->n;
    const int bins = 1 << m;
    const uint64_t want = std::max<uint64_t>(1, p.per / (256 * 32));
    const int parts = (int)std::min<uint64_t>(want, (uint64_t)std::max(1, 4 * sms_of(s->device) / s->batch));
    // one part per member (large batches): the partial histograms are the
    // result, written straight into out_dev with no scratch; otherwise the
    // scratch holds batch * parts <= 4 x SMs histograms
    double *part = out_dev;
    if (parts > 1) {
        QS_TRY(ensure_scratch(s, (size_t)s->batch * parts * bins));
        part = s->scratch;
    }
    ProfScope _ps(s->stream, KC_REDUCE, (double)(s->batch * p.per) * (s->dtype == QS_C64 ? 8 : 16),
                  3.0 * s->batch * p.per);
    const dim3 grid((unsigned)parts, (unsigned)s->batch);
    MargWalkP w;
    if (marginal_walk(s, p, &w)) {
        const float2 *f = (const float2 *)s->data;
        if (s->dtype == QS_C128)
            marginal_walk_kernel<double, 4><<<grid, 256, 0, s->stream>>>((const double2 *)s->data, w, part);
        else if (w.lv == 4)
            marginal_walk_kernel<float, 4><<<grid, 256, 0, s->stream>>>(f, w, part);
        else if (w.lv == 3)
            marginal_walk_kernel<float, 3><<<grid, 256, 0, s->stream>>>(f, w, part);
        else if (w.lv == 2)
            marginal_walk_kernel<float, 2><<<grid, 256, 0, s->stream>>>(f, w, part);
        else if (w.lv == 1)
            marginal_walk_kernel<float, 1><<<grid, 256, 0, s->stream>>>(f, w, part);
        else
            marginal_walk_kernel<float, 0><<<grid, 256, 0, s->stream>>>(f, w, part);
    } else if (s->dtype == QS_C64) {
        marginal_partial_kernel<float><<<grid, 256, 0, s->stream>>>((const float2 *)s->data, p, part);
    } else {
        marginal_partial_kernel<double><<<grid, 256, 0, s->stream>>>((const double2 *)s->data, p, part);
    }
    QS_CUDA_TRY(cudaGetLastError());
    if (parts == 1) return QS_OK;
    const dim3 g2((unsigned)((bins + 31) / 32), (unsigned)s->batch);
    marginal_finalize_kernel<<<g2, 256, 0, s->stream>>>(s->scratch, parts, bins, out_dev);
    QS_CUDA_TRY(cudaGetLastError());
    return QS_OK;
}

// ------------------------------------------------------------------ sampling
constexpr int kSampleBlock = 4096;  // amplitudes per block of the prefix sums
constexpr int kScanChunk = 1024;    // block sums per CTA of the first scan level

constexpr int kSegs = 32;           // points of a block whose cumulative sums are kept (every 128 amplitudes)
constexpr int kGroups = kSampleBlock / 32;  // warp-wide groups of a block

// |a|^2 of the sampling kernels, rounded in one way: the walk must find the sums
// that block_sums_kernel formed for it
template <typename R> __device__ __forceinline__ R prob(V<R> a) { return fma(a.x, a.x, a.y * a.y); }

// sum of |psi|^2 over each block of L amplitudes (one CTA of 256 threads per
// block): per-thread sums in the state's precision, the block total in FP64.
// WHOLE (L = kSampleBlock): all 16 loads of a thread in flight, and the sum of
// every 32 consecutive amplitudes (a warp's load) goes to gsum, added up in the
// order of sample_kernel's warp scan (pairs, fours, ...: the order in which its
// last lane gathers them), 16 groups at a time: 16 shuffles for 16 sums.
// n = 27 complex64: 0.30 ms with the loads one after the other, without gsum.
template <typename R, bool WHOLE>
__global__ void __launch_bounds__(256) block_sums_kernel(const V<R> *__restrict__ q, uint64_t L,
                                                         double *__restrict__ bsum, R *__restrict__ gsum) {
    __shared__ double sh[8];
    const V<R> *b = q + (uint64_t)blockIdx.x * L;
    R acc = 0;
    if constexpr (WHOLE) {
        constexpr int N = kSampleBlock / 256;
        const int lane = threadIdx.x & 31;
        V<R> a[N];
#pragma unroll
        for (int j = 0; j < N; ++j) a[j] = b[threadIdx.x + 256 * j];
        R pr[N];
#pragma unroll
        for (int j = 0; j < N; ++j) pr[j] = prob<R>(a[j]);
#pragma unroll
        for (int j = 0; j < N; ++j) acc += pr[j];
        // level l: lanes that differ in bit l add up half of the groups each
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const bool up = (lane >> l) & 1;
#pragma unroll
            for (int j = 0; j < (N >> (l + 1)); ++j) {
                const int half = N >> (l + 1);
                const R mine = up ? pr[j + half] : pr[j], theirs = up ? pr[j] : pr[j + half];
                pr[j] = mine + __shfl_xor_sync(0xffffffffu, theirs, 1 << l);
            }
        }
        pr[0] += __shfl_xor_sync(0xffffffffu, pr[0], 16);
        // lane bits 0..3, from the top, are the group's number j
        const int j = ((lane & 1) << 3) | ((lane & 2) << 1) | ((lane & 4) >> 1) | ((lane & 8) >> 3);
        if (lane < 16) gsum[(uint64_t)blockIdx.x * kGroups + j * 8 + (threadIdx.x >> 5)] = pr[0];
    } else {
        for (uint64_t i = threadIdx.x; i < L; i += blockDim.x) {
            acc += prob<R>(b[i]);
        }
    }
    double d = (double)acc;
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        bsum[blockIdx.x] = t;
    }
}

// Cumulative sums inside a block, from its prefix on: seg[block * 32 + i] is the
// sum before amplitude 128 (i + 1), its groups of 32 added one after the other,
// as sample_kernel's walk adds them. One thread per block.
template <typename R>
__global__ void __launch_bounds__(128) segment_kernel(const R *__restrict__ gsum, const double *__restrict__ pre,
                                                      uint64_t nb, double *__restrict__ seg) {
    const uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    double running = pre[b];
    const R *g = gsum + b * kGroups;
    for (int i = 0; i < kSegs; i += 4) {
        R v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = g[i * 4 + j];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            running += (double)v[j];
            if (j % 4 == 3) seg[b * kSegs + i + j / 4] = running;
        }
    }
}

// exclusive prefix of v[0..count) within chunks of kScanChunk (one CTA each);
// the chunk's total goes to tot[chunk]
__global__ void __launch_bounds__(kScanChunk) scan_chunks_kernel(const double *__restrict__ v, uint64_t count,
                                                                 double *__restrict__ pre,
                                                                 double *__restrict__ tot) {
    __shared__ double sh[kScanChunk];
    const uint64_t i = (uint64_t)blockIdx.x * kScanChunk + threadIdx.x;
    const double x = i < count ? v[i] : 0.0;
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int o = 1; o < kScanChunk; o <<= 1) {  // inclusive Hillis-Steele scan
        const double t = threadIdx.x >= (unsigned)o ? sh[threadIdx.x - o] : 0.0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    if (i < count) pre[i] = sh[threadIdx.x] - x;
    if (threadIdx.x == kScanChunk - 1) tot[blockIdx.x] = sh[threadIdx.x];
}

// exclusive prefix of the chunk totals in place (one CTA; each thread a run)
__global__ void __launch_bounds__(kScanChunk) scan_totals_kernel(double *__restrict__ tot, uint64_t chunks) {
    __shared__ double sh[kScanChunk];
    const uint64_t per = (chunks + kScanChunk - 1) / kScanChunk;
    const uint64_t b = threadIdx.x * per, e = std::min<uint64_t>(b + per, chunks);
    double run = 0.0;
    for (uint64_t i = b; i < e; ++i) run += tot[i];
    sh[threadIdx.x] = run;
    __syncthreads();
    if (threadIdx.x == 0) {
        double acc = 0.0;
        const int used = (int)((chunks + per - 1) / per);  // threads with a run
        for (int t = 0; t < used; ++t) {
            const double r = sh[t];
            sh[t] = acc;
            acc += r;
        }
    }
    __syncthreads();
    double acc = sh[threadIdx.x];
    for (uint64_t i = b; i < e; ++i) {
        const double r = tot[i];
        tot[i] = acc;
        acc += r;
    }
}

__global__ void __launch_bounds__(kScanChunk) add_offsets_kernel(double *__restrict__ pre, uint64_t count,
                                                                 const double *__restrict__ tot) {
    const uint64_t i = (uint64_t)blockIdx.x * kScanChunk + threadIdx.x;
    if (i < count) pre[i] += tot[blockIdx.x];
}

// one warp per shot: the smallest x with cdf(x) > u * total. With seg, the walk
// starts at the block's first segment of 128 amplitudes that can hold it: 32
// points and a few groups are read instead of up to 4096 amplitudes (10^5 shots
// at n = 27 complex64: 2.2 ms without). Samples are the same either way: the points
// are the walk's own running sums (prob() and the order of a warp's scan in both), and a segment is passed over only if the
// walk could not have stopped in it (a group's scan exceeds its sum by 5
// roundings at most: 2^-17 of the segment is allowed here, and 2 roundings of
// the running sum).
template <typename R>
__global__ void __launch_bounds__(256) sample_kernel(const V<R> *__restrict__ q, const double *__restrict__ pre,
                                                     const double *__restrict__ bsum, const double *__restrict__ seg,
                                                     uint64_t nb, uint64_t L, const double *__restrict__ u,
                                                     uint64_t shots, unsigned long long *__restrict__ out) {
    const uint64_t w = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= shots) return;
    const int lane = threadIdx.x & 31;
    const double total = pre[nb - 1] + bsum[nb - 1];
    // a uniform outside [0, 1) is clamped: below 0 to 0, 1 or above (or NaN) to 1
    double uu = u[w];
    if (!(uu < 1.0)) uu = 1.0;
    if (uu < 0.0) uu = 0.0;
    const double target = uu * total;
    uint64_t lo = 0, hi = nb - 1;  // the last block whose exclusive prefix is <= target
    while (lo < hi) {
        const uint64_t mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= target) lo = mid;
        else hi = mid - 1;
    }
    // the prefix sums are monotone only up to rounding, so the search can end
    // in a block of zero probability: step back to the last block before it
    // that has some (its last nonzero outcome is then the sample)
    while (lo > 0 && !(bsum[lo] > 0.0)) --lo;
    const V<R> *b = q + lo * L;
    double running = pre[lo];
    uint64_t found = ~0ull, last_nz = lo * L, start = 0;
    if (seg) {
        const double end = seg[lo * kSegs + lane];
        double begin = __shfl_up_sync(0xffffffffu, end, 1);
        if (lane == 0) begin = running;
        const unsigned can = __ballot_sync(0xffffffffu, end + ((end - begin) * 0x1p-17 + end * 0x1p-51) > target);
        const int first = can ? __ffs(can) - 1 : kSegs;
        // no segment can: the walk only finds the block's last nonzero outcome
        if (first < kSegs) {
            start = (uint64_t)first * (kSampleBlock / kSegs);
            running = __shfl_sync(0xffffffffu, begin, first);
        }
    }
    for (int pass = 0; pass < 2; ++pass) {
        for (uint64_t c = start; c < L; c += 32) {
            R pr = 0;
            if (c + lane < L) pr = prob<R>(b[c + lane]);
            R sc = pr;  // inclusive warp scan
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const R t = __shfl_up_sync(0xffffffffu, sc, o);
                if (lane >= o) sc += t;
            }
            // only a lane of nonzero probability can be the sample: the scan's
            // rounding differs between lanes, so a zero lane after the target's
            // position can compare above it while the nonzero lane before did not
            const unsigned hit = __ballot_sync(0xffffffffu, pr > (R)0 && running + (double)sc > target);
            const unsigned nz = __ballot_sync(0xffffffffu, pr > (R)0);
            if (nz) last_nz = lo * L + c + (31 - __clz(nz));
            if (hit) {
                found = lo * L + c + (__ffs(hit) - 1);
                break;
            }
            running += (double)__shfl_sync(0xffffffffu, sc, 31);
        }
        // nothing from the start segment on: the block's last nonzero outcome
        // may lie before it
        if (found != ~0ull || start == 0) break;
        start = 0;
        running = pre[lo];
    }
    // the target lies at the block's end only through rounding: its last
    // outcome with nonzero probability
    if (lane == 0) out[w] = found != ~0ull ? found : last_nz;
}

template <typename R>
static qs_status sample_t(qs_state *s, const V<R> *q, uint64_t nb, uint64_t L, bool segments, const double *u_dev,
                          uint64_t shots, uint64_t *out_dev) {
    const uint64_t chunks = (nb + kScanChunk - 1) / kScanChunk;
    double *bsum = s->scratch, *pre = bsum + nb, *tot = pre + nb, *seg = tot + chunks;
    R *gsum = reinterpret_cast<R *>(seg + nb * kSegs);
    if (segments)
        block_sums_kernel<R, true><<<(unsigned)nb, 256, 0, s->stream>>>(q, L, bsum, gsum);
    else
        block_sums_kernel<R, false><<<(unsigned)nb, 256, 0, s->stream>>>(q, L, bsum, nullptr);
    QS_CUDA_TRY(cudaGetLastError());
    scan_chunks_kernel<<<(unsigned)chunks, kScanChunk, 0, s->stream>>>(bsum, nb, pre, tot);
    QS_CUDA_TRY(cudaGetLastError());
    scan_totals_kernel<<<1, kScanChunk, 0, s->stream>>>(tot, chunks);
    QS_CUDA_TRY(cudaGetLastError());
    add_offsets_kernel<<<(unsigned)chunks, kScanChunk, 0, s->stream>>>(pre, nb, tot);
    QS_CUDA_TRY(cudaGetLastError());
    if (segments) {
        segment_kernel<R><<<(unsigned)((nb + 127) / 128), 128, 0, s->stream>>>(gsum, pre, nb, seg);
        QS_CUDA_TRY(cudaGetLastError());
    }
    if (shots == 0) return QS_OK;
    const uint64_t blocks = (shots + 7) / 8;
    for (uint64_t b0 = 0; b0 < blocks; b0 += 1u << 30) {  // grid.x limit, in whole blocks
        const uint64_t nbk = std::min<uint64_t>(blocks - b0, 1u << 30);
        const uint64_t s0 = b0 * 8, ns = std::min<uint64_t>(shots - s0, nbk * 8);
        sample_kernel<R><<<(unsigned)nbk, 256, 0, s->stream>>>(q, pre, bsum, segments ? seg : nullptr, nb, L,
                                                               u_dev + s0, ns, (unsigned long long *)out_dev + s0);
        QS_CUDA_TRY(cudaGetLastError());
    }
    return QS_OK;
}

qs_status k_sample(qs_state *s, int member, const double *u_dev, uint64_t shots, uint64_t *out_dev) {
    const uint64_t per = 1ull << s->n;
    const uint64_t L = std::min<uint64_t>(per, kSampleBlock);
    const uint64_t nb = per / L;
    const uint64_t chunks = (nb + kScanChunk - 1) / kScanChunk;
    const size_t rsize = s->dtype == QS_C64 ? 4 : 8;
    const size_t base = (size_t)(2 * nb + chunks);
    // the points inside the blocks and the groups' sums: 24 bytes (complex128:
    // 40) for 128 amplitudes. Where no memory is left for them, every shot walks
    // its block from the start.
    bool segments = L == kSampleBlock;
    if (segments) {
        const qs_status st = ensure_scratch(s, base + nb * kSegs + nb * kGroups * rsize / sizeof(double));
        if (st == QS_ERR_OOM) {
            clear_error();
            segments = false;
        } else if (st != QS_OK) {
            return st;
        }
    }
    if (!segments) QS_TRY(ensure_scratch(s, base));
    // In complex128 the groups' sums are FP64 additions (2 per clock and SM) on top
    // of the blocks': few shots on a large state are faster without them, although
    // each then walks its block from the start (60 us alone, 0.044 us among many).
    // 1 / 1000 / 10^4 shots with and without: n = 24  196 199 226 | 247 327 816 us; n =
    // 26  600 602 630 | 568 577 1080; n = 28  2230 2230 2260 | 1770 1813 2258; n = 30
    // 8727 8726 8756 | 6714 6735 7211. complex64 has them in FP32 (n = 30, one shot:
    // 1.44 ms, 2.44 without).
    if (s->dtype == QS_C128 && nb >= (1u << 14) && shots < nb / 8) segments = false;
    ProfScope _ps(s->stream, KC_REDUCE, (double)per * (s->dtype == QS_C64 ? 8 : 16), 3.0 * per);
    const uint64_t moff = (uint64_t)member << s->ms;
    return s->dtype == QS_C64
               ? sample_t<float>(s, (const float2 *)s->data + moff, nb, L, segments, u_dev, shots, out_dev)
               : sample_t<double>(s, (const double2 *)s->data + moff, nb, L, segments, u_dev, shots, out_dev);
}

}  // namespace qsim
