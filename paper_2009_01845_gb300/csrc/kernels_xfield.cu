// Expectation of a transverse field, <psi| sum_q c_q X_q |psi> (Sec. 2.4,
// Energy callback): the X terms of an energy read-out, several per pass.
//
// X_q pairs the amplitudes whose indices differ in one bit, so its expectation
// is 2 c_q sum Re(conj(a) b) over those pairs: two FMAs per pair, and the
// state once through memory. One launch per term is bound by memory (a read of
// the state each, expect_partial_kernel). Here a CTA takes a tile of 2^12
// amplitudes and does every term whose bit is a tile bit: 16 amplitudes per
// thread, whose 4 register bits are the tile's bits 8..11 as loaded, then 4..7,
// then 0..3 after a read of the tile back from shared memory under another
// thread mapping (8 bytes written and read per amplitude and view; XOR swizzle,
// no bank conflicts). The first pass has the 12 lowest index bits in the tile;
// a later pass has the 4 lowest (whole 128-byte lines of complex64) and a
// window of 8 others: 12 + 8 per further pass, so 3 reads of the state for 27
// qubits instead of 27. Measured at n = 27, complex64 (1 GiB): 0.19 ms per pass
// (0.81 of the HBM peak), 0.59 ms for the field; one launch per term, 4.8 ms.
//
// Per thread the 16 products of a term are summed in the state's precision (8
// at a time) and added to a running sum that keeps what FP64 would: complex64
// sums the terms of 8 tiles exactly, as three floats, and adds those to an FP64
// sum (float_sum.cuh); an FP64 addition per term would take as long as the read
// of the state, and a pair of floats (0.56 ms at n = 27) holds 48 bits where FP64
// holds 53. FP64 across threads. A state of one tile (n = 12) has its complex64
// products added in FP64 one by one, as expect_partial_kernel does there: 26 us,
// 14 us in lumps of 16 products.
#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "float_sum.cuh"
#include "internal.h"
#include "prof.h"
#include "xfield.h"

namespace qsim {

namespace {

constexpr int kBits = 12;     // tile bits
constexpr int kThreads = 256; // 16 amplitudes per thread
constexpr int kPer = 16;
constexpr int kLow = 4;       // lowest bits every later tile keeps

template <typename R> struct XFieldP {
    R c[kBits];      // 2 c_q of the X on tile bit j, 0: none
    uint32_t active; // tile bits with a term
    int lo, w;       // tile bits 0..lo-1 are index bits 0..lo-1, the others index bits w, w+1, ...
    int ms;          // member shift
    uint64_t tiles;  // per member
    int accumulate;  // add to the partials instead of overwriting
};

template <typename R> struct RunningSum {
    R s = 0;
    __device__ __forceinline__ void add(R v) { s += v; }
    __device__ __forceinline__ void flush() {}
    __device__ __forceinline__ double value() const { return (double)s; }
};
template <> struct RunningSum<float> : FloatSum {};

// the terms on the 4 register bits of a[], which are tile bits b0 .. b0+3
template <typename R, bool WIDE>
__device__ __forceinline__ void view_terms(const V<R> *a, const XFieldP<R> &p, int b0, RunningSum<R> &acc) {
    R v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[j] = 0;
        if (!((p.active >> (b0 + j)) & 1u)) continue;
        const R c = p.c[b0 + j];
        V<R> s = mkc<R>(0, 0);  // products of the real and of the imaginary parts
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            if (r & (1 << j)) continue;
            const V<R> x = a[r], y = a[r | (1 << j)];
            if constexpr (WIDE) {
                acc.sum += (double)(c * fma(x.x, y.x, x.y * y.y));
            } else if constexpr (sizeof(R) == 4) {
                s = pfma(x, y, s);
            } else {
                s.x = fma(x.x, y.x, s.x);
                s.y = fma(x.y, y.y, s.y);
            }
        }
        if constexpr (sizeof(R) == 4) v[j] = __fmul_rn(c, s.x + s.y);  // rounded: not fused into add()'s sums
        else acc.add(c * (s.x + s.y));
    }
    if constexpr (sizeof(R) == 4 && !WIDE) acc.add(v);
}

template <typename R, bool WIDE>
__global__ void __launch_bounds__(kThreads, sizeof(R) == 4 ? 4 : 2)
    expect_xfield_kernel(const V<R> *__restrict__ psi, const __grid_constant__ XFieldP<R> p,
                         double2 *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V<R> *tile = reinterpret_cast<V<R> *>(smem_raw);
    __shared__ double sh[kThreads / 32];
    const uint32_t tid = threadIdx.x;
    const V<R> *q = psi + ((uint64_t)blockIdx.y << p.ms);
    const int gap = p.w - p.lo;  // outside bits between the low bits and the window
    const uint32_t lom = (1u << p.lo) - 1u;
    // index offsets of this thread's tile bits 0..7 and of register bit 0 (tile bit 8)
    const uint64_t toff = (uint64_t)(tid & lom) | ((uint64_t)(tid >> (p.lo < 8 ? p.lo : 8)) << p.w);
    const int cshift = p.lo >= 8 ? 8 : 8 - p.lo + p.w;
    RunningSum<R> acc;
    int tiles = 0;
    for (uint64_t t = blockIdx.x; t < p.tiles; t += gridDim.x) {
        const uint64_t base = ((t & ((1ull << gap) - 1ull)) << p.lo) | ((t >> gap) << (p.w + kBits - p.lo));
        const V<R> *src = q + (base | toff);
        V<R> a[kPer];
#pragma unroll
        for (int c = 0; c < kPer; ++c) a[c] = src[(uint64_t)c << cshift];
        if (p.active & 0xf00u) view_terms<R, WIDE>(a, p, 8, acc);
        if (p.active & 0x0ffu) {
            __syncthreads();  // the previous tile's readers are done
            // tile-local index l at position l ^ (bits 4..7 of l): both reads
            // below put the lanes of a wavefront on distinct banks
#pragma unroll
            for (int c = 0; c < kPer; ++c) tile[(c << 8) | (tid ^ ((tid >> 4) & 15u))] = a[c];
            __syncthreads();
            if (p.active & 0x0f0u) {
                const uint32_t row = (tid >> 4) << 8, col = tid & 15u;
#pragma unroll
                for (int c = 0; c < kPer; ++c) a[c] = tile[row | (c << 4) | (col ^ (uint32_t)c)];
                view_terms<R, WIDE>(a, p, 4, acc);
            }
            if (p.active & 0x00fu) {
                const uint32_t row = tid << 4, col = tid & 15u;
#pragma unroll
                for (int c = 0; c < kPer; ++c) a[c] = tile[row | ((uint32_t)c ^ col)];
                view_terms<R, WIDE>(a, p, 0, acc);
            }
        }
        if ((++tiles & 7) == 0) acc.flush();
    }
    acc.flush();
    double d = acc.value();
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    if ((tid & 31u) == 0) sh[tid >> 5] = d;
    __syncthreads();
    if (tid == 0) {
        double sum = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) sum += sh[w];
        double2 *slot = &part[(uint64_t)blockIdx.y * gridDim.x + blockIdx.x];
        if (p.accumulate)
            slot->x += sum;
        else
            *slot = make_double2(sum, 0.0);
    }
}

template <typename R>
qs_status xfield_t(const V<R> *psi, int n, int ms, int batch, const double *coeff, double2 *part, int blocks,
                   bool accumulate, cudaStream_t st) {
    constexpr size_t smem = sizeof(V<R>) << kBits;
    if (smem > 48 * 1024)
        QS_CUDA_TRY(cudaFuncSetAttribute(expect_xfield_kernel<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem));
    uint64_t left = 0;  // index bits with a term not yet done
    for (int b = 0; b < n; ++b)
        if (coeff[b] != 0.0) left |= 1ull << b;
    while (left) {
        XFieldP<R> p;
        std::memset(&p, 0, sizeof(p));
        const int b = __builtin_ctzll(left);
        p.lo = b < kBits ? kBits : kLow;
        p.w = b < kBits ? kBits : std::min(b, n - (kBits - kLow));
        for (int j = 0; j < kBits; ++j) {
            const int g = j < p.lo ? j : p.w + (j - p.lo);
            if (!((left >> g) & 1ull)) continue;
            p.c[j] = (R)(2.0 * coeff[g]);
            p.active |= 1u << j;
            left &= ~(1ull << g);
        }
        p.ms = ms;
        p.tiles = 1ull << (n - kBits);
        p.accumulate = accumulate ? 1 : 0;
        accumulate = true;
        if (prof_enabled()) {
            const double amps = (double)((uint64_t)batch << n);
            prof_add_work(KC_REDUCE, amps * sizeof(V<R>), 2.0 * amps * __builtin_popcount(p.active));
        }
        if constexpr (sizeof(R) == 4) {
            if (n == kBits)
                expect_xfield_kernel<R, true><<<dim3(blocks, batch), kThreads, smem, st>>>(psi, p, part);
            else
                expect_xfield_kernel<R, false><<<dim3(blocks, batch), kThreads, smem, st>>>(psi, p, part);
        } else {
            expect_xfield_kernel<R, false><<<dim3(blocks, batch), kThreads, smem, st>>>(psi, p, part);
        }
        QS_CUDA_TRY(cudaGetLastError());
    }
    return QS_OK;
}

}  // namespace

bool xfield_fits(int n, int terms) { return n >= kBits && terms >= 2; }

qs_status k_xfield(const void *psi, int n, int ms, int batch, qs_dtype dtype, const double *coeff, void *part,
                   int blocks, bool accumulate, cudaStream_t st) {
    return dtype == QS_C64 ? xfield_t<float>((const float2 *)psi, n, ms, batch, coeff, (double2 *)part, blocks,
                                             accumulate, st)
                           : xfield_t<double>((const double2 *)psi, n, ms, batch, coeff, (double2 *)part, blocks,
                                              accumulate, st);
}

}  // namespace qsim
