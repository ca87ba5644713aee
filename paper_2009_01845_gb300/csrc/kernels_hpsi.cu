// H psi for a Pauli sum H = sum_t c_t P_t (the adjoint gradient's costate seed
// and the exact solvers of Sec. 2.6): (P psi)[y] = i^{#Y} (-1)^{popcount((y ^
// m) & z)} psi[y ^ m] for a term with X mask m and Z mask z.
//
// The host sorts the terms by X mask into four kinds, each with its own loop:
//   * constant groups (no Z bits, a transverse field): partners are added up
//     (those that share one coefficient) or multiplied by a real constant;
//   * single-term strings: one real or imaginary coefficient whose sign is the
//     parity of a thread part (once per string) and a chunk part (uniform);
//   * the Z-only group: its terms of weight <= 2 are an Ising energy, split
//     over the bits outside the tile (fields, per tile), the thread bits (pair
//     energies, once per launch by a Walsh-Hadamard transform over the CTA's
//     threads) and the chunk bits; the others by their parities per chunk mask
//     and a small transform;
//   * the rest (several strings on one X mask): parities per output.
//
// A CTA takes tiles of 2^(TB + PB) consecutive amplitudes: 2^TB threads, 2^PB
// outputs each. Partners inside the tile come from shared memory, the others
// from L2 or DRAM, at constant offsets from one address where the mask has no
// chunk bit, so that a group's loads (and the next group's) are in flight
// together. What the solvers do with H psi next (a Taylor term and its sum, a
// Runge-Kutta stage and the gathered result) is done before it is stored: up
// to two combinations base + c (H psi) per application.
//
// Bound by the partner reads (at n = 24 complex64 an application reads 20
// partners per amplitude from L2 and DRAM, 2.7 GB, 7 TB/s) and, for complex128,
// by splitting them. Measured with a transverse field, 276 pairs, 24 fields and
// 8 strings: n = 24 complex64 0.37 ms with both results (one kernel per
// application without them and separate combinations: 0.74 + 0.13 ms); n = 16
// complex128 18 us (81 us on 32 CTAs, plus 4 us of combinations).
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <utility>
#include <vector>

#include "device.cuh"
#include "hpsi.h"
#include "prof.h"

namespace qsim {

namespace {

constexpr int kMaxGroups = 64;  // of each kind, per launch
constexpr int kMaxTerms = 384;  // of the Z-only and the remaining groups, per launch

template <typename R> struct HpsiP {
    static constexpr int kOutputs = sizeof(R) == 4 ? 16 : 8;  // per thread, at most
    // constant groups: [0, run_in) and [run_in, run0) share one coefficient
    // (partners inside and outside the tile), then [run0, c_in), [c_in, nc)
    int nc, run_in, run0, c_in;
    uint64_t cx[kMaxGroups];
    R cc[kMaxGroups];
    // single-term strings: [0, s_in) with partners inside the tile
    int ns, s_in;
    uint64_t sx[kMaxGroups], sz[kMaxGroups];
    R sc[kMaxGroups];
    uint8_t sim[kMaxGroups];  // the coefficient is i sc
    // remaining groups: terms [gbeg[g], gbeg[g + 1])
    int ng;
    uint64_t gx[kMaxGroups];
    int gbeg[kMaxGroups + 1];
    R cre[kMaxTerms], cim[kMaxTerms];
    uint64_t zb[kMaxTerms];
    // Z-only group (its terms follow the groups' in cre/zb): dord[dmb[m] ..
    // dmb[m + 1]) are those whose chunk bits are m, without the Ising ones
    int diag;
    uint16_t dord[kMaxTerms];
    int dmb[kOutputs + 1];
    // Ising energy qc0 + sum_i qh[i] z_i + sum_{i<j} qJ[i][j] z_i z_j in index
    // bits (z_i = 1 - 2 y_i; qJ symmetric, zero diagonal); qecc: the chunk bits' pairs
    int quad;
    R qc0;
    R qh[32];
    R qJ[32][32];
    R qecc[kOutputs];
    int n, ms;
    uint64_t total;
    const void *part;  // partial sums of earlier launches, or null
    // results: out = base + c h, or c h where base is null; c as (re, im)
    void *out[2];
    const void *base[2];
    R ere[2], eim[2];
};

static_assert(sizeof(HpsiP<double>) <= 32700, "H psi parameters exceed the parameter space");

// Amplitude arithmetic A of the tile kernel: the state's own (complex64), or
// double-float for complex128 (loads split, stores joined; coefficients in R,
// converted per use).
template <typename A, typename R> __device__ __forceinline__ V<A> amp_in(const V<R> *p, uint64_t i) {
    if constexpr (is_dd<A>) {
        const double2 v = p[i];
        return mkc<dd>(dd(v.x), dd(v.y));
    } else {
        return p[i];
    }
}
template <typename A, typename R> __device__ __forceinline__ void amp_out(V<R> *p, uint64_t i, V<A> v) {
    if constexpr (is_dd<A>)
        p[i] = make_double2(to_double(re_of<dd>(v)), to_double(im_of<dd>(v)));
    else
        p[i] = v;
}
template <typename A, typename R> __device__ __forceinline__ V<A> coef(R re, R im) { return mkc<A>(A(re), A(im)); }
template <typename A> __device__ __forceinline__ V<A> cadd(V<A> a, V<A> b) {
    if constexpr (is_dd<A>)
        return dd_cadd(a, b);
    else
        return mkc<A>(a.x + b.x, a.y + b.y);
}
// acc + c v for a real c
template <typename A> __device__ __forceinline__ V<A> rmadd(A c, V<A> v, V<A> acc) {
    if constexpr (is_dd<A>)
        return dd_fma_c2(c, v, acc);
    else
        return mkc<A>(fma(c, v.x, acc.x), fma(c, v.y, acc.y));
}
// i v
template <typename A> __device__ __forceinline__ V<A> mul_i(V<A> v) {
    if constexpr (is_dd<A>) {
        V<A> r;
        r.h = make_float2(-v.h.y, v.h.x);
        r.l = make_float2(-v.l.y, v.l.x);
        return r;
    } else {
        return mkc<A>(-v.y, v.x);
    }
}

template <typename A, typename R>
__device__ __forceinline__ void results(const HpsiP<R> &p, uint64_t i, V<A> h) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        if (!p.out[e]) continue;
        V<A> v = h;
        if (p.base[e])
            v = cmadd<A>(coef<A, R>(p.ere[e], p.eim[e]), h, amp_in<A, R>((const V<R> *)p.base[e], i));
        else if (p.ere[e] != (R)1 || p.eim[e] != (R)0)
            v = cmul<A>(coef<A, R>(p.ere[e], p.eim[e]), h);
        amp_out<A, R>((V<R> *)p.out[e], i, v);
    }
}

// One thread per output, any n: states below a tile (complex128 there in FP64,
// as its gates are) and above 32 index bits.
template <typename R>
__global__ void __launch_bounds__(256) hpsi_kernel(const V<R> *__restrict__ src, const __grid_constant__ HpsiP<R> p) {
    const uint64_t mask = (1ull << p.n) - 1ull;
    for (uint64_t i = global_tid(); i < p.total; i += global_stride()) {
        const uint64_t y = i & mask, m0 = (i >> p.n) << p.ms;
        const V<R> *sm = src + m0;
        V<R> acc = p.part ? ((const V<R> *)p.part)[m0 | y] : mkc<R>(0, 0);
        for (int g = 0; g < p.nc; ++g) acc = rmadd<R>(p.cc[g], sm[y ^ p.cx[g]], acc);
        for (int g = 0; g < p.ns; ++g) {
            const uint64_t x = y ^ p.sx[g];
            const R c = (__popcll(x & p.sz[g]) & 1) ? -p.sc[g] : p.sc[g];
            const V<R> v = sm[x];
            acc = rmadd<R>(c, p.sim[g] ? mul_i<R>(v) : v, acc);
        }
        for (int g = 0; g < p.ng + (p.diag ? 1 : 0); ++g) {
            const uint64_t x = y ^ (g < p.ng ? p.gx[g] : 0ull);
            R fr = 0, fi = 0;
            for (int t = p.gbeg[g]; t < p.gbeg[g + 1]; ++t) {
                const bool odd = __popcll(x & p.zb[t]) & 1;
                fr += odd ? -p.cre[t] : p.cre[t];
                fi += odd ? -p.cim[t] : p.cim[t];
            }
            acc = cmadd<R>(mkc<R>(fr, fi), sm[x], acc);
        }
        results<R, R>(p, m0 | y, acc);
    }
}

// The tile kernel's shapes: TB thread bits, PB chunk bits, CTAs per SM the
// registers are capped for.
template <typename R, typename A, int TB, int PB, int MINB>
__global__ void __launch_bounds__(1 << TB, MINB) hpsi_tile_kernel(const V<R> *__restrict__ src,
                                                                  const __grid_constant__ HpsiP<R> p) {
    constexpr int T = 1 << TB, PER = 1 << PB, K = TB + PB;
    // groups whose loads are in flight together (8 double-float partners take 32 registers)
    constexpr int U = PB >= 3 ? (is_dd<A> ? 1 : 2) : PB == 2 ? 4 : 8;
    __shared__ V<A> tile[1 << K];
    __shared__ R s_w[T];  // transform over the thread bits
    __shared__ R s_f[K];  // Ising fields of the outside bits on the tile bits
    __shared__ R s_eout;  // the outside bits' own energy
    const uint32_t tid = threadIdx.x;
    // once per launch: the thread bits' pair energy, and their fields on the chunk bits
    R e_bb = 0, g_b[PB > 0 ? PB : 1];
    if (p.quad) {
        if (__popc(tid) == 2) e_bb = p.qJ[__ffs(tid) - 1][31 - __clz(tid)];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const R u = __shfl_xor_sync(0xffffffffu, e_bb, o);
            e_bb = (tid & o) ? u - e_bb : e_bb + u;
        }
        for (int o = 32; o < T; o <<= 1) {
            __syncthreads();
            s_w[tid] = e_bb;
            __syncthreads();
            const R u = s_w[tid ^ o];
            e_bb = (tid & o) ? u - e_bb : e_bb + u;
        }
#pragma unroll
        for (int j = 0; j < PB; ++j) {
            R f = 0;
#pragma unroll
            for (int i = 0; i < TB; ++i) f += ((tid >> i) & 1u) ? -p.qJ[TB + j][i] : p.qJ[TB + j][i];
            g_b[j] = f;
        }
    }
    const uint64_t tiles = p.total >> K;
    const int tshift = p.n - K;  // tiles per member: 2^tshift
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint64_t moff = (t >> tshift) << p.ms;
        const uint32_t yb = (uint32_t)((t & ((1ull << tshift) - 1ull)) << K) | tid;  // output j: yb + T j
        const V<R> *sm = src + moff;
        V<A> own[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) own[j] = amp_in<A, R>(sm + yb, T * j);
        __syncthreads();  // the previous tile's readers are done
        if (p.quad) {
            // warp 0: the outside bits' fields on tile bit j (lanes j < K);
            // warp 1: the outside energy, one outside bit per lane, summed
            const int lane = tid & 31, warp = tid >> 5;
            if (warp == 0 && lane < K) {
                R f = p.qh[lane];
                for (int i = K; i < p.n; ++i) f += ((yb >> i) & 1u) ? -p.qJ[lane][i] : p.qJ[lane][i];
                s_f[lane] = f;
            } else if (warp == 1) {
                R u = 0;
                const int i = K + lane;
                if (i < p.n) {
                    R half = 0;
                    for (int j = K; j < p.n; ++j) half += ((yb >> j) & 1u) ? -p.qJ[i][j] : p.qJ[i][j];
                    u = (((yb >> i) & 1u) ? R(-1) : R(1)) * (p.qh[i] + R(0.5) * half);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
                if (lane == 0) s_eout = p.qc0 + u;
            }
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) tile[tid + T * j] = own[j];
        __syncthreads();
        V<A> acc[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j)
            acc[j] = p.part ? amp_in<A, R>((const V<R> *)p.part + moff + yb, T * j) : coef<A, R>(0, 0);
        // partners of X mask m: inside the tile, or at constant offsets from one
        // address where m has no chunk bit
        auto inside = [&](uint32_t m, V<A> *v) {
            const uint32_t mj = m >> TB, x = tid ^ (m & (T - 1));
#pragma unroll
            for (int j = 0; j < PER; ++j) v[j] = tile[x | ((j ^ mj) << TB)];
        };
        auto outside = [&](uint32_t m, V<A> *v) {
            if (((m >> TB) & (PER - 1)) == 0) {
                const V<R> *q = sm + (yb ^ m);
#pragma unroll
                for (int j = 0; j < PER; ++j) v[j] = amp_in<A, R>(q, T * j);
            } else {
#pragma unroll
                for (int j = 0; j < PER; ++j) v[j] = amp_in<A, R>(sm, (yb | (T * j)) ^ m);
            }
        };
        // constant groups: the run with one coefficient, then the others
        for (int g = 0; g < p.run_in; ++g) {
            V<A> v[PER];
            inside((uint32_t)p.cx[g], v);
#pragma unroll
            for (int j = 0; j < PER; ++j) acc[j] = cadd<A>(acc[j], v[j]);
        }
#pragma unroll U
        for (int g = p.run_in; g < p.run0; ++g) {
            V<A> v[PER];
            outside((uint32_t)p.cx[g], v);
#pragma unroll
            for (int j = 0; j < PER; ++j) acc[j] = cadd<A>(acc[j], v[j]);
        }
        if (p.run0 > 0) {
            const A c = A(p.cc[0]);
#pragma unroll
            for (int j = 0; j < PER; ++j) acc[j] = rmadd<A>(c, acc[j], coef<A, R>(0, 0));
        }
        for (int g = p.run0; g < p.nc; ++g) {
            V<A> v[PER];
            if (g < p.c_in) inside((uint32_t)p.cx[g], v);
            else outside((uint32_t)p.cx[g], v);
            const A c = A(p.cc[g]);
#pragma unroll
            for (int j = 0; j < PER; ++j) acc[j] = rmadd<A>(c, v[j], acc[j]);
        }
        // single-term strings
        auto string = [&](int g, const V<A> *v) {
            const uint32_t m = (uint32_t)p.sx[g], z = (uint32_t)p.sz[g];
            const bool base = __popc((yb ^ m) & z) & 1;  // output 0's sign
            const uint32_t zj = (z >> TB) & (PER - 1);
            const A c = base ? -A(p.sc[g]) : A(p.sc[g]);
            const A d = -c;
            if (p.sim[g]) {
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    acc[j] = rmadd<A>((__popc(j & zj) & 1) ? d : c, mul_i<A>(v[j]), acc[j]);
            } else {
#pragma unroll
                for (int j = 0; j < PER; ++j) acc[j] = rmadd<A>((__popc(j & zj) & 1) ? d : c, v[j], acc[j]);
            }
        };
        for (int g = 0; g < p.s_in; ++g) {
            V<A> v[PER];
            inside((uint32_t)p.sx[g], v);
            string(g, v);
        }
#pragma unroll U
        for (int g = p.s_in; g < p.ns; ++g) {
            V<A> v[PER];
            outside((uint32_t)p.sx[g], v);
            string(g, v);
        }
        // Z-only group: the terms' signs outside the chunk summed per chunk mask,
        // a transform over the chunk bits, and the Ising energy
        if (p.diag) {
            R D[PER];
#pragma unroll
            for (int m = 0; m < PER; ++m) {
                R a = 0;
                for (int k = p.dmb[m]; k < p.dmb[m + 1]; ++k) {
                    const int tt = p.dord[k];
                    a += (__popc(yb & (uint32_t)p.zb[tt]) & 1) ? -p.cre[tt] : p.cre[tt];
                }
                D[m] = a;
            }
#pragma unroll
            for (int h = 1; h < PER; h <<= 1)
#pragma unroll
                for (int i = 0; i < PER; ++i)
                    if (!(i & h)) {
                        const R u = D[i], v = D[i | h];
                        D[i] = u + v;
                        D[i | h] = u - v;
                    }
            if (p.quad) {
                R e0 = s_eout + e_bb;
#pragma unroll
                for (int i = 0; i < TB; ++i) e0 += ((tid >> i) & 1u) ? -s_f[i] : s_f[i];
#pragma unroll
                for (int c = 0; c < PER; ++c) {
                    R e = e0 + p.qecc[c];
#pragma unroll
                    for (int j = 0; j < PB; ++j) {
                        const R f = s_f[TB + j] + g_b[j];
                        e += ((c >> j) & 1) ? -f : f;
                    }
                    D[c] += e;
                }
            }
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                // (read back where registers are short)
                const V<A> v = is_dd<A> && PB >= 3 ? tile[tid + T * j] : own[j];
                acc[j] = rmadd<A>(A(D[j]), v, acc[j]);
            }
        }
        // remaining groups
        for (int g = 0; g < p.ng; ++g) {
            const uint32_t m = (uint32_t)p.gx[g];
            V<A> v[PER];
            if (m >> K) outside(m, v);
            else inside(m, v);
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const uint32_t x = (yb | (T * j)) ^ m;
                R fr = 0, fi = 0;
                for (int tt = p.gbeg[g]; tt < p.gbeg[g + 1]; ++tt) {
                    const bool odd = __popc(x & (uint32_t)p.zb[tt]) & 1;
                    fr += odd ? -p.cre[tt] : p.cre[tt];
                    fi += odd ? -p.cim[tt] : p.cim[tt];
                }
                acc[j] = cmadd<A>(coef<A, R>(fr, fi), v[j], acc[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) results<A, R>(p, moff + yb + T * j, acc[j]);
    }
}

// Thread and chunk bits for `total` outputs of n bits per member; tb = 0: one
// thread per output. Large tiles keep more partners in shared memory and walk
// the groups for more outputs at once; small ones give small states enough
// CTAs (2^16 amplitudes are 256 tiles of 2^8, 16 of 2^12). Microseconds per
// application (transverse field, dense Ising, 8 strings, Runge-Kutta's two
// results) with 1, 4, 8 outputs per thread in complex64, at n = 16, 18, 20, 22, 24:
//   7.9  13.6  33.5  151  596 | 11.6  12.7  26.6  103  495 | 16.4  16.7  23.0   87   385
// and of a Runge-Kutta step in complex128 (field, all pairs, 8 strings) with 1 (n =
// 18), 2 (20) or 4 (22, 25) outputs against 8: 373 364, 733 687, 2307 1973 us, 18.2 15.0 ms.
// What moves the lines: Z-only strings of weight > 2 (`strings`) are summed per
// chunk mask, so more outputs per thread share a string's sign, and in complex128
// each is an FP64 addition. The same step with 250 of them, 1 output (or 2) against
// 8: n = 16  618 554, n = 17  940 558, n = 18  1556 568, n = 20  2627 1175; with 8 / 32 /
// 64 of them at n = 18: 352 345, 458 363, 621 391; with 32 / 64 at n = 17: 336 354, 413
// 386. Terms with X and Z bits (`mixed`) go the other way in a state of few tiles: n =
// 17, 40 strings, 0 / 24 / 60 of them, 399 371, 440 490, 530 636. So do X masks with
// several strings (`several` terms), per output and in FP64: a Heisenberg chain in a
// field, 2 (n = 19, 20) and 4 outputs against 8: 938 1125, 1735 2181, n = 22  7334 7830,
// n = 25  63.0 67.0 ms. complex64, 8 outputs of 512 threads against 16 of 256: n = 25,
// 0 / 80 / 120 / 250 strings, 3.02 3.65, 3.64 3.98, 3.97 4.03, 5.41 4.47 ms (Dormand-Prince
// 6.70 6.53, 7.20 6.63, 9.49 7.37); n = 19 from 4 outputs, 100 / 250 strings, 293 300,
// 436 392 us.
struct Shape {
    int tb = 0, pb = 0;
};
Shape shape_for(qs_dtype dtype, int n, uint64_t total, const qs_pauli_term *terms, size_t count) {
    if (n > 32) return {};
    size_t strings = 0, mixed = 0;
    for (size_t t = 0; t < count; ++t) {
        strings += terms[t].x_mask == 0 && __builtin_popcountll(terms[t].z_mask) > 2;
        mixed += terms[t].x_mask != 0 && terms[t].z_mask != 0;
    }
    if (dtype == QS_C64) {
        if (n >= 12 && total >= (1ull << 19) && strings >= 100) return {8, 4};
        if (n >= 12 && total >= (1ull << 20)) return {9, 3};
        if (n >= 10 && total >= (1ull << 18)) return {8, 2};
        return n >= 8 ? Shape{8, 0} : Shape{};
    }
    // below 11 qubits complex128 stays in FP64
    if (n < 11) return {};
    const uint64_t t16 = std::min<uint64_t>(total >> 16, 8);
    if (t16 == 8 || t16 * t16 * strings >= 160 + 4 * mixed) {
        std::vector<std::pair<uint64_t, bool>> x;  // X masks, and whether the term has Z bits
        for (size_t t = 0; t < count && mixed > 0; ++t)
            if (terms[t].x_mask) x.push_back({terms[t].x_mask, terms[t].z_mask != 0});
        std::sort(x.begin(), x.end());
        size_t several = 0;
        for (size_t i = 0, j; i < x.size(); i = j) {
            for (j = i; j < x.size() && x[j].first == x[i].first; ++j) {}
            if (j - i > 1 && x[j - 1].second) several += j - i;
        }
        if (several <= strings) return {8, 3};
    }
    if (total >= (1ull << 21)) return {9, 2};
    if (total >= (1ull << 19)) return {8, 1};
    return {8, 0};
}

uint64_t reversed(uint64_t mask, int n) {
    uint64_t r = 0;
    for (; mask; mask &= mask - 1) r |= 1ull << (n - 1 - __builtin_ctzll(mask));
    return r;
}

}  // namespace

struct HpsiOp::Impl {
    StateView shape;
    Shape tile;
    double terms = 0;
    std::vector<HpsiP<float>> f;
    std::vector<HpsiP<double>> d;
};

namespace {

// the terms of one X mask
struct Group {
    uint64_t x = 0;
    std::vector<int> t;
    bool constant = true;  // no Z bits
    double c = 0.0;        // constant: the coefficient
};

template <typename R>
qs_status prepare_t(const StateView &s, const Shape &shape, const qs_pauli_term *terms, size_t count,
                    std::vector<HpsiP<R>> *out) {
    const int n = s.n, K = shape.tb + shape.pb;
    const uint64_t total = (uint64_t)s.batch << n;
    std::vector<Group> groups;
    std::vector<uint64_t> zb(count);
    for (size_t t = 0; t < count; ++t) {
        const uint64_t x = reversed(terms[t].x_mask, n);
        zb[t] = reversed(terms[t].z_mask, n);
        size_t g = 0;
        while (g < groups.size() && groups[g].x != x) ++g;
        if (g == groups.size()) {
            groups.emplace_back();
            groups.back().x = x;
        }
        groups[g].t.push_back((int)t);
        groups[g].c += terms[t].coeff;
        if (zb[t]) groups[g].constant = false;
    }
    auto outside = [&](uint64_t x) { return K > 0 && (x >> K) != 0; };
    // constant groups: the coefficient shared by most of them leads
    std::vector<const Group *> cst, str, rest;
    const Group *diag = nullptr;
    for (const Group &g : groups) {
        if (g.constant)
            cst.push_back(&g);
        else if (g.x == 0)
            diag = &g;
        else
            (g.t.size() == 1 ? str : rest).push_back(&g);
    }
    double lead = 0.0;
    size_t lead_n = 0;
    for (const Group *a : cst) {
        if (a->x == 0) continue;
        size_t k = 0;
        for (const Group *b : cst) k += b->x != 0 && (R)b->c == (R)a->c;
        if (k > lead_n) {
            lead_n = k;
            lead = a->c;
        }
    }
    // a run of one saves nothing, and a zero coefficient would lose what it multiplies
    const bool run = lead_n >= 2 && K > 0;
    auto rank = [&](const Group *g) {
        const bool in_run = run && g->x != 0 && (R)g->c == (R)lead;
        return (in_run ? 0 : 2) + (outside(g->x) ? 1 : 0);
    };
    std::stable_sort(cst.begin(), cst.end(), [&](const Group *a, const Group *b) { return rank(a) < rank(b); });
    std::stable_sort(str.begin(), str.end(),
                     [&](const Group *a, const Group *b) { return outside(a->x) < outside(b->x); });
    // real and imaginary part of a term's coefficient c i^{#Y}
    auto parts = [&](int t, double *re, double *im) {
        const int ny = __builtin_popcountll(terms[t].x_mask & terms[t].z_mask) & 3;
        const double c = terms[t].coeff;
        *re = ny == 0 ? c : ny == 2 ? -c : 0.0;
        *im = ny == 1 ? c : ny == 3 ? -c : 0.0;
    };
    for (const Group &g : groups)
        if (g.t.size() > (size_t)kMaxTerms) {
            set_error("a Pauli group has more than %d terms", kMaxTerms);
            return QS_ERR_UNSUPPORTED;
        }
    size_t ic = 0, is = 0, ir = 0;
    bool diag_left = diag != nullptr;
    do {
        out->emplace_back();
        HpsiP<R> &p = out->back();
        std::memset(&p, 0, sizeof(p));
        p.n = n;
        p.ms = s.ms;
        p.total = total;
        const bool first = out->size() == 1;
        for (; ic < cst.size() && p.nc < kMaxGroups; ++ic, ++p.nc) {
            const int rk = rank(cst[ic]);
            p.cx[p.nc] = cst[ic]->x;
            p.cc[p.nc] = (R)cst[ic]->c;
            // the run is multiplied once, before anything else is added: first launch only
            if (first && rk == 0) p.run_in = p.nc + 1;
            if (first && rk <= 1) p.run0 = p.nc + 1;
        }
        p.c_in = p.run0;
        while (p.c_in < p.nc && !outside(p.cx[p.c_in])) ++p.c_in;
        for (; is < str.size() && p.ns < kMaxGroups; ++is, ++p.ns) {
            const int t = str[is]->t[0];
            double re, im;
            parts(t, &re, &im);
            p.sx[p.ns] = str[is]->x;
            p.sz[p.ns] = zb[t];
            p.sim[p.ns] = im != 0.0;
            p.sc[p.ns] = (R)(im != 0.0 ? im : re);
            if (!outside(str[is]->x)) p.s_in = p.ns + 1;
        }
        int nt = 0;
        for (; ir < rest.size() && p.ng < kMaxGroups && nt + (int)rest[ir]->t.size() <= kMaxTerms; ++ir, ++p.ng) {
            p.gx[p.ng] = rest[ir]->x;
            p.gbeg[p.ng] = nt;
            for (int t : rest[ir]->t) {
                double re, im;
                parts(t, &re, &im);
                p.cre[nt] = (R)re;
                p.cim[nt] = (R)im;
                p.zb[nt++] = zb[t];
            }
        }
        p.gbeg[p.ng] = nt;
        if (diag_left && nt + (int)diag->t.size() <= kMaxTerms && p.ng < kMaxGroups) {
            diag_left = false;
            p.diag = 1;
            const int d0 = nt;
            for (int t : diag->t) {
                p.cre[nt] = (R)terms[t].coeff;
                p.zb[nt++] = zb[t];
            }
            p.gbeg[p.ng + 1] = nt;
            if (K > 0) {
                std::vector<double> h(32, 0.0), J(32 * 32, 0.0);
                double c0 = 0.0;
                std::vector<char> ising(nt, 0);
                for (int i = d0; i < nt; ++i) {
                    const uint64_t z = p.zb[i];
                    const double c = terms[diag->t[i - d0]].coeff;
                    const int w = __builtin_popcountll(z);
                    if (w > 2) continue;
                    ising[i] = 1;
                    p.quad = 1;
                    const int a = w ? __builtin_ctzll(z) : 0, b = w ? 63 - __builtin_clzll(z) : 0;
                    if (w == 0) c0 += c;
                    else if (w == 1) h[a] += c;
                    else J[a * 32 + b] += c, J[b * 32 + a] += c;
                }
                p.qc0 = (R)c0;
                for (int i = 0; i < 32; ++i) {
                    p.qh[i] = (R)h[i];
                    for (int j = 0; j < 32; ++j) p.qJ[i][j] = (R)J[i * 32 + j];
                }
                const int pb = shape.pb, tb = shape.tb;
                for (int c = 0; c < (1 << pb); ++c) {
                    double e = 0.0;
                    for (int i = 0; i < pb; ++i)
                        for (int j = i + 1; j < pb; ++j)
                            e += ((((c >> i) ^ (c >> j)) & 1) ? -1.0 : 1.0) * J[(tb + i) * 32 + tb + j];
                    p.qecc[c] = (R)e;
                }
                int k = 0;
                for (int m = 0; m < (1 << pb); ++m) {
                    p.dmb[m] = k;
                    for (int i = d0; i < nt; ++i)
                        if (!ising[i] && (int)((p.zb[i] >> tb) & ((1u << pb) - 1u)) == m) p.dord[k++] = (uint16_t)i;
                }
                p.dmb[1 << pb] = k;
            }
        }
    } while (ic < cst.size() || is < str.size() || ir < rest.size() || diag_left);
    return QS_OK;
}

int sm_count_hpsi() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

template <typename R, typename A, int TB, int PB, int MINB>
void launch_tile(const V<R> *src, const HpsiP<R> &p, cudaStream_t st) {
    const uint64_t tiles = p.total >> (TB + PB);
    const unsigned grid = (unsigned)std::min<uint64_t>(tiles, (uint64_t)sm_count_hpsi() * MINB);
    hpsi_tile_kernel<R, A, TB, PB, MINB><<<grid, 1 << TB, 0, st>>>(src, p);
}

template <typename R>
qs_status launch_t(const Shape &shape, const V<R> *src, const HpsiP<R> &p, cudaStream_t st) {
    if (shape.tb == 0) {
        const uint64_t blocks = std::min<uint64_t>((p.total + 255) / 256, (uint64_t)sm_count_hpsi() * 32);
        hpsi_kernel<R><<<(unsigned)std::max<uint64_t>(1, blocks), 256, 0, st>>>(src, p);
    } else if constexpr (sizeof(R) == 4) {
        if (shape.pb == 4) launch_tile<float, float, 8, 4, 2>(src, p, st);
        else if (shape.pb == 3) launch_tile<float, float, 9, 3, 2>(src, p, st);
        else if (shape.pb == 2) launch_tile<float, float, 8, 2, 4>(src, p, st);
        else launch_tile<float, float, 8, 0, 6>(src, p, st);
    } else {
        if (shape.pb == 3) launch_tile<double, dd, 8, 3, 2>(src, p, st);
        else if (shape.pb == 2) launch_tile<double, dd, 9, 2, 1>(src, p, st);
        else if (shape.pb == 1) launch_tile<double, dd, 8, 1, 3>(src, p, st);
        else launch_tile<double, dd, 8, 0, 4>(src, p, st);
    }
    QS_CUDA_TRY(cudaGetLastError());
    return QS_OK;
}

template <typename R>
qs_status apply_t(const Shape &shape, const std::vector<HpsiP<R>> &blocks, const StateView &src, const HpsiOut *o,
                  void *spare, cudaStream_t st) {
    for (size_t i = 0; i < blocks.size(); ++i) {
        static thread_local HpsiP<R> p;
        std::memcpy(&p, &blocks[i], sizeof(p));
        p.ms = src.ms;
        p.part = i > 0 ? spare : nullptr;
        if (i + 1 < blocks.size()) {
            p.out[0] = spare;
            p.ere[0] = 1;
        } else {
            for (int e = 0; e < 2; ++e) {
                p.out[e] = o[e].out;
                p.base[e] = o[e].base;
                p.ere[e] = (R)o[e].c.real();
                p.eim[e] = (R)o[e].c.imag();
            }
        }
        QS_TRY(launch_t<R>(shape, (const V<R> *)src.data, p, st));
    }
    return QS_OK;
}

}  // namespace

qs_status hpsi_prepare(const StateView &s, const qs_pauli_term *terms, size_t count, HpsiOp *op) {
    op->impl = std::make_shared<HpsiOp::Impl>();
    HpsiOp::Impl &im = *op->impl;
    im.shape = s;
    im.tile = shape_for(s.dtype, s.n, (uint64_t)s.batch << s.n, terms, count);
    im.terms = (double)count;
    return s.dtype == QS_C64 ? prepare_t<float>(s, im.tile, terms, count, &im.f)
                             : prepare_t<double>(s, im.tile, terms, count, &im.d);
}

qs_status hpsi_apply(const HpsiOp &op, const StateView &src, const HpsiOut &a, const HpsiOut &b, void *spare,
                     cudaStream_t st) {
    const HpsiOp::Impl &im = *op.impl;
    const double total = (double)((uint64_t)src.batch << src.n);
    const double states = 1.0 + (a.out != nullptr) + (a.base != nullptr) + (b.out != nullptr) + (b.base != nullptr);
    ProfScope _ps(st, KC_HPSI, states * total * (src.dtype == QS_C64 ? 8 : 16), 8.0 * total * im.terms);
    const HpsiOut o[2] = {a, b};
    return src.dtype == QS_C64 ? apply_t<float>(im.tile, im.f, src, o, spare, st)
                               : apply_t<double>(im.tile, im.d, src, o, spare, st);
}

qs_status k_pauli_apply(const StateView &src, const StateView &dst, const qs_pauli_term *terms, size_t count,
                        cudaStream_t st) {
    HpsiOp op;
    QS_TRY(hpsi_prepare(src, terms, count, &op));
    HpsiOut o;
    o.out = dst.data;
    return hpsi_apply(op, src, o, HpsiOut{}, dst.data, st);
}

}  // namespace qsim
