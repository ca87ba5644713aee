// Gate queues on small states: a whole queue in one launch.
//
// A state below a tile (up to 12 qubits complex64, 11 complex128; 32 KiB) is
// too small for a launch per gate: a launch and its drain take about 1.3 us in
// a CUDA graph and 3 us from the host, the gate itself 0.1 us. Here one CTA per
// batch member loads the member into shared memory, applies the queue's gates
// one after the other (a barrier between gates, none between diagonal gates,
// whose amplitudes stay with their threads) and stores it back. Each gate's
// arithmetic has its one-gate kernel's precision and order of products
// (kernels_basic.cu, kernels_dfloat.cu); per-member rotations leave out the
// products with entries that are zero, and the two may fuse different products,
// so results agree to an FMA's rounding (a few 2^-24 per gate in complex64). The
// sines and cosines of per-member angles are formed once per launch, one thread
// per gate. Descriptors and matrices are kernel parameters (up to 32
// KB a launch: 512 gates), so a captured graph holds them by value; the CTA
// copies them to shared memory first.
//
// Bound by latency (about 90 instructions per warp and gate: decode, a
// shared-memory round trip, a barrier) for complex64, and by the FP64 pipe (2
// FMAs per clock and SM) for the per-member rotations of complex128, which stay
// in FP64. Measured: 150 mixed gates at n = 10 complex64 from a plan 59 us (197
// with a launch per gate); energy and gradient of 4 layers at n = 10, 8
// members, complex128 0.37 ms (1.23 ms). 512 threads: 59 us; 256, 128 and 64
// threads are within 5% at n = 10 and 1.3 to 4 times slower at n = 12.
#include <algorithm>
#include <cstring>

#include "adjoint.h"
#include "dd_sum.cuh"
#include "device.cuh"
#include "prof.h"
#include "small.h"
#include "tiled.h"

namespace qsim {

namespace {

constexpr int kMaxOps = 512;
constexpr int kMatBytes = 22016;
constexpr int kMaxSlots = 256;   // per-member angles per launch
constexpr int kMaxGrads = 64;    // gradient ops per launch
constexpr int kMaxThreads = 512;
// the state, then the launch's angles, matrices, ops and gradient sums
constexpr int kMaxSmem = (32 << 10) + kMaxSlots * 16 + kMatBytes + kMaxOps * 16 + kMaxGrads * (kMaxThreads / 32) * 8;

enum SOp : uint8_t {
    SO_DENSE,   // k = 1..3 targets, matrix at m
    SO_DENSEDF, // the same for complex128 in double-float (k = 1, 2), entries as float pairs
    SO_SWAP,
    SO_PHASE,   // amplitudes whose mask bits are 1 times m[0]
    SO_NEG,     // ... negated
    SO_DIAG,    // diagonal on k targets, entries at m
    SO_RX,      // per-member rotations, (cos, sin) of half the angle in `slot`
    SO_RY,
    SO_RZ,
    SO_PPHASE,  // per-member phase (cos, sin of the angle) on the mask bits
    SO_GRAD,    // Im<lambda|P|phi>, generator k (GEN_*)
};

struct __align__(16) SmallOp {
    uint8_t type, k;
    uint8_t barrier;   // the next op's threads read other threads' amplitudes
    uint8_t fixed;     // bits a group of amplitudes fixes: targets and controls
    uint16_t m;        // first matrix entry
    int16_t slot;      // per-member angle, or the gradient op's row
    uint16_t mask;     // control bits; phases: all required bits
    uint16_t t[3];     // target bits; diagonals: 5-bit positions in t[1], t[2]
};
static_assert(sizeof(SmallOp) == sizeof(uint4), "an op is one 16-byte load");

template <typename R> struct SmallP {
    int n, ms, n_ops, n_mats, n_slots, n_grads;
    int n_params, batch;
    double sign;
    const double *params;
    double *gpart;
    int32_t pidx[kMaxSlots];    // parameter column of slot j
    uint8_t phase[kMaxSlots];   // the whole angle (a phase), not half of it
    int32_t gslot[kMaxGrads];   // gpart row of gradient op j
    SmallOp op[kMaxOps];
    __align__(16) V<R> mat[kMatBytes / sizeof(V<R>)];
};
static_assert(sizeof(SmallP<float>) <= 32700 && sizeof(SmallP<double>) <= 32700,
              "small-state descriptors exceed the parameter space");

// first index of group g: zero bits inserted at the set bits of `fixed`
__device__ __forceinline__ uint32_t group_base(uint32_t g, uint32_t fixed) {
#pragma unroll 1
    while (fixed) {
        const uint32_t b = fixed & (0u - fixed);
        g += g & (0u - b);
        fixed ^= b;
    }
    return g;
}

template <typename R, int K>
__device__ __forceinline__ void dense(V<R> *s, const SmallOp &op, const V<R> *m, int n) {
    constexpr int D = 1 << K;
    uint32_t off[D];
#pragma unroll
    for (int l = 0; l < D; ++l) {
        off[l] = op.mask;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((l >> (K - 1 - j)) & 1) off[l] |= op.t[j];
    }
    uint32_t fixed = op.mask;
#pragma unroll
    for (int j = 0; j < K; ++j) fixed |= op.t[j];
    const uint32_t total = 1u << (n - op.fixed);
#pragma unroll 1
    for (uint32_t g = threadIdx.x; g < total; g += blockDim.x) {
        const uint32_t base = group_base(g, fixed);
        V<R> a[D];
#pragma unroll
        for (int l = 0; l < D; ++l) a[l] = s[base | off[l]];
#pragma unroll
        for (int r = 0; r < D; ++r) {
            V<R> acc = mkc<R>(0, 0);
#pragma unroll
            for (int c = 0; c < D; ++c) acc = cmadd<R>(m[r * D + c], a[c], acc);
            s[base | off[r]] = acc;
        }
    }
}

// 3 targets: a thread takes rows of the product (8 products each) instead of
// all 8 of a group, so that a small state keeps its threads busy: inputs are
// read, the CTA waits, the rows are written. Rows per thread: kRows3 at most.
constexpr int kRows3 = (1 << 12) / kMaxThreads;
template <typename R>
__device__ __forceinline__ void dense3(V<R> *s, const SmallOp &op, const V<R> *m, int n) {
    const uint32_t fixed = op.mask | op.t[0] | op.t[1] | op.t[2];
    const uint32_t total = 8u << (n - op.fixed);  // rows of all groups; group = row / 8
    auto offset = [&](uint32_t l) {
        return (uint32_t)op.mask | ((l & 4u) ? op.t[0] : 0u) | ((l & 2u) ? op.t[1] : 0u) | ((l & 1u) ? op.t[2] : 0u);
    };
    V<R> out[kRows3];
#pragma unroll
    for (int i = 0; i < kRows3; ++i) {
        const uint32_t t = threadIdx.x + i * blockDim.x;
        if (t >= total) break;
        const uint32_t base = group_base(t >> 3, fixed);
        const V<R> *row = m + (t & 7u) * 8;
        V<R> acc = mkc<R>(0, 0);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc = cmadd<R>(row[c], s[base | offset(c)], acc);
        out[i] = acc;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRows3; ++i) {
        const uint32_t t = threadIdx.x + i * blockDim.x;
        if (t >= total) break;
        s[group_base(t >> 3, fixed) | offset(t & 7u)] = out[i];
    }
}

template <int K>
__device__ __forceinline__ void dense_df(double2 *s, const SmallOp &op, const double2 *mat, int n) {
    constexpr int D = 1 << K;
    const ddc *m = reinterpret_cast<const ddc *>(mat);
    uint32_t off[D];
#pragma unroll
    for (int l = 0; l < D; ++l) {
        off[l] = op.mask;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((l >> (K - 1 - j)) & 1) off[l] |= op.t[j];
    }
    uint32_t fixed = op.mask;
#pragma unroll
    for (int j = 0; j < K; ++j) fixed |= op.t[j];
    const uint32_t total = 1u << (n - op.fixed);
#pragma unroll 1
    for (uint32_t g = threadIdx.x; g < total; g += blockDim.x) {
        const uint32_t base = group_base(g, fixed);
        ddc a[D];
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const double2 v = s[base | off[c]];
            a[c] = mkc<dd>(dd(v.x), dd(v.y));
        }
#pragma unroll
        for (int r = 0; r < D; ++r) {
            ProdSum acc = prod_first(m[r * D], a[0]);
#pragma unroll
            for (int c = 1; c < D; ++c) prod_add(acc, m[r * D + c], a[c]);
            const ddc w = prod_result(acc);
            s[base | off[r]] = make_double2(to_double(re_of<dd>(w)), to_double(im_of<dd>(w)));
        }
    }
}

// The per-member rotations: m00 a0 + m01 a1, m10 a0 + m11 a1 with the products
// by entries that are zero left out (they add exact zeros).
template <typename R>
__device__ __forceinline__ void rotate(V<R> *s, const SmallOp &op, R c, R sn, int n) {
    const uint32_t t = op.t[0], fixed = op.mask | t, total = 1u << (n - op.fixed);
#pragma unroll 1
    for (uint32_t g = threadIdx.x; g < total; g += blockDim.x) {
        const uint32_t i = group_base(g, fixed) | op.mask;
        const V<R> x = s[i], y = s[i | t];
        if (op.type == SO_RY) {  // [[c, -s], [s, c]]
            s[i] = mkc<R>(fma(-sn, y.x, c * x.x), fma(-sn, y.y, c * x.y));
            s[i | t] = mkc<R>(fma(c, y.x, sn * x.x), fma(c, y.y, sn * x.y));
        } else if (op.type == SO_RX) {  // [[c, -i s], [-i s, c]]
            s[i] = mkc<R>(fma(sn, y.y, c * x.x), fma(-sn, y.x, c * x.y));
            s[i | t] = mkc<R>(fma(c, y.x, sn * x.y), fma(c, y.y, -sn * x.x));
        } else {  // diag(c - i s, c + i s)
            s[i] = cmul<R>(mkc<R>(c, -sn), x);
            s[i | t] = cmul<R>(mkc<R>(c, sn), y);
        }
    }
}

// Im<lambda|P|phi> over this thread's share, in FP64 (phi below the top bit, lambda above)
template <typename R>
__device__ __forceinline__ double grad(const V<R> *s, const SmallOp &op, int n) {
    const uint32_t half = 1u << (n - 1), t = op.t[0];
    double acc = 0.0;
#pragma unroll 1
    for (uint32_t x = threadIdx.x; x < half; x += blockDim.x) {
        if ((x & op.mask) != op.mask) continue;
        const V<R> f = s[op.k <= GEN_Y ? (x ^ t) : x], l = s[x | half];
        double v;
        if (op.k == GEN_Y)
            v = (double)l.x * f.x + (double)l.y * f.y;
        else
            v = (double)l.x * f.y - (double)l.y * f.x;
        const bool one = (x & t) != 0;
        const bool neg = op.k == GEN_Y ? !one : op.k == GEN_Z && one;
        acc += neg ? -v : v;
    }
    return acc;
}

template <typename R>
__global__ void __launch_bounds__(kMaxThreads) small_kernel(V<R> *__restrict__ psi,
                                                            const __grid_constant__ SmallP<R> p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V<R> *s = reinterpret_cast<V<R> *>(smem_raw);
    double2 *cs = reinterpret_cast<double2 *>(smem_raw + (sizeof(V<R>) << p.n));
    V<R> *mat = reinterpret_cast<V<R> *>(cs + p.n_slots);
    uint4 *ops = reinterpret_cast<uint4 *>(mat + p.n_mats);
    double *gs = reinterpret_cast<double *>(ops + p.n_ops);  // per gradient op and warp
    const int tid = threadIdx.x, nt = blockDim.x, warps = (nt + 31) >> 5;
    // descriptors and matrices, read once through the global path: one at a
    // time through the constant cache, each miss would be waited for
    {
        const SmallP<R> *pp = &p;
        asm volatile("" : "+l"(pp));
        const uint4 *go = reinterpret_cast<const uint4 *>(pp->op);
        for (int i = tid; i < p.n_ops; i += nt) ops[i] = go[i];
        const V<R> *gm = pp->mat;
        for (int i = tid; i < p.n_mats; i += nt) mat[i] = gm[i];
    }
    const uint64_t b = blockIdx.x;
    V<R> *q = psi + (b << p.ms);
    const int size = 1 << p.n;
    for (int i = tid; i < size; i += nt) s[i] = q[i];
    for (int j = tid; j < p.n_slots; j += nt) {
        const double th = p.sign * p.params[b * p.n_params + p.pidx[j]];
        double sn, c;
        sincos(p.phase[j] ? th : 0.5 * th, &sn, &c);
        cs[j] = make_double2(c, sn);
    }
    __syncthreads();
    uint4 ahead = ops[0];
    for (int o = 0; o < p.n_ops; ++o) {
        SmallOp op;
        memcpy(&op, &ahead, sizeof(op));
        if (o + 1 < p.n_ops) ahead = ops[o + 1];
        switch (op.type) {
        case SO_DENSE:
            if (op.k == 1) dense<R, 1>(s, op, &mat[op.m], p.n);
            else if (op.k == 2) dense<R, 2>(s, op, &mat[op.m], p.n);
            else dense3<R>(s, op, &mat[op.m], p.n);
            break;
        case SO_DENSEDF:
            if constexpr (sizeof(R) == 8) {
                if (op.k == 1) dense_df<1>(s, op, &mat[op.m], p.n);
                else dense_df<2>(s, op, &mat[op.m], p.n);
            }
            break;
        case SO_SWAP: {
            const uint32_t A = op.t[0], B = op.t[1], fixed = op.mask | A | B, total = 1u << (p.n - op.fixed);
#pragma unroll 1
            for (uint32_t g = tid; g < total; g += nt) {
                const uint32_t x = group_base(g, fixed) | op.mask;
                const V<R> u = s[x | A], v = s[x | B];
                s[x | A] = v;
                s[x | B] = u;
            }
            break;
        }
        // diagonal ops: thread tid keeps the amplitudes tid + i nt
        case SO_PHASE: {
            const V<R> ph = mat[op.m];
#pragma unroll 1
            for (int x = tid; x < size; x += nt)
                if ((x & op.mask) == op.mask) s[x] = cmul<R>(s[x], ph);
            break;
        }
        case SO_NEG:
#pragma unroll 1
            for (int x = tid; x < size; x += nt)
                if ((x & op.mask) == op.mask) s[x] = cneg<R>(s[x]);
            break;
        case SO_DIAG: {
            const uint32_t pos = op.t[1] | (uint32_t)op.t[2] << 16;  // target positions, 5 bits each
#pragma unroll 1
            for (int x = tid; x < size; x += nt) {
                if ((x & op.mask) != op.mask) continue;
                int l = 0;
                for (int j = 0; j < op.k; ++j) l = (l << 1) | ((x >> ((pos >> (5 * j)) & 31u)) & 1);
                s[x] = cmul<R>(s[x], mat[op.m + l]);
            }
            break;
        }
        case SO_PPHASE: {
            const double2 v = cs[op.slot];
            const V<R> ph = mkc<R>((R)v.x, (R)v.y);
#pragma unroll 1
            for (int x = tid; x < size; x += nt)
                if ((x & op.mask) == op.mask) s[x] = cmul<R>(s[x], ph);
            break;
        }
        case SO_GRAD: {
            double v = grad<R>(s, op, p.n);
            for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
            if ((tid & 31) == 0) gs[op.slot * warps + (tid >> 5)] = v;
            break;
        }
        default: {
            const double2 v = cs[op.slot];
            rotate<R>(s, op, (R)v.x, (R)v.y, p.n);
            break;
        }
        }
        if (op.barrier) __syncthreads();
    }
    __syncthreads();
    for (int i = tid; i < size; i += nt) q[i] = s[i];
    for (int j = tid; j < p.n_grads; j += nt) {
        double sum = 0.0;
        for (int w = 0; w < warps; ++w) sum += gs[j * warps + w];
        p.gpart[(uint64_t)p.gslot[j] * p.batch + b] = sum;
    }
}

bool diagonal_op(int type) { return type == SO_PHASE || type == SO_NEG || type == SO_DIAG || type == SO_PPHASE; }

template <typename R>
qs_status run_t(qs_state *s, const std::vector<LGate> &G, const double *params, int n_params, double sign,
                double *gpart) {
    constexpr int kMats = kMatBytes / (int)sizeof(V<R>);
    const int n = s->n;
    const int threads = std::min(kMaxThreads, std::max(32, 1 << (n - 1)));
    const double amps = (double)((uint64_t)s->batch << n);
    static thread_local SmallP<R> p;
    int mats = 0;
    auto start = [&]() {
        p.n = n;
        p.ms = s->ms;
        p.n_ops = p.n_slots = p.n_grads = 0;
        p.n_params = n_params;
        p.batch = s->batch;
        p.sign = sign;
        p.params = params;
        p.gpart = gpart;
        mats = 0;
    };
    auto flush = [&]() -> qs_status {
        if (p.n_ops == 0) return QS_OK;
        for (int o = 0; o < p.n_ops; ++o) {
            const bool last = o + 1 == p.n_ops;
            const int a = p.op[o].type, b = last ? a : (int)p.op[o + 1].type;
            // diagonal ops keep their thread's amplitudes, gradient ops only read
            p.op[o].barrier = !last && !(diagonal_op(a) && diagonal_op(b)) && !(a == SO_GRAD && b == SO_GRAD);
        }
        mats += mats & 1;  // whole 16-byte words before the ops
        p.n_mats = mats;
        const size_t smem = (sizeof(V<R>) << n) + sizeof(double2) * p.n_slots + sizeof(V<R>) * mats +
                            sizeof(SmallOp) * p.n_ops + sizeof(double) * p.n_grads * ((threads + 31) / 32);
        if (smem > 48 * 1024)
            QS_CUDA_TRY(cudaFuncSetAttribute(small_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
        ProfScope _ps(s->stream, KC_TILED, 2.0 * amps * sizeof(V<R>), 14.0 * amps * p.n_ops);
        small_kernel<R><<<(unsigned)s->batch, threads, smem, s->stream>>>((V<R> *)s->data, p);
        QS_CUDA_TRY(cudaGetLastError());
        start();
        return QS_OK;
    };
    start();
    for (const LGate &g : G) {
        const int D = 1 << g.k;
        SmallOp op;
        std::memset(&op, 0, sizeof(op));
        op.k = (uint8_t)g.k;
        op.mask = (uint16_t)g.cmask;
        for (int j = 0; j < std::min(g.k, 3); ++j) op.t[j] = (uint16_t)(1u << g.tbit[j]);
        uint16_t all = op.mask;  // controls and targets
        for (int j = 0; j < g.k; ++j) all |= (uint16_t)(1u << g.tbit[j]);
        int need = 0;
        const bool is_grad = g.kind == kKindGrad, param = !is_grad && g.param_index >= 0;
        if (is_grad) {
            op.type = SO_GRAD;
            op.k = (uint8_t)g.grad_gen;
            if (g.grad_gen == GEN_PROJ) op.mask = all;
        } else if (param) {
            switch (g.kind) {
            case QS_GATE_RX: op.type = SO_RX; break;
            case QS_GATE_RY: op.type = SO_RY; break;
            case QS_GATE_RZ: op.type = SO_RZ; break;
            default:
                op.type = SO_PPHASE;
                op.mask = all;
            }
        } else if (g.is_swap) {
            op.type = SO_SWAP;
        } else if (g.phase_only) {
            const cd ph = g.m[D * D - 1];
            if (ph == cd(1.0, 0.0)) continue;  // identity
            op.type = ph == cd(-1.0, 0.0) ? SO_NEG : SO_PHASE;
            op.mask = all;
            need = 1;
        } else if (g.diagonal) {
            op.type = SO_DIAG;
            uint32_t pos = 0;
            for (int j = 0; j < g.k; ++j) pos |= (uint32_t)g.tbit[j] << (5 * j);
            op.t[1] = (uint16_t)pos;
            op.t[2] = (uint16_t)(pos >> 16);
            need = D;
        } else if (sizeof(R) == 8 && g.k <= 2 && !c128_fp64()) {
            op.type = SO_DENSEDF;
            need = D * D;
        } else if (g.k <= 3) {
            op.type = SO_DENSE;
            need = D * D;
        } else {  // dense on 4 or 5 targets: a pass of its own
            QS_TRY(flush());
            QS_TRY(k_apply_unfused(s, g));
            continue;
        }
        if (p.n_ops == kMaxOps || mats + need > kMats || p.n_slots == kMaxSlots || p.n_grads == kMaxGrads)
            QS_TRY(flush());
        op.fixed = (uint8_t)__builtin_popcount(all);
        op.m = (uint16_t)mats;
        auto entry = [&](const cd &v) { p.mat[mats++] = mkc<R>((R)v.real(), (R)v.imag()); };
        if (is_grad) {
            op.slot = (int16_t)p.n_grads;
            p.gslot[p.n_grads++] = g.grad_slot;
        } else if (param) {
            op.slot = (int16_t)p.n_slots;
            p.pidx[p.n_slots] = g.param_index;
            p.phase[p.n_slots++] = op.type == SO_PPHASE;
        } else if (op.type == SO_PHASE) {
            entry(g.m[D * D - 1]);
        } else if (op.type == SO_DIAG) {
            for (int l = 0; l < D; ++l) entry(g.m[l * D + l]);
        } else if (op.type == SO_DENSE) {
            for (int l = 0; l < D * D; ++l) entry(g.m[l]);
        } else if (op.type == SO_DENSEDF) {
            if constexpr (sizeof(R) == 8)
                for (int l = 0; l < D * D; ++l) {
                    const ddc v = mkc<dd>(dd(g.m[l].real()), dd(g.m[l].imag()));
                    std::memcpy(&p.mat[mats++], &v, sizeof(v));
                }
        }
        p.op[p.n_ops++] = op;
    }
    return flush();
}

}  // namespace

bool small_state(const qs_state *s) { return s->n < tile_bits(s->dtype); }

// Where the one launch is the faster form. It costs 8 us more than a first gate's
// launch (descriptors, the state's copy in shared memory) and saves 3.5 us for
// every further gate while launches bound both; a large batch fills the chip in
// one-gate launches too, and CTAs that hold a member each then only add the
// copies and the descriptors, so the batch it may have grows with the gates.
// Time against a launch per gate, mean of queues of mixed, dense 1-qubit, CZ and
// dense 2-qubit gates (65535 members: 30 gates and more):
//   complex64   n =  4: 3 gates 1.0, 4 gates 0.91; 30 gates at 64 / 8192 / 65535
//               members 0.42 / 0.59 / 1.6; n = 8: 0.41 / 0.92 / 1.2; n = 10, at 64 /
//               2048 / 65535: 0.42 / 0.99 / 1.3; n = 12: 0.49 / 0.93 / 0.73
//   complex128  n =  4: 0.47 / 1.04 / 3.0; n = 8, at 64 / 2048 / 65535: 0.46 / 0.84 / 1.3;
//               n = 11, at 64 / 256 / 65535: 0.64 / 0.80 / 1.4
// Per-member angles cost one-gate launches a sine and cosine per pair of
// amplitudes, here one per member: complex128 from n = 6 on 0.26 to 0.91 at any
// batch, complex64 at n = 12 0.28 to 0.80; at n = 10 with 76 gates 0.29 (256
// members), 1.04 (4096), 1.4 (65535).
bool one_launch(const qs_state *s, const std::vector<LGate> &G) {
    if (!small_state(s)) return false;
    const bool c64 = s->dtype == QS_C64;
    const int n = s->n, gates = (int)std::min<size_t>(G.size(), 1u << 20);
    int angles = 0;
    for (const LGate &g : G) angles += g.param_index >= 0;
    int members;  // per gate
    if (angles > 0 && 4ll * angles >= gates) {
        if (gates < 3) return false;
        if (n >= (c64 ? 11 : 6)) return true;
        members = 1 << std::min(10, 17 - n);
    } else {
        if (gates < 4) return false;
        if (c64 && n == 12 && gates >= 16) return true;
        members = c64 ? std::min(1 << 9, std::max(1 << 6, (1 << 16) >> n))
                      : std::min(1 << 7, std::max(1 << 4, (1 << 14) >> n));
    }
    return s->batch <= members * std::min(gates, 32);
}

qs_status run_small(qs_state *s, const std::vector<LGate> &G, const double *params, int n_params, double param_sign,
                    double *gpart) {
    return s->dtype == QS_C64 ? run_t<float>(s, G, params, n_params, param_sign, gpart)
                              : run_t<double>(s, G, params, n_params, param_sign, gpart);
}

}  // namespace qsim
