// Per-gate kernels: one HBM pass applies one (controlled) single-qubit update
// (Eq. 1) to the whole state.  These are the "plain" per-gate path and the
// building block every other mode is checked against.
//
// Access pattern.  Amplitudes are moved as 16-byte vectors: two complex64
// amplitudes (float4) or one complex128 amplitude (double2).  For a target
// qubit above the vector width the two partners of a pair sit in two
// different vectors 2^(t-W) vectors apart and each thread streams several
// such vector pairs (UNR) so enough bytes are in flight per SM; for the
// complex64 target qubit 0 the pair is inside one float4.  A control qubit
// above the vector width is folded into the work index (only the half with
// the control set is read); a control inside the vector is a per-lane test.
// Diagonal gates with u00 = 1 (T, S, Z, P, CZ, CP) read and write only the
// amplitudes they change.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "sv_internal.h"

namespace sv {
namespace {

template <typename R>
struct VecT;
template <>
struct VecT<float> {
    using T = float4;
    static constexpr int W = 1;  // log2 amplitudes per vector
};
template <>
struct VecT<double> {
    using T = double2;
    static constexpr int W = 0;
};

template <typename R>
struct C2 {
    R re, im;
};

template <typename R>
struct GateArgs {
    uint64_t nwork;       // work items
    uint64_t tbit;        // vector-index bit of the target (across kernel)
    uint64_t set_mask;    // vector-index bits forced to 1 (controls, phase mask)
    int ins[3];           // ascending vector-index positions where zero bits are inserted
    int nins;
    int lane_mask;        // amplitude-within-vector bits that must be 1 (W = 1 only)
    R u[8];               // 2x2 row-major (re, im)
};

__device__ __forceinline__ uint64_t insert_zero(uint64_t x, int p) {
    const uint64_t lo = x & ((uint64_t(1) << p) - 1);
    return ((x ^ lo) << 1) | lo;
}

template <typename R>
__device__ __forceinline__ uint64_t expand(uint64_t w, const GateArgs<R> &a) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (k < a.nins) w = insert_zero(w, a.ins[k]);
    return w | a.set_mask;
}

// Form of a 2x2 update, chosen on the host from the matrix's exact values.
// complex128 is bound by the FP64 pipe (two lanes per SM and clock), not by
// memory: 16 operations per pair for a general matrix, so the named gates use
// the fewest their structure allows (each form is one or two roundings per
// result, as the general one has three):
//   G_REAL    real entries                                   8 per pair
//   G_HAD     c [[1, 1], [1, -1]]: c a shared by both rows   6
//   G_SX(D)   (1 +- i)/2 [[1, -+i], [-+i, 1]]               10
//   G_SY(D)   (1 + i)/2 [[1, -1], [1, 1]] and its adjoint   10
//   G_SWAP    [[0, 1], [1, 0]]                               0
// 26 qubits: H 391 us, SX / SY 645, general 1028 (all three took 1027 before);
// 20 qubits, 590 gates of the random family: 7.43 ms before, 4.00 ms now.
enum GateForm { G_GENERAL = 0, G_REAL, G_HAD, G_SX, G_SXD, G_SY, G_SYD, G_SWAP };

template <int F, typename R>
__device__ __forceinline__ void apply2(const R *u, R &ar, R &ai, R &br, R &bi) {
    const R h = R(0.5);
    if constexpr (F == G_REAL) {
        const R nar = u[0] * ar + u[2] * br, nai = u[0] * ai + u[2] * bi;
        br = u[4] * ar + u[6] * br;
        bi = u[4] * ai + u[6] * bi;
        ar = nar;
        ai = nai;
    } else if constexpr (F == G_HAD) {
        const R c = u[0], p = c * ar, q = c * ai, x = br, y = bi;
        ar = fma(c, x, p);
        br = fma(-c, x, p);
        ai = fma(c, y, q);
        bi = fma(-c, y, q);
    } else if constexpr (F == G_SX || F == G_SXD) {
        // e = (a -+ i b) / 2, f = (b -+ i a) / 2; a' = (1 +- i) e, b' = (1 +- i) f
        const R p = h * ar, q = h * ai;
        if constexpr (F == G_SX) {
            const R er = fma(h, bi, p), ei = fma(-h, br, q), fr = fma(h, br, q), fi = fma(h, bi, -p);
            ar = er - ei;
            ai = er + ei;
            br = fr - fi;
            bi = fr + fi;
        } else {
            const R er = fma(-h, bi, p), ei = fma(h, br, q), fr = fma(h, br, -q), fi = fma(h, bi, p);
            ar = er + ei;
            ai = ei - er;
            br = fr + fi;
            bi = fi - fr;
        }
    } else if constexpr (F == G_SY || F == G_SYD) {
        const R p = h * ar, q = h * ai;
        const R sr = fma(h, br, p), si = fma(h, bi, q);
        if constexpr (F == G_SY) {  // a' = (1 + i) (a - b) / 2, b' = (1 + i) (a + b) / 2
            const R dr = fma(-h, br, p), di = fma(-h, bi, q);
            ar = dr - di;
            ai = dr + di;
            br = sr - si;
            bi = sr + si;
        } else {  // a' = (1 - i) (a + b) / 2, b' = (1 - i) (b - a) / 2
            const R dr = fma(h, br, -p), di = fma(h, bi, -q);
            ar = sr + si;
            ai = si - sr;
            br = dr + di;
            bi = di - dr;
        }
    } else if constexpr (F == G_SWAP) {
        const R x = ar, y = ai;
        ar = br;
        ai = bi;
        br = x;
        bi = y;
    } else {
        const R nar = u[0] * ar - u[1] * ai + u[2] * br - u[3] * bi;
        const R nai = u[0] * ai + u[1] * ar + u[2] * bi + u[3] * br;
        const R nbr = u[4] * ar - u[5] * ai + u[6] * br - u[7] * bi;
        const R nbi = u[4] * ai + u[5] * ar + u[6] * bi + u[7] * br;
        ar = nar;
        ai = nai;
        br = nbr;
        bi = nbi;
    }
}

// Vector pairs in flight per thread and threads per CTA.  complex64 is bound
// by memory and wants bytes in flight; complex128 is bound by the FP64 pipe
// (0.52 T operations/s measured), where the work has to spread evenly over the
// SMs at every size: small CTAs (20 qubits, 590 gates: 4.74 ms with 4 x 256,
// 4.15 with 2 x 128, 4.00 with 1 x 128; 26 qubits: the same within 1%).
template <typename R>
struct Shape1 {
    static constexpr int unr = 4, threads = 256;
};
template <>
struct Shape1<double> {
    static constexpr int unr = 1, threads = 128;
};

// Pair across two vectors (target >= W).
template <typename R, int F>
__global__ void __launch_bounds__(Shape1<R>::threads) k_gate_across(typename VecT<R>::T *__restrict__ v, GateArgs<R> a) {
    constexpr int kUnr = Shape1<R>::unr;
    using V = typename VecT<R>::T;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t base = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; base < a.nwork; base += stride * kUnr) {
        V x[kUnr], y[kUnr];
        uint64_t i0[kUnr];
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                i0[k] = expand(w, a);
                x[k] = v[i0[k]];
                y[k] = v[i0[k] | a.tbit];
            }
        }
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                if constexpr (VecT<R>::W == 1) {
                    if (!(a.lane_mask & 1)) apply2<F>(a.u, x[k].x, x[k].y, y[k].x, y[k].y);
                    apply2<F>(a.u, x[k].z, x[k].w, y[k].z, y[k].w);
                } else {
                    apply2<F>(a.u, x[k].x, x[k].y, y[k].x, y[k].y);
                }
                v[i0[k]] = x[k];
                v[i0[k] | a.tbit] = y[k];
            }
        }
    }
}

// complex64 target qubit 0: the pair is the two halves of one float4.
__global__ void __launch_bounds__(Shape1<float>::threads) k_gate_inner(float4 *__restrict__ v, GateArgs<float> a) {
    constexpr int kUnr = Shape1<float>::unr;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t base = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; base < a.nwork; base += stride * kUnr) {
        float4 x[kUnr];
        uint64_t i0[kUnr];
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                i0[k] = expand(w, a);
                x[k] = v[i0[k]];
            }
        }
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                apply2<G_GENERAL>(a.u, x[k].x, x[k].y, x[k].z, x[k].w);
                v[i0[k]] = x[k];
            }
        }
    }
}

// u11 of a diagonal gate with u00 = 1 on one amplitude.  Sign flips and
// quarter turns (CZ, Z, S) are exact moves: no FP64 operations, and 4 for
// another phase.
enum PhaseForm { P_GENERAL = 0, P_NEG, P_I, P_MI };

// -x as a flip of the sign bit: the compiler's own negation of a double that
// is stored as it is goes through the FP64 pipe.
__device__ __forceinline__ float neg(float x) { return -x; }
__device__ __forceinline__ double neg(double x) {
    return __hiloint2double(__double2hiint(x) ^ int(0x80000000u), __double2loint(x));
}

template <int F, typename R>
__device__ __forceinline__ void phase1(R pr, R pi, R &x, R &y) {
    if constexpr (F == P_NEG) {
        x = neg(x);
        y = neg(y);
    } else if constexpr (F == P_I || F == P_MI) {
        const R t = F == P_I ? x : neg(x);
        x = F == P_I ? neg(y) : y;
        y = t;
    } else {
        const R r = x * pr - y * pi, i = x * pi + y * pr;
        x = r;
        y = i;
    }
}

// Diagonal gate with u00 = 1: multiply the amplitudes whose masked bits are
// all set by u11.  Vectors are enumerated with the vector-level mask bits
// forced to 1; lane_mask selects amplitudes inside a float4.
template <typename R, int F>
__global__ void __launch_bounds__(Shape1<R>::threads) k_phase(typename VecT<R>::T *__restrict__ v, GateArgs<R> a) {
    constexpr int kUnr = Shape1<R>::unr;
    using V = typename VecT<R>::T;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const R pr = a.u[6], pi = a.u[7];
    for (uint64_t base = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; base < a.nwork; base += stride * kUnr) {
        V x[kUnr];
        uint64_t i0[kUnr];
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                i0[k] = expand(w, a);
                x[k] = v[i0[k]];
            }
        }
#pragma unroll
        for (int k = 0; k < kUnr; ++k) {
            const uint64_t w = base + k * stride;
            if (w < a.nwork) {
                if constexpr (VecT<R>::W == 1) {
                    if (!(a.lane_mask & 1)) phase1<F>(pr, pi, x[k].x, x[k].y);
                    phase1<F>(pr, pi, x[k].z, x[k].w);
                } else {
                    phase1<F>(pr, pi, x[k].x, x[k].y);
                }
                v[i0[k]] = x[k];
            }
        }
    }
}

template <typename R>
int grid_for(uint64_t nwork) {
    constexpr uint64_t per = uint64_t(Shape1<R>::threads) * Shape1<R>::unr;
    uint64_t b = (nwork + per - 1) / per;
    if (b < 1) b = 1;
    const uint64_t cap = 152ull * 32 * (256 / Shape1<R>::threads);
    return int(b < cap ? b : cap);
}

void sort_small(int *p, int n) {
    for (int i = 1; i < n; ++i)
        for (int j = i; j > 0 && p[j - 1] > p[j]; --j) {
            int t = p[j];
            p[j] = p[j - 1];
            p[j - 1] = t;
        }
}

template <typename R>
int gate_form(const R *u) {
    auto is = [&](R a, R b, R c, R d, R e, R f, R g, R h) {
        const R w[8] = {a, b, c, d, e, f, g, h};
        for (int k = 0; k < 8; ++k)
            if (u[k] != w[k]) return false;
        return true;
    };
    const R h = R(0.5);
    if (is(0, 0, 1, 0, 1, 0, 0, 0)) return G_SWAP;
    if (is(h, h, h, -h, h, -h, h, h)) return G_SX;
    if (is(h, -h, h, h, h, h, h, -h)) return G_SXD;
    if (is(h, h, -h, -h, h, h, h, h)) return G_SY;
    if (is(h, -h, h, -h, -h, h, h, -h)) return G_SYD;
    if (u[1] == 0 && u[3] == 0 && u[5] == 0 && u[7] == 0)
        return u[0] == u[2] && u[0] == u[4] && u[0] == -u[6] ? G_HAD : G_REAL;
    return G_GENERAL;
}

template <typename R>
int phase_form(const R *u) {
    if (u[6] == -1 && u[7] == 0) return P_NEG;
    if (u[6] == 0 && u[7] == 1) return P_I;
    if (u[6] == 0 && u[7] == -1) return P_MI;
    return P_GENERAL;
}

// Diagonal with u00 = 1: only the amplitudes with the target (and control)
// bits set change.
bool is_phase(const Gate1 &g) {
    return g.u[1].re == 0 && g.u[1].im == 0 && g.u[2].re == 0 && g.u[2].im == 0 && g.u[0].re == 1 && g.u[0].im == 0;
}

template <typename R>
cudaError_t gate1_impl(sv_state *h, const Gate1 &g) {
    using V = typename VecT<R>::T;
    constexpr int W = VecT<R>::W;
    GateArgs<R> a{};
    for (int k = 0; k < 4; ++k) {
        a.u[2 * k] = R(g.u[k].re);
        a.u[2 * k + 1] = R(g.u[k].im);
    }
    const int n = h->n;
    const int nv_log = n - W;  // log2 number of vectors
    V *v = static_cast<V *>(h->data);
    const int t = g.target, c = g.control;
    if (is_phase(g)) {
        // phase on amplitudes with bit t (and bit c) set
        int ins[2], ni = 0;
        uint64_t setm = 0;
        int lane = 0;
        for (int b : {t, c}) {
            if (b < 0) continue;
            if (b >= W) {
                ins[ni++] = b - W;
                setm |= uint64_t(1) << (b - W);
            } else {
                lane |= 1 << b;
            }
        }
        sort_small(ins, ni);
        for (int k = 0; k < ni; ++k) a.ins[k] = ins[k];
        a.nins = ni;
        a.set_mask = setm;
        a.lane_mask = lane;
        a.nwork = uint64_t(1) << (nv_log - ni);
        const int grid = grid_for<R>(a.nwork);
        if constexpr (W == 0) {  // FP64: the forms; complex64 is bound by memory
            switch (phase_form(a.u)) {
                case P_NEG: k_phase<R, P_NEG><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case P_I: k_phase<R, P_I><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case P_MI: k_phase<R, P_MI><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                default: k_phase<R, P_GENERAL><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
            }
        } else {
            k_phase<R, P_GENERAL><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a);
        }
        return cudaGetLastError();
    }
    int ins[2], ni = 0;
    uint64_t setm = 0;
    int lane = 0;
    if (c >= 0) {
        if (c >= W) {
            ins[ni++] = c - W;
            setm |= uint64_t(1) << (c - W);
        } else {
            lane |= 1 << c;
        }
    }
    if (t >= W) {
        ins[ni++] = t - W;
        a.tbit = uint64_t(1) << (t - W);
    }
    sort_small(ins, ni);
    for (int k = 0; k < ni; ++k) a.ins[k] = ins[k];
    a.nins = ni;
    a.set_mask = setm;
    a.lane_mask = lane;
    a.nwork = uint64_t(1) << (nv_log - ni);
    if (t >= W) {
        const int grid = grid_for<R>(a.nwork);
        if constexpr (W == 0) {
            switch (gate_form(a.u)) {
                case G_REAL: k_gate_across<R, G_REAL><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_HAD: k_gate_across<R, G_HAD><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_SX: k_gate_across<R, G_SX><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_SXD: k_gate_across<R, G_SXD><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_SY: k_gate_across<R, G_SY><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_SYD: k_gate_across<R, G_SYD><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                case G_SWAP: k_gate_across<R, G_SWAP><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
                default: k_gate_across<R, G_GENERAL><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a); break;
            }
        } else {
            k_gate_across<R, G_GENERAL><<<grid, Shape1<R>::threads, 0, h->stream>>>(v, a);
        }
    } else {
        if constexpr (W == 1) {
            k_gate_inner<<<grid_for<float>(a.nwork), Shape1<float>::threads, 0, h->stream>>>(reinterpret_cast<float4 *>(v), a);
        }
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- small states
// A run of per-gate updates on a state that fits one CTA's shared memory, in
// one launch: the state is loaded once, the gates are applied in circuit
// order, and it is stored once.  One launch per gate of such a state is all
// launch latency (10 qubits, 145 gates, graph replay: 1.2 us per gate).  The
// gates are taken in stages of consecutive gates with at most S distinct
// targets (diagonal gates have none): each thread gathers the 2^S amplitudes
// of those qubits into registers, applies the stage's gates and scatters them
// back, so a stage costs one shared-memory round trip and one barrier.  The
// gates come as a
// kernel parameter, so a launch needs no device memory of its own.
template <typename R>
struct SmallOp {
    uint8_t code;    // pair updates: GateForm * 2 + slot; 16 + PhaseForm; a stage header: number of its gates
    uint8_t rmask;   // register-index bits that must be 1
    uint8_t s[2];    // stage header: its qubits
    uint32_t imask;  // other amplitude-index bits that must be 1
    R u[8];
};
template <typename R>
struct SmallRun {
    static constexpr int kMaxOps = sizeof(R) == 4 ? 200 : 112;  // 8 KB of parameters
    int n, nops;
    SmallOp<R> op[kMaxOps];
};

// Swizzled position of amplitude i: rows of 128 bytes, the column permuted by
// the row number (linear over XOR), so that gathers of low qubits spread over
// the banks.
template <typename R>
__device__ __forceinline__ uint32_t small_pos(uint32_t i) {
    return sizeof(R) == 4 ? i ^ ((i >> 4) & 15u) : i ^ ((i >> 3) & 7u);
}

template <int F, int SLOT, int S, typename R>
__device__ __forceinline__ void small_pairs(C2<R> (&x)[1 << S], const SmallOp<R> &op) {
    if constexpr (SLOT < S) {
#pragma unroll
        for (int v = 0; v < (1 << S); ++v) {
            if (v >> SLOT & 1) continue;
            const int w = v | 1 << SLOT;
            if ((v & op.rmask) == op.rmask) apply2<F>(op.u, x[v].re, x[v].im, x[w].re, x[w].im);
        }
    }
}
template <int F, int S, typename R>
__device__ __forceinline__ void small_phase(C2<R> (&x)[1 << S], const SmallOp<R> &op) {
#pragma unroll
    for (int v = 0; v < (1 << S); ++v)
        if ((v & op.rmask) == op.rmask) phase1<F>(op.u[6], op.u[7], x[v].re, x[v].im);
}

template <int S, typename R>
__device__ __forceinline__ void small_gate(C2<R> (&x)[1 << S], const SmallOp<R> &op) {
#define SV_SMALL_FORM(F)                                        \
    case 2 * F: small_pairs<F, 0, S>(x, op); break;             \
    case 2 * F + 1: small_pairs<F, 1, S>(x, op); break;
    switch (op.code) {
        SV_SMALL_FORM(G_GENERAL)
        SV_SMALL_FORM(G_REAL)
        SV_SMALL_FORM(G_HAD)
        SV_SMALL_FORM(G_SX)
        SV_SMALL_FORM(G_SXD)
        SV_SMALL_FORM(G_SY)
        SV_SMALL_FORM(G_SYD)
        SV_SMALL_FORM(G_SWAP)
        case 16 + P_NEG: small_phase<P_NEG, S>(x, op); break;
        case 16 + P_I: small_phase<P_I, S>(x, op); break;
        case 16 + P_MI: small_phase<P_MI, S>(x, op); break;
        default: small_phase<P_GENERAL, S>(x, op); break;
    }
#undef SV_SMALL_FORM
}

template <typename R>
constexpr int kSmallThreads = sizeof(R) == 4 ? 1024 : 512;

template <typename R, int S>
__global__ void __launch_bounds__(kSmallThreads<R>) k_small_run(C2<R> *__restrict__ psi, const __grid_constant__ SmallRun<R> a) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    C2<R> *sm = reinterpret_cast<C2<R> *>(small_smem);
    __shared__ __align__(16) SmallOp<R> ops[SmallRun<R>::kMaxOps];
    const uint32_t namps = 1u << a.n;
    for (uint32_t i = threadIdx.x; i < a.nops * uint32_t(sizeof(SmallOp<R>) / 8); i += blockDim.x)
        reinterpret_cast<uint2 *>(ops)[i] = reinterpret_cast<const uint2 *>(a.op)[i];
    for (uint32_t i = threadIdx.x; i < namps; i += blockDim.x) sm[small_pos<R>(i)] = psi[i];
    __syncthreads();
    for (int k = 0; k < a.nops;) {
        const int cnt = ops[k].code;
        const int s0 = ops[k].s[0], s1 = ops[k].s[1];
        const uint32_t d0 = small_pos<R>(1u << s0), d1 = small_pos<R>(1u << s1);
        for (uint32_t w = threadIdx.x; w < namps >> S; w += blockDim.x) {
            uint32_t i = w + (w & ~((1u << s0) - 1));  // a zero bit inserted at s0
            if (S > 1) i += i & ~((1u << s1) - 1);
            const uint32_t p = small_pos<R>(i);
            C2<R> x[1 << S];
#pragma unroll
            for (int v = 0; v < (1 << S); ++v)
                x[v] = sm[p ^ (v & 1 ? d0 : 0u) ^ (v & 2 ? d1 : 0u)];
            for (int j = k + 1; j <= k + cnt; ++j) {
                const SmallOp<R> &op = ops[j];
                if ((i & op.imask) == op.imask) small_gate<S>(x, op);
            }
#pragma unroll
            for (int v = 0; v < (1 << S); ++v)
                sm[p ^ (v & 1 ? d0 : 0u) ^ (v & 2 ? d1 : 0u)] = x[v];
        }
        __syncthreads();
        k += cnt + 1;
    }
    for (uint32_t i = threadIdx.x; i < namps; i += blockDim.x) psi[i] = sm[small_pos<R>(i)];
}

// Fill a with a stage (or the part of it that fits) starting at gate i;
// returns the next gate.
template <typename R, int S>
size_t small_stage(int n, const Gate1 *g, size_t i, size_t count, SmallRun<R> *a) {
    constexpr int kMax = SmallRun<R>::kMaxOps;
    uint32_t qs = 0;  // the stage's qubits
    size_t e = i;
    for (; e < count && int(e - i) + 1 < kMax - a->nops && e - i < 255; ++e) {
        if (is_phase(g[e])) continue;
        const uint32_t b = 1u << g[e].target;
        if (!(qs & b) && __builtin_popcount(qs) == S) break;
        qs |= b;
    }
    for (int q = n - 1; q >= 0 && __builtin_popcount(qs) < S; --q) qs |= 1u << q;  // high ones: no bank conflicts
    int slot[32], s[2] = {0, 0}, ns = 0;
    for (int q = 0; q < n; ++q) {
        slot[q] = -1;
        if (qs >> q & 1u) {
            s[ns] = q;
            slot[q] = ns++;
        }
    }
    SmallOp<R> &hd = a->op[a->nops++];
    hd = SmallOp<R>{};
    hd.code = uint8_t(e - i);
    hd.s[0] = uint8_t(s[0]);
    hd.s[1] = uint8_t(s[1]);
    for (; i < e; ++i) {
        SmallOp<R> &op = a->op[a->nops++];
        op = SmallOp<R>{};
        for (int k = 0; k < 4; ++k) {
            op.u[2 * k] = R(g[i].u[k].re);
            op.u[2 * k + 1] = R(g[i].u[k].im);
        }
        uint32_t cond = g[i].control < 0 ? 0u : 1u << g[i].control;
        if (is_phase(g[i])) {
            cond |= 1u << g[i].target;
            op.code = uint8_t(16 + phase_form(op.u));
        } else {
            op.code = uint8_t(2 * gate_form(op.u) + slot[g[i].target]);
        }
        for (int q = 0; q < n; ++q)
            if (cond >> q & 1u) {
                if (slot[q] >= 0) op.rmask |= uint8_t(1u << slot[q]);
                else op.imask |= 1u << q;
            }
    }
    return e;
}

template <typename R, int S>
cudaError_t small_run(sv_state *h, const Gate1 *g, size_t count) {
    const int n = h->n;
    const int tlog = n - S;
    const int threads = tlog < 5 ? 32 : (1 << tlog) > kSmallThreads<R> ? kSmallThreads<R> : 1 << tlog;
    const int smem = int(sizeof(C2<R>)) << n;
    for (size_t i = 0; i < count;) {
        SmallRun<R> a;
        a.n = n;
        a.nops = 0;
        while (i < count && a.nops + 2 <= SmallRun<R>::kMaxOps) i = small_stage<R, S>(n, g, i, count, &a);
        k_small_run<R, S><<<1, threads, smem, h->stream>>>(static_cast<C2<R> *>(h->data), a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------- states in L2
// A per-gate plan of a state that stays in L2 takes several gates per launch:
// a thread holds the 2^S amplitudes of S chosen qubits in registers, applies
// the run's gates and stores them back (plan_gate_runs chooses the runs).  One
// launch per gate of such a state is bound by launches and L2 round trips, in
// complex128 also by the FP64 pipe (two lanes per SM and clock), so the scalar
// factors of H, SX, SY and their adjoints (powers of e^(i pi/4) and 2^(-1/2),
// counted exactly on the host) are owed: those gates are then 4 additions per
// pair instead of 6 to 10 operations, and a multiplication per component pays
// 2^-4 (complex128: 2^-12) whenever as much is owed, the last launch the rest.
// The powers of two are exact, and no value in between exceeds the state's norm
// by more than that factor.  20 qubits, 590 gates of the random family
// in complex128: 4.00 ms with a launch per gate, 2.77 in runs that multiply for
// every H, 1.85 now; 236 gates in complex64: 0.097 ms.
// Few forms keep the code small (a launch starts with it uncached), and the
// gates come as kernel parameters, so that branches and factors are uniform.
enum RunKind : uint8_t { R_HAD, R_SX, R_SXD, R_SY, R_SYD, R_GENERAL, R_SWAP, R_NEG, R_TURN, R_PHASE, R_SCALE };

// Factors 2^(-1/2) owed at most, and what R_SCALE multiplies by to pay them.
// complex64 pays early, for the range of its exponent: a 32nd of a run's
// operations, under its launches.
template <typename R>
constexpr int kRunOwed = sizeof(R) == 4 ? 8 : 24;
template <typename R>
constexpr R kRunScale = R(1) / R(1 << kRunOwed<R> / 2);

template <typename R>
struct RunArgs {
    uint32_t q[kRunSlots];   // the registers' qubits, ascending
    int nops, odd, quarter;  // factor paid at the end: (1 + i)^odd i^quarter m
    R m;
    GateRunHead op[kRunMaxOps];
    R u[8 * kRunMaxOps];
};

// A warp's qubits other than 0..4, and the places of the registers' among all.
struct RunRows {
    uint32_t far[kRunSlots], rank[kRunSlots];
};
struct NoRows {};

// Without their factors: H (a + b, a - b), SX (a - i b, b - i a), SY (a - b,
// a + b) and the adjoints of the last two.
template <int K, typename R>
__device__ __forceinline__ void run_pair(C2<R> &a, C2<R> &b) {
    const C2<R> x = a, y = b;
    if constexpr (K == R_SX) {
        a = C2<R>{x.re + y.im, x.im - y.re};
        b = C2<R>{y.re + x.im, y.im - x.re};
    } else if constexpr (K == R_SXD) {
        a = C2<R>{x.re - y.im, x.im + y.re};
        b = C2<R>{y.re - x.im, y.im + x.re};
    } else {
        const C2<R> s = {x.re + y.re, x.im + y.im};
        const C2<R> d = K == R_SYD ? C2<R>{y.re - x.re, y.im - x.im} : C2<R>{x.re - y.re, x.im - y.im};
        a = K == R_SY ? d : s;
        b = K == R_SY ? s : d;
    }
}

template <int K, int SLOT, int S, typename R>
__device__ __forceinline__ void run_all(C2<R> (&x)[1 << S]) {
#pragma unroll
    for (int v = 0; v < (1 << S); ++v)
        if (!(v >> SLOT & 1)) run_pair<K>(x[v], x[v | 1 << SLOT]);
}

template <int SLOT, int S, typename R>
__device__ __forceinline__ void run_pairs(C2<R> (&x)[1 << S], const GateRunHead &op, const R *u) {
    if constexpr (SLOT < S) {
        const uint32_t mask = op.rmask;
        switch (op.kind) {
            case R_HAD: run_all<R_HAD, SLOT, S>(x); break;
            case R_SX: run_all<R_SX, SLOT, S>(x); break;
            case R_SXD: run_all<R_SXD, SLOT, S>(x); break;
            case R_SY: run_all<R_SY, SLOT, S>(x); break;
            case R_SYD: run_all<R_SYD, SLOT, S>(x); break;
            case R_SWAP:
#pragma unroll
                for (int v = 0; v < (1 << S); ++v) {
                    if (v >> SLOT & 1) continue;
                    const int w = v | 1 << SLOT;
                    if ((v & mask) == mask) apply2<G_SWAP>(u, x[v].re, x[v].im, x[w].re, x[w].im);
                }
                break;
            default:
#pragma unroll
                for (int v = 0; v < (1 << S); ++v) {
                    if (v >> SLOT & 1) continue;
                    const int w = v | 1 << SLOT;
                    if ((v & mask) == mask) apply2<G_GENERAL>(u, x[v].re, x[v].im, x[w].re, x[w].im);
                }
                break;
        }
    }
}

template <int F, int S, typename R>
__device__ __forceinline__ void run_phase(C2<R> (&x)[1 << S], uint32_t mask, R pr, R pi) {
#pragma unroll
    for (int v = 0; v < (1 << S); ++v)
        if ((v & mask) == mask) phase1<F>(pr, pi, x[v].re, x[v].im);
}

// The same for one mask known to the compiler: a test per register becomes a
// predicate, and a predicated FP64 instruction takes its turn in the pipe also
// where no lane executes it (20-qubit Fourier transform in complex128 1.78 ms with
// tests, 0.96 so; 0.74 now that H owes its factor too).
template <uint32_t MASK, int S, typename R>
__device__ __forceinline__ void run_phase_of(C2<R> (&x)[1 << S], R pr, R pi) {
    if constexpr (MASK < (1u << S)) {
#pragma unroll
        for (uint32_t v = 0; v < (1u << S); ++v)
            if ((v & MASK) == MASK) phase1<P_GENERAL>(pr, pi, x[v].re, x[v].im);
    }
}
template <int S, typename R>
__device__ __forceinline__ void run_phase_general(C2<R> (&x)[1 << S], uint32_t mask, R pr, R pi) {
    switch (mask) {  // a diagonal gate has at most two qubits
        case 0: run_phase_of<0, S>(x, pr, pi); break;
        case 1: run_phase_of<1, S>(x, pr, pi); break;
        case 2: run_phase_of<2, S>(x, pr, pi); break;
        case 3: run_phase_of<3, S>(x, pr, pi); break;
        case 4: run_phase_of<4, S>(x, pr, pi); break;
        case 5: run_phase_of<5, S>(x, pr, pi); break;
        case 6: run_phase_of<6, S>(x, pr, pi); break;
        case 8: run_phase_of<8, S>(x, pr, pi); break;
        case 9: run_phase_of<9, S>(x, pr, pi); break;
        case 10: run_phase_of<10, S>(x, pr, pi); break;
        default: run_phase_of<12, S>(x, pr, pi); break;
    }
}

template <int S, typename R>
__device__ __forceinline__ void run_gate(C2<R> (&x)[1 << S], const GateRunHead &op, const R *u) {
    if (op.kind >= R_NEG) {
        if (op.kind == R_NEG) run_phase<P_NEG, S>(x, op.rmask, R(0), R(0));
        else if (op.kind == R_PHASE) run_phase_general<S>(x, op.rmask, u[0], u[1]);
        else if (op.arg == 1) run_phase<P_I, S>(x, op.rmask, R(0), R(0));
        else if (op.arg == 3) run_phase<P_MI, S>(x, op.rmask, R(0), R(0));
        else {  // R_SCALE
#pragma unroll
            for (int v = 0; v < (1 << S); ++v) {
                x[v].re *= kRunScale<R>;
                x[v].im *= kRunScale<R>;
            }
        }
        return;
    }
    switch (op.slot) {
        case 0: run_pairs<0, S>(x, op, u); break;
        case 1: run_pairs<1, S>(x, op, u); break;
        case 2: run_pairs<2, S>(x, op, u); break;
        default: run_pairs<3, S>(x, op, u); break;
    }
}

template <typename R>
struct Amp2;
template <>
struct Amp2<float> {
    using T = float2;
};
template <>
struct Amp2<double> {
    using T = double2;
};

constexpr int kRunThreads = 64;  // small CTAs: even work per SM (20 qubits: 1024 CTAs, 6.7 per SM)

template <typename R, int S, bool LOW>
__global__ void __launch_bounds__(kRunThreads) k_gate_run(typename Amp2<R>::T *__restrict__ psi,
                                                          const __grid_constant__ RunArgs<R> a,
                                                          const __grid_constant__ std::conditional_t<LOW, RunRows, NoRows> w) {
    using V = typename Amp2<R>::T;
    uint32_t i = blockIdx.x * kRunThreads + threadIdx.x;
#pragma unroll
    for (int k = 0; k < S; ++k) i += i & ~((1u << a.q[k]) - 1u);  // a zero bit inserted at q[k]
    C2<R> x[1 << S];
    // LOW: a warp's amplitudes (its S + 5 qubits always contain 0..4) are moved
    // in rows of 32 consecutive ones, and change hands in shared memory.  A
    // thread that holds several of qubits 0..3 itself makes every 8-byte access
    // of its warp touch up to 32 lines instead of 2 (complex64, 4 H: on qubits
    // 0..3 at 23 qubits 67.8 us direct, 23.3 by rows, 16.4 on high qubits; on 0, 1
    // and two high ones 36.9 and 23.5; at 20 qubits 12.3 and 6.3).  With one low
    // qubit, or two but 0 and 1, rows gain nothing (23 qubits 18.6 and 22.9, 20.6
    // and 26.8), nor for states up to 17 qubits.
    __shared__ V rows[LOW ? kRunThreads << S : 1];
    const uint32_t lane = threadIdx.x & 31u;
    V *const warp = rows + (LOW ? (threadIdx.x & ~31u) << S : 0u);
    [[maybe_unused]] auto row = [&](int v) {
        uint32_t j = __shfl_sync(0xffffffffu, i, 0) | lane;
#pragma unroll
        for (int k = 0; k < S; ++k)
            if constexpr (LOW) j |= (v >> k & 1) << w.far[k];
        return psi + j;
    };
    uint32_t own = lane;  // this thread's amplitudes in the warp's order
    if constexpr (LOW) {
#pragma unroll
        for (int k = 0; k < S; ++k) own += own & ~((1u << w.rank[k]) - 1u);
        own = small_pos<R>(own);
    }
    [[maybe_unused]] auto held = [&](int v) {
        uint32_t j = own;
#pragma unroll
        for (int k = 0; k < S; ++k)
            if constexpr (LOW) j ^= v >> k & 1 ? small_pos<R>(1u << w.rank[k]) : 0u;
        return warp + j;
    };
    auto at = [&](int v) {
        uint32_t j = i;
#pragma unroll
        for (int k = 0; k < S; ++k)
            if (v >> k & 1) j |= 1u << a.q[k];
        return psi + j;
    };
    if constexpr (LOW) {
#pragma unroll
        for (int v = 0; v < (1 << S); ++v) warp[small_pos<R>(uint32_t(v) << 5 | lane)] = *row(v);
        __syncwarp();
    }
#pragma unroll
    for (int v = 0; v < (1 << S); ++v) {
        V z;
        if constexpr (LOW) z = *held(v);
        else z = *at(v);
        x[v].re = z.x;
        x[v].im = z.y;
    }
    for (int k = 0; k < a.nops; ++k)
        if ((i & a.op[k].imask) == a.op[k].imask) run_gate<S>(x, a.op[k], a.u + 2 * a.op[k].arg);
    if (a.odd) {
#pragma unroll
        for (int v = 0; v < (1 << S); ++v) {
            const R r = x[v].re - x[v].im;
            x[v].im = x[v].re + x[v].im;
            x[v].re = r;
        }
    }
    if (a.m != R(1)) {
#pragma unroll
        for (int v = 0; v < (1 << S); ++v) {
            x[v].re *= a.m;
            x[v].im *= a.m;
        }
    }
    if (a.quarter & 1) run_phase<P_I, S>(x, 0u, R(0), R(0));
    if (a.quarter & 2) run_phase<P_NEG, S>(x, 0u, R(0), R(0));
#pragma unroll
    for (int v = 0; v < (1 << S); ++v) {
        V z;
        z.x = x[v].re;
        z.y = x[v].im;
        if constexpr (LOW) *held(v) = z;
        else *at(v) = z;
    }
    if constexpr (LOW) {
        __syncwarp();
#pragma unroll
        for (int v = 0; v < (1 << S); ++v) *row(v) = warp[small_pos<R>(uint32_t(v) << 5 | lane)];
    }
}

template <typename R, int S>
cudaError_t gate_runs_impl(sv_state *h, const GateRuns &p, const std::vector<Gate1> &g) {
    for (const GateRun &r : p.runs) {
        for (int i : r.alone) {
            const cudaError_t e = launch_gate1(h, g[size_t(i)]);
            if (e != cudaSuccess) return e;
        }
        if (r.count == 0) continue;
        RunArgs<R> a;
        for (int k = 0; k < S; ++k) a.q[k] = uint32_t(r.q[k]);
        a.nops = r.count;
        std::copy_n(p.ops.begin() + long(r.first), r.count, a.op);
        for (int k = 0; k < r.ucount; ++k) a.u[k] = R(p.u[r.ufirst + size_t(k)]);
        a.odd = r.odd;
        a.quarter = r.quarter;
        a.m = R(r.m);
        auto *psi = static_cast<typename Amp2<R>::T *>(h->data);
        const unsigned grid = 1u << (h->n - S - 6);
        bool rows = false;
        if constexpr (sizeof(R) == 4 && S == 4) {
            RunRows w;
            rows = r.q[1] == 1 || r.q[2] < 4;
            if (rows) {
                // the warp's qubits, ascending: the registers' and the lowest 5 others
                int all[S + 5], na = 0, lanes = 0;
                for (int q = 0; na < S + 5; ++q) {
                    const bool reg = std::find(r.q, r.q + S, q) != r.q + S;
                    if (!reg && lanes == 5) continue;
                    lanes += !reg;
                    all[na++] = q;
                }
                for (int k = 0; k < S; ++k) {
                    w.far[k] = uint32_t(all[5 + k]);
                    w.rank[k] = uint32_t(std::find(all, all + S + 5, r.q[k]) - all);
                }
                k_gate_run<R, S, true><<<grid, kRunThreads, 0, h->stream>>>(psi, a, w);
            }
        }
        if (!rows) k_gate_run<R, S, false><<<grid, kRunThreads, 0, h->stream>>>(psi, a, NoRows{});
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------- set basis
template <typename R>
__global__ void k_set_one(C2<R> *psi, uint64_t idx) {
    psi[idx].re = R(1);
    psi[idx].im = R(0);
}

__global__ void k_enc_set_one(char2 *codes, float *scales, uint64_t idx) {
    codes[idx] = make_char2(127, 0);
    scales[idx >> kEncBlockLog2] = 1.0f;
}

// ---------------------------------------------------------------- norm
constexpr int kNormBlocks = 152 * 8;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ double block_sum(double v) {
    __shared__ double sh[32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    if (wid == 0) v = warp_sum(v);
    return v;
}

// complex64: 8 squares (two float4) summed in FP32, then accumulated in FP64.
__global__ void __launch_bounds__(256) k_norm_c64(const float4 *__restrict__ v, uint64_t npairs, uint64_t nvec,
                                                  double *__restrict__ partials) {
    double acc = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride) {
        const float4 x = v[2 * i], y = v[2 * i + 1];
        float s = x.x * x.x;
        s = fmaf(x.y, x.y, s);
        s = fmaf(x.z, x.z, s);
        s = fmaf(x.w, x.w, s);
        s = fmaf(y.x, y.x, s);
        s = fmaf(y.y, y.y, s);
        s = fmaf(y.z, y.z, s);
        s = fmaf(y.w, y.w, s);
        acc += double(s);
    }
    // odd vector count (n = 1): the last float4
    if (blockIdx.x == 0 && threadIdx.x == 0 && (nvec & 1)) {
        const float4 x = v[nvec - 1];
        acc += double(x.x) * x.x + double(x.y) * x.y + double(x.z) * x.z + double(x.w) * x.w;
    }
    const double b = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

__global__ void __launch_bounds__(256) k_norm_c128(const double2 *__restrict__ v, uint64_t namps,
                                                   double *__restrict__ partials) {
    double acc = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < namps; i += stride) {
        const double2 x = v[i];
        acc = fma(x.x, x.x, acc);
        acc = fma(x.y, x.y, acc);
    }
    const double b = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// Fixed-order final reduction of the block partials (deterministic).
__global__ void __launch_bounds__(256) k_norm_final(const double *__restrict__ partials, int np, double *out) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) acc += partials[i];
    const double b = block_sum(acc);
    if (threadIdx.x == 0) *out = b;
}

// ---------------------------------------------------------------- gather
template <typename R>
__global__ void k_gather(const C2<R> *__restrict__ psi, const uint64_t *__restrict__ idx, size_t m,
                         double2 *__restrict__ out) {
    for (size_t j = size_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m; j += size_t(gridDim.x) * blockDim.x) {
        const C2<R> a = psi[idx[j]];
        out[j] = make_double2(double(a.re), double(a.im));
    }
}

}  // namespace

int norm_partials_needed(const sv_state *) { return kNormBlocks; }

const char *gate1_kernel_name(const sv_state *h, const Gate1 &g) {
    if (h->dt == SV_ENC2B) {
        auto is = [](const Cplx &z, double re) { return z.re == re && z.im == 0.0; };
        const Cplx *u = g.u;
        if (h->n >= kEncBlockLog2) {
            if (is(u[1], 0) && is(u[2], 0) && (is(u[0], 1) || is(u[0], -1)) && (is(u[3], 1) || is(u[3], -1)))
                return "k_enc_flip";
            if (is(u[0], 0) && is(u[3], 0) && is(u[1], 1) && is(u[2], 1)) {
                if (g.target < kEncBlockLog2) return "k_enc_xin";
                if (g.control < 0 || g.control >= kEncBlockLog2) return "k_enc_xblocks";
            }
        }
        if (g.target < kEncBlockLog2 || h->n < kEncBlockLog2) return "k_enc_gate_in";
        // diagonal with u00 = 1 in the FP32 entries the kernels use: only the upper blocks
        auto zero32 = [](const Cplx &z) { return float(z.re) == 0.0f && float(z.im) == 0.0f; };
        if (zero32(u[1]) && zero32(u[2]) && float(u[0].re) == 1.0f && float(u[0].im) == 0.0f)
            return "k_enc_gate_across<diag1>";
        return "k_enc_gate_across";
    }
    const bool c64 = h->dt == SV_C64;
    if (is_phase(g)) return c64 ? "k_phase<f32>" : "k_phase<f64>";
    if (c64 && g.target == 0) return "k_gate_inner<f32>";
    return c64 ? "k_gate_across<f32>" : "k_gate_across<f64>";
}

cudaError_t launch_gate1(sv_state *h, const Gate1 &g) {
    if (h->dt == SV_C64) return gate1_impl<float>(h, g);
    if (h->dt == SV_C128) return gate1_impl<double>(h, g);
    return launch_enc_gate1(h, g);
}

// Largest small state: beyond it one CTA is slower than runs of gates on many
// (k_gate_run).  Random circuits of depth 10, one CTA against runs: complex64 10
// qubits 33 and 33 us, 11 qubits 42 and 37, 12 qubits 66 and 40; complex128 9
// qubits 82 and 58, 10 qubits 152 and 60.
int small_run_max_n(sv_dtype dt) { return dt == SV_C64 ? 10 : dt == SV_C128 ? 8 : 0; }

cudaError_t launch_small_run(sv_state *h, const Gate1 *g, size_t count) {
    // amplitudes per thread: two target bits in complex64 (10 qubits, 145 gates:
    // 35 us; 41 with one bit, 39 with three); one in complex128, whose FP64
    // chains want many warps (8 qubits, 115 gates: 60 us against 86)
    return h->dt == SV_C128 ? small_run<double, 1>(h, g, count) : small_run<float, 2>(h, g, count);
}

// States of at most 64 MiB (half of L2): a gate's pass reads and writes L2.
bool gate_runs_fit(sv_dtype dt, int n) {
    return dt != SV_ENC2B && n > small_run_max_n(dt) && n <= (dt == SV_C64 ? 23 : 22);
}

// Time of a gate in a launch of its own, and of a run of gates, in us: a
// launch, the bytes over L2 and in complex128 the FP64 operations (a run's
// FP64 work overlaps half of its traffic).  Of the diagonal gates a launch
// visits only the amplitudes that change; a run computes where a lane of the
// warp has the condition met (lanes: the state's qubits inside a warp).
double launch_us(sv_dtype dt, int n, const Gate1 &g, int kind) {
    const double amps = std::ldexp(1.0, n);
    const int first = dt == SV_C64 ? 1 : 0;  // (qubit 0 lies inside complex64's vectors)
    double part = 1.0;
    if (g.control >= first) part /= 2;
    if (is_phase(g) && g.target >= first) part /= 2;
    const double ops = kind == R_PHASE ? 4 : kind == R_GENERAL ? 8 : kind == R_HAD ? 3 : kind <= R_SYD ? 5 : 0;
    const double fp64 = dt == SV_C128 ? part * amps * ops / 0.52e6 : 0.0;
    return 1.6 + std::max(part * amps * (dt == SV_C64 ? 16 : 32) / 12e6, fp64);
}
double run_us(sv_dtype dt, int n, const GateRunHead *op, int count, uint32_t lanes) {
    // (complex64 of 23 qubits, half of L2, runs at 11 TB/s)
    const double amps = std::ldexp(1.0, n), l2 = amps * (dt == SV_C64 ? 16 : 32) / (dt == SV_C64 && n > 22 ? 11e6 : 15e6);
    double fp64 = 0.0;
    for (int k = 0; k < count && dt == SV_C128; ++k) {
        const int kind = op[k].kind;
        const int conds = __builtin_popcount(op[k].imask & ~lanes) + (kind == R_PHASE ? __builtin_popcount(op[k].rmask) : 0);
        const double ops = kind == R_PHASE ? 4 : kind == R_GENERAL ? 8 : kind <= R_SYD || kind == R_SCALE ? 2 : 0;
        fp64 += std::ldexp(ops, -conds) * amps / 0.52e6 + (kind == R_PHASE ? 0.8 : 0.0);  // (0.8: its branches)
    }
    return 2.1 + std::max(l2, l2 / 2 + fp64);
}

// Runs of gates for k_gate_run.  A run's register qubits are the targets of
// the first gates that can be applied next (at most `slots` distinct ones);
// then every gate that commutes with all the skipped gates before it joins if
// its target is one of them.  A diagonal gate that costs arithmetic waits for
// a run that holds one of its qubits (on half of the registers, not of the
// lanes) until no other gate is left; sign flips and quarter turns join at once.
// A run that its gates beat in launches of their own by a seventh is left to
// them: a few diagonal gates on a large state, which visit a quarter of it each
// (23 qubits complex64, two CZ 14.4 us in a run and 12.9 so; 22 qubits
// complex128, 21 controlled phases on neighbours 294 and 199, 20 qubits 94 and 66;
// states below 8 MiB are all launches: 15 qubits, two phases 4.2 and 6.2).
void plan_gate_runs(sv_dtype dt, int n, const std::vector<Gate1> &g, GateRuns *out) {
    constexpr size_t kWindow = 1024;  // gates looked at ahead of the first unplaced one
    // Register qubits.  A small complex128 state is bound by the FP64 pipes of
    // the few SMs that its threads fill (random circuits of depth 8: 11 qubits
    // 58 us with two, 131 with four; 15 qubits 82 and 183), a larger one by the
    // passes over L2 (22 qubits 3.08 ms with two, 3.04 with four; its Fourier
    // transform 3.17 and 2.97); complex64 15 qubits 41 us with three and 47 with
    // four, 23 qubits 545 and 495.
    const int slots = dt == SV_C128 ? (n <= 18 ? 2 : 4) : (n <= 17 ? 3 : 4);
    out->slots = slots;
    std::vector<char> placed(g.size(), 0);
    std::vector<char> phase(g.size());
    std::vector<GateRunHead> base(g.size());
    auto factors = [&](size_t i, double u[8]) {
        for (int k = 0; k < 4; ++k) {
            u[2 * k] = g[i].u[k].re;
            u[2 * k + 1] = g[i].u[k].im;
        }
    };
    for (size_t i = 0; i < g.size(); ++i) {
        phase[i] = is_phase(g[i]);
        GateRunHead &o = base[i];
        o = GateRunHead{};
        double u[8];
        factors(i, u);
        const int pf = phase_form(u);
        if (phase[i]) {
            o.kind = pf == P_GENERAL ? R_PHASE : pf == P_NEG ? R_NEG : R_TURN;
            o.arg = pf == P_I ? 1 : 3;
            continue;
        }
        const int form = gate_form(u);
        o.kind = form == G_SWAP ? R_SWAP : R_GENERAL;
        if (g[i].control >= 0) continue;
        switch (form) {
            case G_HAD:  // the gate table's 1 / sqrt(2) is one place below the rounded sqrt(1/2)
                o.kind = std::fabs(u[0] - std::sqrt(0.5)) <= 1.2e-16 ? R_HAD : R_GENERAL;
                break;
            case G_SX: o.kind = R_SX; break;
            case G_SXD: o.kind = R_SXD; break;
            case G_SY: o.kind = R_SY; break;
            case G_SYD: o.kind = R_SYD; break;
            default: break;
        }
    }
    const int owed = dt == SV_C128 ? kRunOwed<double> : kRunOwed<float>;
    int eighths = 0, halves = 0;  // factor owed: e^(i pi eighths / 4) 2^(-halves / 2)
    size_t start = 0;
    while (true) {
        while (start < g.size() && placed[start]) ++start;
        if (start == g.size()) break;
        const size_t end = std::min(g.size(), start + kWindow);
        uint64_t qs = 0, wish = 0;  // register qubits; qubits of waiting diagonal gates
        GateRun r;
        r.first = out->ops.size();
        r.ufirst = out->u.size();
        const int eighths0 = eighths, halves0 = halves;
        std::vector<int> taken;
        double alone = 0.0;
        for (int round = 0; round < 2; ++round) {  // 0: choose the qubits, 1: take the gates
            uint64_t diag = 0, any = 0;            // qubits on which a skipped gate is diagonal / is not
            const bool only_phases = qs == 0;      // (of round 1)
            if (round == 1) {
                for (uint64_t from : {wish, (uint64_t(1) << n) - 1})
                    for (int q = n - 1; q >= 0; --q)
                        if (__builtin_popcountll(qs) < slots && (from >> q & 1)) qs |= uint64_t(1) << q;
                for (int q = 0, k = 0; q < n; ++q)
                    if (qs >> q & 1) r.q[k++] = q;
            }
            for (size_t i = start; i < end && r.count + 1 < kRunMaxOps; ++i) {  // (room for a gate and R_SCALE)
                if (placed[i]) continue;
                const uint64_t t = uint64_t(1) << g[i].target;
                const uint64_t c = g[i].control < 0 ? 0 : uint64_t(1) << g[i].control;
                bool take = phase[i] ? !((t | c) & any) : !(t & (diag | any)) && !(c & any);
                if (take && round == 0) {
                    if (phase[i]) {
                        if (base[i].kind == R_PHASE) wish |= t;
                    } else if (!(qs & t) && __builtin_popcountll(qs) == slots) {
                        take = false;
                    } else {
                        qs |= t;
                    }
                } else if (take) {
                    take = phase[i] ? only_phases || base[i].kind != R_PHASE || ((t | c) & qs) : (qs & t) != 0;
                }
                if (!take) {
                    (phase[i] ? diag : any) |= t;
                    diag |= c;
                    continue;
                }
                if (round == 0) continue;
                placed[i] = 1;
                taken.push_back(int(i));
                alone += launch_us(dt, n, g[i], base[i].kind);
                ++r.count;
                out->ops.push_back(base[i]);
                GateRunHead &o = out->ops.back();
                const uint64_t cond = phase[i] ? t | c : c;
                for (int k = 0; k < slots; ++k) {
                    if (cond >> r.q[k] & 1) o.rmask |= uint8_t(1u << k);
                    if (r.q[k] == g[i].target) o.slot = uint8_t(k);
                }
                o.imask = uint32_t(cond & ~qs);
                if (o.kind <= R_SYD) {  // SX, SY: e^(i pi/4) 2^(-1/2), H: 2^(-1/2)
                    eighths += o.kind == R_SX || o.kind == R_SY ? 1 : o.kind == R_SXD || o.kind == R_SYD ? -1 : 0;
                    if (++halves == owed) {
                        GateRunHead pay{};
                        pay.kind = R_SCALE;
                        out->ops.push_back(pay);  // (o is no longer valid)
                        ++r.count;
                        halves = 0;
                    }
                } else if (o.kind == R_GENERAL || o.kind == R_PHASE) {
                    double u[8];
                    factors(i, u);
                    const double *from = o.kind == R_GENERAL ? u : u + 6;
                    const size_t len = o.kind == R_GENERAL ? 8 : 2;
                    size_t at = r.ufirst;  // the same factors again (the T gates of a run) share their place
                    while (at < out->u.size() && (at + len > out->u.size() || !std::equal(from, from + len, &out->u[at])))
                        at += 2;
                    if (at == out->u.size()) out->u.insert(out->u.end(), from, from + len);
                    o.arg = uint8_t((at - r.ufirst) / 2);
                }
            }
        }
        r.ucount = int(out->u.size() - r.ufirst);
        while (start < g.size() && placed[start]) ++start;
        uint32_t lanes = 0;  // the five lowest qubits outside the registers
        for (int q = 0; __builtin_popcount(lanes) < 5; ++q)
            if (!(qs >> q & 1)) lanes |= 1u << q;
        const bool last = start == g.size(), big = n >= (dt == SV_C64 ? 20 : 19);
        if (big && !(last && (halves0 || eighths0 & 7)) &&
            alone < 0.85 * run_us(dt, n, &out->ops[r.first], r.count, lanes)) {
            out->ops.resize(r.first);
            out->u.resize(r.ufirst);
            eighths = eighths0;
            halves = halves0;
            r.count = r.ucount = 0;
            r.alone = std::move(taken);
            out->runs.push_back(r);
            continue;
        }
        if (last) {  // the rest of the factor
            const int k = eighths & 7;
            r.odd = k & 1;
            r.quarter = k >> 1;
            halves += r.odd;  // e^(i pi / 4) = (1 + i) 2^(-1/2)
            r.m = std::ldexp(halves & 1 ? std::sqrt(0.5) : 1.0, -(halves >> 1));
        }
        out->runs.push_back(r);
    }
}

cudaError_t launch_gate_runs(sv_state *h, const GateRuns &p, const std::vector<Gate1> &g) {
    if (h->dt == SV_C128) return p.slots == 2 ? gate_runs_impl<double, 2>(h, p, g) : gate_runs_impl<double, 4>(h, p, g);
    return p.slots == 3 ? gate_runs_impl<float, 3>(h, p, g) : gate_runs_impl<float, 4>(h, p, g);
}

cudaError_t launch_set_basis(sv_state *h, uint64_t idx) {
    cudaError_t e = cudaMemsetAsync(h->data, 0, h->bytes, h->stream);
    if (e != cudaSuccess) return e;
    if (h->dt == SV_C64)
        k_set_one<float><<<1, 1, 0, h->stream>>>(static_cast<C2<float> *>(h->data), idx);
    else if (h->dt == SV_C128)
        k_set_one<double><<<1, 1, 0, h->stream>>>(static_cast<C2<double> *>(h->data), idx);
    else
        k_enc_set_one<<<1, 1, 0, h->stream>>>(static_cast<char2 *>(h->data), h->scales, idx);
    return cudaGetLastError();
}

cudaError_t launch_norm(sv_state *h, double *d_out) {
    const uint64_t namps = uint64_t(1) << h->n;
    if (h->dt == SV_C64) {
        const uint64_t nvec = namps / 2 ? namps / 2 : 1;
        k_norm_c64<<<kNormBlocks, 256, 0, h->stream>>>(static_cast<const float4 *>(h->data), nvec / 2, nvec,
                                                       h->d_partials);
    } else if (h->dt == SV_C128) {
        k_norm_c128<<<kNormBlocks, 256, 0, h->stream>>>(static_cast<const double2 *>(h->data), namps,
                                                        h->d_partials);
    } else {
        return cudaErrorInvalidValue;  // encoded norm goes through launch_enc_norm
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_norm_final<<<1, 256, 0, h->stream>>>(h->d_partials, kNormBlocks, d_out);
    return cudaGetLastError();
}

cudaError_t launch_gather(sv_state *h, const uint64_t *d_idx, size_t m, double *d_out) {
    if (m == 0) return cudaSuccess;
    const int blocks = int((m + 255) / 256 < 1024 ? (m + 255) / 256 : 1024);
    if (h->dt == SV_C64)
        k_gather<float><<<blocks, 256, 0, h->stream>>>(static_cast<const C2<float> *>(h->data), d_idx, m,
                                                       reinterpret_cast<double2 *>(d_out));
    else if (h->dt == SV_C128)
        k_gather<double><<<blocks, 256, 0, h->stream>>>(static_cast<const C2<double> *>(h->data), d_idx, m,
                                                        reinterpret_cast<double2 *>(d_out));
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace sv
