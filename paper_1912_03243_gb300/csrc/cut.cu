// Decomposition of entangling gates across partitions (Sec. 4, Eq. 2-3).
//
// Rewrite (host): the qubits fall into P partitions.  Every CZ or CP between
// two partitions becomes a branch slot k; a CX between them is first written
// as H CZ H on its target.  Decomposition forms (a = the gate's first qubit,
// b = its second):
//   projector: CP_ab(th) = P0(a) (x) 1 + P1(a) (x) P(th)(b)   (weight 1)
//   Eq. 2:     CZ_ab = 1/2 sum_{s=+-1} D_s(a) (x) D_s(b),
//              D_s = exp(i sigma^z (x s - pi/4)), cos 2x = i  (weight 1/2 each)
// so the circuit is a sum over s in {0,1}^S of a product of circuits that
// each act on one partition (Sec. 4), and <z|C|0> = sum_s prod_p
// <z_p|W_p(s)|0_p> (Eq. 3).  W_p depends only on the bits of the cuts that
// touch partition p.
//
// Batched simulation (GPU): for each partition p the branch vectors are one
// vector of 2^(n_p + S_p) complex64 amplitudes whose top index bits are the
// S_p branch bits of the cuts touching p.
// A branch operator is then an ordinary diagonal gate coupling a half's qubit
// to branch bit k (the projector zeroes amplitudes where bit a != s_k; P(th)
// and D_s are phases selected by (bit, s_k)).  Branch bits only ever appear
// in diagonal gates, so the tile planner keeps them outside the tiles (a
// constant per CTA) and every pass runs over all branches of a half in one
// launch.
//
// Stages (branch-prefix sharing).  The gates before a branch bit's first
// operator are the same for both its values, so a stage of gates runs on the
// branches that are live, and the vector forks to the next branch bits
// between stages: the first pass of a stage reads the previous stage's smaller
// vector once per new branch and writes its own, so a fork costs no copy, and
// a stage of nothing but branch operators joins the next stage's first pass
// (prepend_diagonals: the same factors in the same order).  The last stage
// runs in chunks of its top branch bits on one buffer (kChunkQubits), only the
// amplitudes that the bit strings name are kept of each chunk, and its last
// pass runs on the tiles that hold one: the 48-qubit grid of 256 branches
// needs 4.3 GB instead of 64 GB, whose cudaFree alone took 24 ms.
//
// Sum (GPU): one warp per output bit string (its partition indices gathered
// from the string's bits by the first P lanes), lanes over s, products of the
// P partitions' amplitudes and the sum in FP64, times the weight.
//
// 48-qubit grid (2 x 24 qubits, 256 branches, 1024 strings): 161 ms with a copy
// and a pass for every branch bit and both halves' vectors whole, 72 ms with
// stages, chunks and wanted tiles, 64 ms with zero tiles written without
// computing (now: bound by the last stage's three passes over 2 x 2^32
// amplitudes, HBM and FP32 alike).  (Levels by light cone, each gate on as few branches as its operators
// allow, would take 27 ms, but reorder gates and so round differently.)
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdlib>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "plan.h"
#include "tile.h"

namespace sv {
namespace {

using cd = std::complex<double>;

__global__ void k_branch_init(float2 *psi, int np, int S) {
    const uint64_t ns = uint64_t(1) << S;
    for (uint64_t s = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < ns; s += uint64_t(gridDim.x) * blockDim.x)
        psi[s << np] = make_float2(1.0f, 0.0f);
}

constexpr int kMaxParts = 16;
constexpr int kMaxPartQubits = 40;  // a partition's state, like any state
constexpr int kMaxCutBits = 24;     // branch bits of one partition
constexpr int kMaxCutQubits = 128;  // qubits of the circuit

struct CutSumArgs {
    int P, Sv, nwords;
    int accumulate;  // add to out (the sum over several branch parts) instead of writing it
    uint64_t m;
    double w;
    const float2 *vec[kMaxParts];
    int nlocal[kMaxParts], nbits[kMaxParts];
    uint8_t cutbit[kMaxParts][kMaxCutBits];      // partition bit j <- batched branch bit cutbit[p][j]
    uint8_t qubit[kMaxParts][kMaxPartQubits];    // partition qubit i <- circuit qubit qubit[p][i]
    uint8_t table[kMaxParts];  // vec[p] holds the strings' amplitudes only: branch s of string j at s m + j
};

// The index of every bit string inside one partition.
__global__ void k_cut_index(const uint64_t *__restrict__ z, const CutSumArgs a, int p, uint64_t *__restrict__ zl) {
    for (uint64_t j = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < a.m; j += uint64_t(gridDim.x) * blockDim.x) {
        uint64_t v = 0;
        for (int i = 0; i < a.nlocal[p]; ++i) {
            const int q = a.qubit[p][i];
            v |= ((z[j * a.nwords + (q >> 6)] >> (q & 63)) & 1ull) << i;
        }
        zl[j] = v;
    }
}

// Keep the strings' amplitudes of a chunk of branches: out[s m + j] =
// vec[(s << nlocal) | zl[j]].
__global__ void k_cut_keep(const float2 *__restrict__ vec, const uint64_t *__restrict__ zl, uint64_t m, int nlocal,
                           uint64_t nbranch, float2 *__restrict__ out) {
    const uint64_t total = nbranch * m;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t s = i / m, j = i - s * m;
        out[i] = vec[(s << nlocal) | zl[j]];
    }
}

__global__ void k_cut_sum(const uint64_t *__restrict__ z, const CutSumArgs a, double2 *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const size_t warps = size_t(gridDim.x) * (blockDim.x >> 5);
    const uint64_t ns = uint64_t(1) << a.Sv;
    for (size_t j = size_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); j < a.m; j += warps) {
        // lane p < P: the index of z_j inside partition p
        uint64_t mine = 0;
        if (lane < a.P)
            for (int i = 0; i < a.nlocal[lane]; ++i) {
                const int q = a.qubit[lane][i];
                mine |= ((z[j * a.nwords + (q >> 6)] >> (q & 63)) & 1ull) << i;
            }
        uint64_t zl[kMaxParts];
#pragma unroll
        for (int p = 0; p < kMaxParts; ++p) zl[p] = __shfl_sync(0xffffffffu, mine, p);
        double re = 0.0, im = 0.0;
        for (uint64_t s = lane; s < ns; s += 32) {
            double pr = 1.0, pi = 0.0;
            for (int p = 0; p < a.P; ++p) {
                uint64_t sp = 0;
                for (int k = 0; k < a.nbits[p]; ++k) sp |= ((s >> a.cutbit[p][k]) & 1ull) << k;
                const float2 v = a.vec[p][a.table[p] ? sp * a.m + j : (sp << a.nlocal[p]) | zl[p]];
                const double r = pr * v.x - pi * v.y;
                pi = pr * v.y + pi * v.x;
                pr = r;
            }
            re += pr;
            im += pi;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (lane == 0) {
            double2 v = make_double2(a.w * re, a.w * im);
            if (a.accumulate) {
                const double2 o = out[j];
                v.x += o.x;
                v.y += o.y;
            }
            out[j] = v;
        }
    }
}

// Eq. 2 factor for branch bit value sb (0 <-> s = +1, 1 <-> s = -1):
// exp(i sigma^z phi) = diag(e^{i phi}, e^{-i phi}), phi = x s - pi/4.
void eq2_diag(int sb, cd d[2]) {
    const cd x = std::acos(cd(0.0, 1.0)) / 2.0;  // cos 2x = i, principal branch
    const double s = sb ? -1.0 : 1.0;
    const cd phi = x * s - 3.14159265358979323846 / 4.0;
    d[0] = std::exp(cd(0, 1) * phi);
    d[1] = std::exp(-cd(0, 1) * phi);
}

PGate phase_gate(uint64_t mask, uint64_t val, cd ph) {
    PGate g{};
    g.kind = 1;
    g.target = -1;
    g.cmask = mask;
    g.cval = val;
    g.u[0] = Cplx{ph.real(), ph.imag()};
    g.scale = Cplx{1, 0};
    return g;
}

// Lower one instruction acting inside a half (qubits already local).
void append_lowered(const Instr &ins, std::vector<PGate> *out) {
    Circuit one;
    one.n = 64;
    one.instrs.push_back(ins);
    const std::vector<PGate> g = lower_for_tiles(one);
    out->insert(out->end(), g.begin(), g.end());
}

// A stage of a partition's simulation: compiled passes over the vector whose
// first `level` branch bits are live.
struct HalfStage {
    std::vector<void *> fns;
    int level = 0, rb = 0;
    uint64_t last_tile = 0;  // tile qubits of the last pass
};

struct Half {            // one partition
    int nlocal = 0;     // qubits of the partition
    int nbits = 0;      // batched branch bits of the cuts touching it
    int nq = 0;         // qubits of the batched vector (local + branch, padded to a tile)
    std::vector<PGate> gates;
    std::vector<int> qubits;   // circuit qubit of local qubit i
    std::vector<int> cutbits;  // batched branch bit of partition bit j
    float2 *d = nullptr;       // the whole vector, or (chunked) the strings' amplitudes
    bool init_all = false;     // every branch starts at its own |0> (no prefix sharing)
    bool remap = false;        // stages read the previous stage's vector (else copies in place)
    int chunk = 0;             // branch bits of a chunk of the last stage (nbits: one chunk)
    std::vector<unsigned> want;  // chunked: the tiles of the last pass that hold a string's index (empty: all)
    const unsigned *d_want = nullptr;
    std::vector<HalfStage> stages;
};

// Plan and compile a stage as tiled passes over 2^nrun amplitudes, with the
// pure branch-operator stages `before` it in its first pass.  With *remap the
// passes read one vector and write another, which needs every branch bit
// outside the tiles; *remap is cleared where that fails.
sv_status plan_stage(HalfStage *st, const std::vector<std::vector<PGate>> &before, const std::vector<PGate> &gates,
                     int nlocal, int nrun, bool *remap) {
    if (gates.empty()) return SV_OK;
    TilePlan<float> tp;
    sv_status s = plan_tiles<float>(gates, nrun, tile_config64(), &tp);
    if (!s) s = prepend_diagonals(before, &tp);
    if (s) return s;
    for (const TilePassArgs &pa : tp.passes) *remap = *remap && int(pa.tile_pos[tp.m - 1]) < nlocal;
    tp.remap = *remap;
    st->rb = tp.rb;
    st->last_tile = 0;
    for (int k = 0; k < tp.m && !tp.passes.empty(); ++k) st->last_tile |= uint64_t(1) << tp.passes.back().tile_pos[k];
    return jit_tile_plan(tp, &st->fns);
}

// Branch-prefix sharing (on unless SV_CUT_PREFIX=0).
bool prefix_sharing() {
    const char *e = std::getenv("SV_CUT_PREFIX");
    return !(e && e[0] == '0');
}

// Schedules by partition content (its gates, sizes, branch-bit count and the
// code-generation settings): a repeated decomposition skips the planning, and
// the compiled passes it names stay loaded for the process.
struct Schedule {
    bool init_all, remap;
    std::vector<HalfStage> stages;
};
std::mutex g_sched_mu;
std::unordered_map<std::string, Schedule> g_sched;
constexpr size_t kSchedCacheMax = 256;

std::string schedule_key(const Half &h, int S, bool remap) {
    std::string k = std::to_string(h.nlocal) + "," + std::to_string(h.nq) + "," + std::to_string(S) + "," +
                    std::to_string(int(prefix_sharing())) + "," + std::to_string(int(remap)) + "," +
                    tile_config_name(tile_config64()) + "," + tile_codegen_key() + "," + std::to_string(plan_lookahead_width()) + "|";
    int dev = 0;
    cudaGetDevice(&dev);
    k += std::to_string(dev) + "|";
    for (const PGate &g : h.gates) {
        k.append(reinterpret_cast<const char *>(&g.kind), sizeof g.kind);
        k.append(reinterpret_cast<const char *>(&g.target), sizeof g.target);
        k.append(reinterpret_cast<const char *>(&g.cmask), sizeof g.cmask);
        k.append(reinterpret_cast<const char *>(&g.cval), sizeof g.cval);
        k.append(reinterpret_cast<const char *>(g.u), sizeof g.u);
        k.append(reinterpret_cast<const char *>(&g.scale), sizeof g.scale);
    }
    return k;
}

sv_status plan_half_uncached(Half &h, int S, bool remap);

// The schedule of a partition: planned and compiled once, then run for every
// branch part (the fixed branch bits of a part are launch parameters).
// remap: stages may read the previous stage's vector; else copies in place,
// which need no memory besides the vector.
sv_status plan_half(Half &h, int S, bool remap) {
    const std::string key = schedule_key(h, S, remap);
    {
        std::lock_guard<std::mutex> lock(g_sched_mu);
        auto it = g_sched.find(key);
        if (it != g_sched.end()) {
            h.init_all = it->second.init_all;
            h.remap = it->second.remap;
            h.stages = it->second.stages;
            return SV_OK;
        }
    }
    const sv_status s = plan_half_uncached(h, S, remap);
    if (s) return s;
    std::lock_guard<std::mutex> lock(g_sched_mu);
    if (g_sched.size() >= kSchedCacheMax) g_sched.clear();
    g_sched[key] = Schedule{h.init_all, h.remap, h.stages};
    return SV_OK;
}

sv_status plan_half_uncached(Half &h, int S, bool remap_ok) {
    h.stages.clear();
    h.init_all = !prefix_sharing();
    h.remap = remap_ok && !h.init_all && h.nlocal >= tile_config64().m;
    if (h.init_all) {
        HalfStage st;
        st.level = S;
        const sv_status s = plan_stage(&st, {}, h.gates, h.nlocal, h.nq, &h.remap);
        h.stages.push_back(std::move(st));
        return s;
    }
    // the gates between the first operators of successive branch bits, in
    // circuit order; entry k runs with k branch bits live
    std::vector<std::vector<PGate>> at(size_t(S) + 1);
    {
        int live = 0;
        for (const PGate &g : h.gates) {
            // batched branch bits are only ever conditions of diagonal gates
            const uint64_t branch = g.kind == 1 ? ((g.cmask & kQubitBits) >> h.nlocal) : 0;
            while (branch >> live) ++live;
            at[size_t(live)].push_back(g);
        }
    }
    auto diagonal = [](const std::vector<PGate> &gates) {
        for (const PGate &g : gates)
            if (g.kind != 1 || g.scale.re != 1.0 || g.scale.im != 0.0) return false;
        return true;
    };
    for (int attempt = 0; attempt < 2; ++attempt) {
        h.stages.clear();
        const bool remap = h.remap;
        std::vector<std::vector<PGate>> before;
        for (int k = 0; k <= S; ++k) {
            if (k > 0 && k < S && diagonal(at[size_t(k)])) {  // joins the next stage (if it is not empty)
                if (!at[size_t(k)].empty()) before.push_back(at[size_t(k)]);
                continue;
            }
            HalfStage st;
            st.level = k;
            const int nrun = k == S ? h.nq : std::max(h.nlocal + k, kTileM64);
            const sv_status s = plan_stage(&st, before, at[size_t(k)], h.nlocal, nrun, &h.remap);
            if (s) return s;
            before.clear();
            h.stages.push_back(std::move(st));
        }
        if (h.remap == remap) break;  // (a stage whose tiles hold branch bits: all of them in place)
    }
    return SV_OK;
}

// Amplitudes of the last stage's buffer above which it runs in chunks, and
// the room the strings' amplitudes may take.
constexpr int kChunkQubits = 28;
constexpr size_t kKeepBytes = size_t(1) << 30;

void choose_chunk(Half &h, size_t m) {
    h.chunk = h.nbits;
    if (!h.remap || h.nlocal + h.nbits <= kChunkQubits || h.stages.size() < 2) return;
    if ((m << h.nbits) * sizeof(float2) > kKeepBytes) return;
    const int prev = h.stages[h.stages.size() - 2].level;
    h.chunk = std::min(h.nbits, std::max(prev, std::max(0, kChunkQubits - h.nlocal)));
}

// The tiles of a chunked partition's last pass that hold an amplitude of one
// of the m strings (each tile of every branch needs running only if it does):
// 1024 strings name 39% of the 2048 tiles of 24 qubits.
void choose_tiles(Half &h, size_t m, const uint64_t *z, int nwords) {
    h.want.clear();
    if (h.chunk >= h.nbits) return;  // (a chunked partition has at least a tile's qubits)
    if (m > uint64_t(1) << (h.nlocal - tile_config64().m)) return;
    const uint64_t tile = h.stages.back().last_tile;
    for (size_t j = 0; j < m; ++j) {
        uint64_t t = 0;
        int k = 0;
        for (int i = 0; i < h.nlocal; ++i) {
            if (tile >> i & 1) continue;
            const int q = h.qubits[size_t(i)];
            t |= ((z[j * size_t(nwords) + size_t(q >> 6)] >> (q & 63)) & 1u) << k++;
        }
        h.want.push_back(unsigned(t));
    }
    std::sort(h.want.begin(), h.want.end());
    h.want.erase(std::unique(h.want.begin(), h.want.end()), h.want.end());
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Where the stages' vectors are: two areas, by turns, because a stage reads
// the previous one's vector only.  The last stage's area is the chunk buffer,
// or h.d itself where the last stage runs whole (the stages before it that
// share the area are smaller); the other is workspace.
int stage_area(const Half &h, size_t i) { return int((h.stages.size() - 1 - i) & 1); }
bool area_in_work(const Half &h, int area) { return area == 1 || h.chunk < h.nbits; }
size_t area_bytes(const Half &h, int area) {
    size_t b = 0;
    for (size_t i = 0; i < h.stages.size(); ++i) {
        const int live = i + 1 == h.stages.size() ? h.chunk : h.stages[i].level;
        if (stage_area(h, i) == area) b = std::max(b, sizeof(float2) << (h.nlocal + live));
    }
    return align256(b);
}

// Bytes of the areas in the workspace.
size_t work_bytes(const Half &h) {
    size_t b = 0;
    for (int area = 0; area < 2; ++area)
        if (h.remap && area_in_work(h, area)) b += area_bytes(h, area);
    return b;
}

// Bytes of h.d.
size_t result_bytes(const Half &h, size_t m) {
    return h.chunk < h.nbits ? (m << h.nbits) * sizeof(float2) : sizeof(float2) << h.nq;
}

// Run a partition's schedule for the branch part whose fixed bits are param.
// work: work_bytes(h); zl: the strings' indices in this partition (chunked).
sv_status exec_half(Half &h, cudaStream_t st, int S, uint64_t param, char *work, const uint64_t *zl, size_t m) {
    if (!h.remap) {
        // in place: the live amplitudes grow by copies (zeros above them up to one tile)
        const size_t live = sizeof(float2) << (h.nlocal > kTileM64 ? h.nlocal : kTileM64);
        SV_CUDA_TRY(cudaMemsetAsync(h.d, 0, h.init_all ? sizeof(float2) << h.nq : live, st));
        if (h.init_all) k_branch_init<<<64, 256, 0, st>>>(h.d, h.nlocal, S);
        else k_branch_init<<<1, 32, 0, st>>>(h.d, h.nlocal, 0);
        sv_status s = check_launch(cudaGetLastError(), "k_branch_init");
        if (s) return s;
        sv_state tmp;
        tmp.dt = SV_C64;
        tmp.data = h.d;
        tmp.stream = st;
        SV_CUDA_TRY(cudaGetDevice(&tmp.device));
        int level = h.init_all ? S : 0;
        for (const HalfStage &stage : h.stages) {
            for (; level < stage.level; ++level) {
                const size_t bytes = sizeof(float2) << (h.nlocal + level);
                const cudaError_t e =
                    cudaMemcpyAsync(reinterpret_cast<char *>(h.d) + bytes, h.d, bytes, cudaMemcpyDeviceToDevice, st);
                if (e != cudaSuccess) return cuda_status(e, "cudaMemcpyAsync (branch fork)");
            }
            tmp.n = h.init_all ? h.nq : std::max(h.nlocal + level, kTileM64);
            for (void *fn : stage.fns) {
                s = check_launch(launch_jit_pass(&tmp, fn, tmp.n, stage.rb, param), "branch pass");
                if (s) break;
            }
            if (s) break;
        }
        tmp.data = nullptr;
        return s;
    }
    const int tile = tile_config64().m;
    auto tiles = [&](int level) { return uint64_t(1) << (h.nlocal + level - tile); };
    float2 *area[2];
    for (int k = 0; k < 2; ++k) {
        area[k] = area_in_work(h, k) ? reinterpret_cast<float2 *>(work) : h.d;
        if (area_in_work(h, k)) work += area_bytes(h, k);
    }
    const float2 *src = nullptr;
    int src_level = 0;
    for (size_t i = 0; i < h.stages.size(); ++i) {
        const HalfStage &stage = h.stages[i];
        const bool last = i + 1 == h.stages.size();
        const int live = last ? h.chunk : stage.level;  // branch bits of this stage's vector
        float2 *dst = area[stage_area(h, i)];
        if (i == 0) {  // |0...0> of branch 0
            SV_CUDA_TRY(cudaMemsetAsync(dst, 0, sizeof(float2) << h.nlocal, st));
            k_branch_init<<<1, 32, 0, st>>>(dst, h.nlocal, 0);
            const sv_status s = check_launch(cudaGetLastError(), "k_branch_init");
            if (s) return s;
            src = dst;
        }
        for (uint64_t c = 0; c < uint64_t(1) << (stage.level - live); ++c) {
            const float2 *from = src;
            uint64_t smask = tiles(src_level) - 1;
            const uint64_t dmask = tiles(live) - 1;
            for (size_t k = 0; k < stage.fns.size(); ++k) {
                RemapTiles r{from, dst, c * tiles(live), tiles(live), smask, dmask};
                if (smask < dmask) {
                    // a fork: the tiles that read the same source tile run next
                    // to each other, so that HBM delivers it once (2^28
                    // amplitudes from 2^25: 598 us in plain order, 446 so)
                    r.group = smask + 1;
                    r.rot = unsigned(live - src_level);
                }
                if (last && h.d_want && k + 1 == stage.fns.size()) {
                    r.list = h.d_want;
                    r.nlist = unsigned(h.want.size());
                    r.group = tiles(0);
                    r.ntiles = uint64_t(h.want.size()) << live;
                }
                const sv_status s = check_launch(launch_jit_remap(stage.fns[k], stage.rb, r, param, st), "branch pass");
                if (s) return s;
                from = dst;
                smask = dmask;
            }
            if (last && h.chunk < h.nbits) {
                const uint64_t nb = uint64_t(1) << live;
                const uint64_t blocks = (nb * m + 255) / 256;
                k_cut_keep<<<unsigned(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(dst, zl, m, h.nlocal, nb,
                                                                                    h.d + c * nb * m);
                const sv_status s = check_launch(cudaGetLastError(), "k_cut_keep");
                if (s) return s;
            }
        }
        src = dst;
        src_level = live;
    }
    return SV_OK;
}

}  // namespace
}  // namespace sv

using namespace sv;

// Sum over the branches s with s mod 2^plog in the list plist (plog = 0,
// plist = {0}: all of them).  For each listed part the low plog branch bits
// are fixed: their branch operators are plain diagonal gates on the
// partitions' qubits, and only the other S - plog bits are batched; the parts
// run one after another on the same device buffers and their sums add up in
// FP64 on the device.  z: m bit strings of nwords 64-bit words (qubit q is bit
// q % 64 of word q / 64).
static sv_status cut_impl(const char *text, int n, const uint8_t *part_of, int P, int form, const uint64_t *plist,
                          size_t nlist, int plog, size_t m, const uint64_t *z, int nwords, double *out, int *n_cut_out,
                          void *stream) {
    if (n < 2 || n > kMaxCutQubits || P < 2 || P > kMaxParts || !part_of || (form != 0 && form != 1) ||
        nwords != (n + 63) / 64 || (m > 0 && (!z || !out))) {
        set_error("bad arguments (n=%d, P=%d, form=%d, nwords=%d)", n, P, form, nwords);
        return SV_ERR_ARG;
    }
    Half parts[kMaxParts];
    int side[kMaxCutQubits], loc[kMaxCutQubits];
    for (int q = 0; q < n; ++q) {
        if (part_of[q] >= P) {
            set_error("qubit %d: partition %d outside 0..%d", q, int(part_of[q]), P - 1);
            return SV_ERR_ARG;
        }
        side[q] = part_of[q];
        loc[q] = parts[side[q]].nlocal++;
        parts[side[q]].qubits.push_back(q);
    }
    for (int p = 0; p < P; ++p)
        if (parts[p].nlocal == 0) {
            set_error("partition %d has no qubits", p);
            return SV_ERR_ARG;
        }
    const int top = n - 64 * (nwords - 1);  // qubits in the last word
    for (size_t j = 0; j < m; ++j)
        if (top < 64 && (z[j * nwords + nwords - 1] >> top)) {
            set_error("bit string %zu has bits above qubit %d", j, n - 1);
            return SV_ERR_ARG;
        }
    Circuit c;
    sv_status s = parse_circuit(text, n, &c);
    if (s) return s;

    // count the decomposed gates first
    int S = 0;
    for (const Instr &ins : c.instrs) {
        if (ins.nq != 2 || side[ins.q[0]] == side[ins.q[1]]) continue;
        if (ins.name == "SWAP") {
            set_error("a SWAP across partitions cannot be decomposed");
            return SV_ERR_UNSUPPORTED;
        }
        if (form == 1 && ins.name == "CP") {
            set_error("the Eq. 2 form decomposes CZ only (CP across partitions)");
            return SV_ERR_UNSUPPORTED;
        }
        ++S;
    }
    if (n_cut_out) *n_cut_out = S;
    if (S - plog > 16) {
        set_error("%d decomposed gates, %d of them batched (at most 16)", S, S - plog);
        return SV_ERR_UNSUPPORTED;
    }
    const int Svar = S > plog ? S - plog : 0;  // batched branch bits
    if (n_cut_out) *n_cut_out = S;
    // the listed parts that hold branches (a part whose low bits exceed every
    // branch index has none)
    std::vector<uint64_t> todo;
    for (size_t i = 0; i < nlist; ++i)
        if (!(S < 64 && (plist[i] >> S) != 0)) todo.push_back(plist[i]);
    if (todo.empty()) {
        for (size_t j = 0; j < 2 * m; ++j) out[j] = 0.0;
        return SV_OK;
    }
    // branch operators: a Z-basis projector (or Eq. 2 phase) on the first
    // qubit's partition, the phase on the second's, conditioned on the cut's
    // branch bit, which each partition holds above its own qubits
    auto build = [&]() -> sv_status {
    for (int p = 0; p < P; ++p) {
        parts[p].gates.clear();
        parts[p].cutbits.clear();
        parts[p].nbits = 0;
    }
    int k = 0;
    for (const Instr &ins0 : c.instrs) {
        Instr ins = ins0;
        if (ins.nq == 1 || side[ins.q[0]] == side[ins.q[1]]) {
            const int p = side[ins.q[0]];
            for (int j = 0; j < ins.nq; ++j) ins.q[j] = loc[ins.q[j]];
            append_lowered(ins, &parts[p].gates);
            continue;
        }
        const int qa = ins.q[0], qb = ins.q[1];
        Half &A = parts[side[qa]], &B = parts[side[qb]];
        const double theta = ins.name == "CP" ? ins.p[0] : 3.14159265358979323846;
        Instr h;
        h.name = "H";
        h.nq = 1;
        if (ins.name == "CX") {  // CX = H_t CZ H_t
            h.q[0] = loc[qb];
            append_lowered(h, &B.gates);
        }
        const uint64_t la = uint64_t(1) << loc[qa], lb = uint64_t(1) << loc[qb];
        // a fixed branch bit (one of the low plog) is a launch parameter bit:
        // the same compiled passes serve every part
        const bool fixed = k < plog;
        uint64_t ka = uint64_t(1) << (kParamBit0 + k), kb = ka;
        if (!fixed) {
            if (A.nbits >= kMaxCutBits || B.nbits >= kMaxCutBits) {
                set_error("a partition touches more than %d batched cuts", kMaxCutBits);
                return SV_ERR_UNSUPPORTED;
            }
            A.cutbits.push_back(k - plog);
            B.cutbits.push_back(k - plog);
            ka = uint64_t(1) << (A.nlocal + A.nbits++);
            kb = uint64_t(1) << (B.nlocal + B.nbits++);
        }
        if (form == 0) {
            A.gates.push_back(phase_gate(la | ka, la, 0.0));  // bit a = 1, s_k = 0: P0 removes it
            A.gates.push_back(phase_gate(la | ka, ka, 0.0));  // bit a = 0, s_k = 1: P1 removes it
            B.gates.push_back(phase_gate(lb | kb, lb | kb, std::polar(1.0, theta)));
        } else {
            for (int sb = 0; sb < 2; ++sb) {
                cd d[2];
                eq2_diag(sb, d);
                const uint64_t sva = sb ? ka : 0, svb = sb ? kb : 0;
                A.gates.push_back(phase_gate(la | ka, sva, d[0]));
                A.gates.push_back(phase_gate(la | ka, la | sva, d[1]));
                B.gates.push_back(phase_gate(lb | kb, svb, d[0]));
                B.gates.push_back(phase_gate(lb | kb, lb | svb, d[1]));
            }
        }
        if (ins.name == "CX") append_lowered(h, &B.gates);
        ++k;
    }
    for (int p = 0; p < P; ++p) {
        Half &h = parts[p];
        h.nq = h.nlocal + h.nbits < kTileM64 ? kTileM64 : h.nlocal + h.nbits;
        if (h.nlocal > kMaxPartQubits || h.nq > kMaxQubits) {
            set_error("partition %d needs %d qubits (local %d + %d branch bits)", p, h.nq, h.nlocal, h.nbits);
            return SV_ERR_UNSUPPORTED;
        }
    }
    return SV_OK;
    };
    s = build();
    if (s) return s;
    if (m == 0) return SV_OK;

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // device memory: the vectors (or kept amplitudes), one workspace for the
    // partitions, which run one after another, bit strings, indices, results
    size_t bytesV = 0, bytesW = 0, bytesI = 0, total = 0;
    const size_t bytesZ = align256(m * size_t(nwords) * sizeof(uint64_t)), bytesO = align256(m * sizeof(double2));
    size_t free_b = 0, total_b = 0, least = 0;
    for (int p = 0; p < P; ++p) {
        s = plan_half(parts[p], parts[p].nbits, true);
        if (s) return s;
        choose_chunk(parts[p], m);
        choose_tiles(parts[p], m, z, nwords);
    }
    // Where the stages' own vectors do not fit beside the results, partitions
    // whose last stage runs whole take the schedule in place (no vector but
    // the result), and where that does not fit either, every partition.
    for (int attempt = 0;; ++attempt) {
        auto in_place = [&](const Half &h) { return attempt == 2 || (attempt == 1 && h.chunk == h.nbits); };
        bytesV = bytesW = bytesI = 0;
        for (int p = 0; p < P; ++p) {
            const Half &h = parts[p];
            if (in_place(h)) {
                bytesV += align256(sizeof(float2) << h.nq);
                continue;
            }
            bytesV += align256(result_bytes(h, m)) + align256(h.want.size() * sizeof(unsigned));
            bytesW = std::max(bytesW, work_bytes(h));
            if (h.chunk < h.nbits) bytesI = align256(m * sizeof(uint64_t));
        }
        total = bytesV + bytesW + bytesZ + bytesO + bytesI;
        least = attempt == 0 ? total : std::min(least, total);
        SV_CUDA_TRY(cudaMemGetInfo(&free_b, &total_b));
        if (total + (size_t(256) << 20) <= free_b) {
            for (int p = 0; p < P; ++p) {
                if (!in_place(parts[p]) || !parts[p].remap) continue;
                s = plan_half(parts[p], parts[p].nbits, false);
                if (s) return s;
                choose_chunk(parts[p], m);
                choose_tiles(parts[p], m, z, nwords);
            }
            break;
        }
        if (attempt == 2) {
            set_error("decomposition needs %zu bytes of device memory, %zu free", least, free_b);
            return SV_ERR_OOM;
        }
    }
    if (fault_injected("alloc")) {
        set_error("injected allocation failure");
        return SV_ERR_OOM;
    }
    char *mem = nullptr;
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&mem), total);
    if (e != cudaSuccess) return cuda_status(e, "cudaMalloc (decomposition)");
    char *at = mem;
    auto take = [&](size_t b) {
        char *r = at;
        at += b;
        return r;
    };
    for (int p = 0; p < P; ++p) parts[p].d = reinterpret_cast<float2 *>(take(align256(result_bytes(parts[p], m))));
    char *work = take(bytesW);
    uint64_t *dz = reinterpret_cast<uint64_t *>(take(bytesZ));
    double2 *dout = reinterpret_cast<double2 *>(take(bytesO));
    uint64_t *dzl = reinterpret_cast<uint64_t *>(take(bytesI));
    CutSumArgs a{};
    a.P = P;
    a.Sv = Svar;
    a.nwords = nwords;
    a.m = m;
    a.w = form == 1 ? std::ldexp(1.0, -S) : 1.0;
    for (int p = 0; p < P; ++p) {
        a.vec[p] = parts[p].d;
        a.nlocal[p] = parts[p].nlocal;
        a.nbits[p] = parts[p].nbits;
        a.table[p] = parts[p].chunk < parts[p].nbits;
        for (int j = 0; j < parts[p].nbits; ++j) a.cutbit[p][j] = uint8_t(parts[p].cutbits[size_t(j)]);
        for (int i = 0; i < parts[p].nlocal; ++i) a.qubit[p][i] = uint8_t(parts[p].qubits[size_t(i)]);
    }
    e = cudaMemcpyAsync(dz, z, m * size_t(nwords) * sizeof(uint64_t), cudaMemcpyHostToDevice, st);
    for (int p = 0; p < P && e == cudaSuccess; ++p) {
        parts[p].d_want = nullptr;
        if (parts[p].want.empty()) continue;
        const size_t b = parts[p].want.size() * sizeof(unsigned);
        unsigned *w = reinterpret_cast<unsigned *>(take(align256(b)));
        e = cudaMemcpyAsync(w, parts[p].want.data(), b, cudaMemcpyHostToDevice, st);
        parts[p].d_want = w;
    }
    if (e != cudaSuccess) s = cuda_status(e, "cudaMemcpyAsync");
    const size_t blocks = (m + 7) / 8 < 4096 ? (m + 7) / 8 : 4096;
    for (size_t ip = 0; ip < todo.size() && s == SV_OK; ++ip) {
        // every part runs the same compiled passes (its fixed branch bits are
        // the launch parameter) on the same buffers; the stream orders its
        // halves after the previous part's sum
        for (int p = 0; p < P && s == SV_OK; ++p) {
            if (a.table[p]) {
                k_cut_index<<<unsigned(blocks), 256, 0, st>>>(dz, a, p, dzl);
                s = check_launch(cudaGetLastError(), "k_cut_index");
                if (s) break;
            }
            s = exec_half(parts[p], st, parts[p].nbits, todo[ip], work, dzl, m);
        }
        if (s != SV_OK) break;
        a.accumulate = ip > 0;
        k_cut_sum<<<unsigned(blocks), 256, 0, st>>>(dz, a, dout);
        s = check_launch(cudaGetLastError(), "k_cut_sum");
    }
    if (s == SV_OK) {
        e = cudaMemcpyAsync(out, dout, m * sizeof(double2), cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) s = cuda_status(e, "cudaMemcpyAsync");
    }
    if (s == SV_OK) s = sync_stream(st, "sv_cut_amplitudes");
    if (s != SV_OK) cudaStreamSynchronize(st);
    cudaFree(mem);
    return s;
}

// Two partitions given by a mask (partition 0 = the mask's qubits).
static sv_status cut_mask(const char *text, int n, uint64_t maskA, int form, const uint64_t *plist, size_t nlist,
                          int plog, size_t m, const uint64_t *z, double *out, int *n_cut_out, void *stream) {
    if (n < 2 || n > 64) {
        set_error("n = %d outside 2..64 (sv_cut_amplitudes_multi takes up to %d qubits)", n, kMaxCutQubits);
        return SV_ERR_ARG;
    }
    const uint64_t all = n == 64 ? ~uint64_t(0) : ((uint64_t(1) << n) - 1);
    if ((maskA & all) == 0 || (maskA & all) == all || (maskA & ~all)) {
        set_error("maskA must select a proper, nonempty subset of the %d qubits", n);
        return SV_ERR_ARG;
    }
    uint8_t part_of[64];
    for (int q = 0; q < n; ++q) part_of[q] = (maskA >> q & 1) ? 0 : 1;
    return cut_impl(text, n, part_of, 2, form, plist, nlist, plog, m, z, 1, out, n_cut_out, stream);
}

// A list of branch parts: each < 2^plog and none repeated.
static sv_status check_parts(const uint64_t *plist, size_t nlist, int plog) {
    if (plog < 0 || plog > 16 || nlist == 0 || nlist > (size_t(1) << plog) || !plist) {
        set_error("bad part list (%zu parts of 2^%d)", nlist, plog);
        return SV_ERR_ARG;
    }
    std::vector<char> seen(size_t(1) << plog, 0);
    for (size_t i = 0; i < nlist; ++i) {
        if ((plist[i] >> plog) != 0 || seen[plist[i]]) {
            set_error("part %llu at position %zu is out of range or repeated (2^%d parts)",
                      (unsigned long long)plist[i], i, plog);
            return SV_ERR_ARG;
        }
        seen[plist[i]] = 1;
    }
    return SV_OK;
}

extern "C" sv_status sv_cut_amplitudes(const char *text, int n, uint64_t maskA, int form, size_t m, const uint64_t *z,
                                       double *out, int *n_cut_out, void *stream) {
    const uint64_t all = 0;
    return cut_mask(text, n, maskA, form, &all, 1, 0, m, z, out, n_cut_out, stream);
}

extern "C" sv_status sv_cut_amplitudes_parts(const char *text, int n, uint64_t maskA, int form, int nparts_log2,
                                             size_t nlist, const uint64_t *parts, size_t m, const uint64_t *z,
                                             double *out, int *n_cut_out, void *stream) {
    sv_status s = check_parts(parts, nlist, nparts_log2);
    return s ? s : cut_mask(text, n, maskA, form, parts, nlist, nparts_log2, m, z, out, n_cut_out, stream);
}

extern "C" sv_status sv_cut_amplitudes_multi_parts(const char *text, int n, const uint8_t *part_of, int P, int form,
                                                   int nparts_log2, size_t nlist, const uint64_t *parts, size_t m,
                                                   const uint64_t *z, double *out, int *n_cut_out, void *stream) {
    sv_status s = check_parts(parts, nlist, nparts_log2);
    return s ? s
             : cut_impl(text, n, part_of, P, form, parts, nlist, nparts_log2, m, z, (n + 63) / 64, out, n_cut_out,
                        stream);
}

extern "C" sv_status sv_cut_amplitudes_part(const char *text, int n, uint64_t maskA, int form, uint64_t part,
                                            int nparts_log2, size_t m, const uint64_t *z, double *out, int *n_cut_out,
                                            void *stream) {
    if (nparts_log2 < 0 || nparts_log2 > 16 || (part >> nparts_log2) != 0) {
        set_error("bad part %llu of 2^%d", (unsigned long long)part, nparts_log2);
        return SV_ERR_ARG;
    }
    return cut_mask(text, n, maskA, form, &part, 1, nparts_log2, m, z, out, n_cut_out, stream);
}

extern "C" sv_status sv_cut_amplitudes_multi(const char *text, int n, const uint8_t *part_of, int P, int form,
                                             uint64_t part, int nparts_log2, size_t m, const uint64_t *z,
                                             double *out, int *n_cut_out, void *stream) {
    if (nparts_log2 < 0 || nparts_log2 > 16 || (part >> nparts_log2) != 0) {
        set_error("bad part %llu of 2^%d", (unsigned long long)part, nparts_log2);
        return SV_ERR_ARG;
    }
    return cut_impl(text, n, part_of, P, form, &part, 1, nparts_log2, m, z, (n + 63) / 64, out, n_cut_out, stream);
}
