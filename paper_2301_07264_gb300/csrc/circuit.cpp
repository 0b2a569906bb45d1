// Circuit compiler: gate matrices, error-location table, fused pass schedule.
//
// A circuit (Sec. II) is a list of one- and two-qubit gates. Every gate gets
// one error location per qubit (Sec. IV-B.2: a two-qubit gate draws an error
// on each of its qubits), so L = k + 2m (Eq. (3)).
//
// Engines:
//  * resident  - the whole 2^n state lives in one CTA's shared memory for the
//                entire circuit (n <= 13 for complex64, 12 for complex128);
//  * streaming - the state lives in HBM and is swept by fused passes. A pass
//                is a set of t "tile qubits" (always including the low qubits
//                0..c-1 so that global accesses stay contiguous) and a list of
//                gates acting only on tile qubits; each CTA loads one tile of
//                2^t amplitudes into shared memory, applies all of the pass's
//                gates (and the trajectory's error gates that follow them),
//                and writes the tile back: one HBM round trip per pass.
//
// The pass builder chooses each pass's tile qubits, then places gates in
// circuit order: a gate joins the pass when its qubits are tile qubits and none
// is blocked; otherwise its qubits become blocked for the rest of the pass, and
// so does every later gate that touches a blocked qubit. The set of gates
// placed in a pass is therefore closed under the circuit's dependencies, and
// concatenating the passes gives an engine order that is a valid topological
// reordering of the circuit. Error gates stay attached to the gate they
// follow, which keeps them correct: a gate moved ahead of gate g never touches
// g's qubits after g. The tile set starts from the low qubits and the qubits of
// the first unplaced gate and grows one qubit at a time, each time by the qubit
// whose addition places the most gates (lowest index on ties); when no single
// qubit adds a gate, it takes the qubits of the earliest gate still left out.
#include <algorithm>
#include <set>
#include <cmath>
#include <cstring>
#include <functional>

#include "internal.h"

namespace arso {

using cd = std::complex<double>;

void matrix_for(const arso_gate &g, HostGate &h) {
    const double s2 = 1.0 / std::sqrt(2.0);
    const double th = g.param;
    const cd I(0, 1);
    for (auto &v : h.m) v = 0;
    auto set2 = [&](cd a, cd b, cd c, cd d) { h.m[0] = a; h.m[1] = b; h.m[2] = c; h.m[3] = d; };
    switch (g.kind) {
        case ARSO_GATE_ID: set2(1, 0, 0, 1); h.cls = GC_NOP; break;
        case ARSO_GATE_H: set2(s2, s2, s2, -s2); h.cls = GC_H; break;
        case ARSO_GATE_X: set2(0, 1, 1, 0); h.cls = GC_X; break;
        case ARSO_GATE_Y: set2(0, -I, I, 0); h.cls = GC_DENSE1; break;
        // diag(1, e^{i k pi/4}): Z (k=4), S (2), SDG (6), T (1), TDG (7)
        case ARSO_GATE_Z: set2(1, 0, 0, -1); h.cls = GC_OMEGA; h.omega_k = 4; break;
        case ARSO_GATE_S: set2(1, 0, 0, I); h.cls = GC_OMEGA; h.omega_k = 2; break;
        case ARSO_GATE_SDG: set2(1, 0, 0, -I); h.cls = GC_OMEGA; h.omega_k = 6; break;
        case ARSO_GATE_T: set2(1, 0, 0, std::polar(1.0, M_PI / 4)); h.cls = GC_OMEGA; h.omega_k = 1; break;
        case ARSO_GATE_TDG: set2(1, 0, 0, std::polar(1.0, -M_PI / 4)); h.cls = GC_OMEGA; h.omega_k = 7; break;
        case ARSO_GATE_RX:
            set2(std::cos(th / 2), -I * std::sin(th / 2), -I * std::sin(th / 2), std::cos(th / 2));
            h.cls = GC_DENSE1;
            break;
        case ARSO_GATE_RY:
            set2(std::cos(th / 2), -std::sin(th / 2), std::sin(th / 2), std::cos(th / 2));
            h.cls = GC_DENSE1;
            break;
        case ARSO_GATE_RZ: set2(std::polar(1.0, -th / 2), 0, 0, std::polar(1.0, th / 2)); h.cls = GC_DIAG1; break;
        case ARSO_GATE_P: set2(1, 0, 0, std::polar(1.0, th)); h.cls = GC_DIAG1; break;
        case ARSO_GATE_U:
            ARSO_REQUIRE(g.matrix != nullptr, "U gate needs a 2x2 matrix");
            for (int i = 0; i < 4; ++i) h.m[i] = cd(g.matrix[2 * i], g.matrix[2 * i + 1]);
            h.cls = GC_DENSE1;
            break;
        case ARSO_GATE_CX:
            for (int i = 0; i < 4; ++i) h.m[5 * i] = 1;
            h.m[5] = 0; h.m[15] = 0; h.m[1 * 4 + 3] = 1; h.m[3 * 4 + 1] = 1;
            h.cls = GC_CX;
            break;
        case ARSO_GATE_CZ:
            h.m[0] = 1; h.m[5] = 1; h.m[10] = 1; h.m[15] = -1; h.cls = GC_CZ; break;
        case ARSO_GATE_CP:
            h.m[0] = 1; h.m[5] = 1; h.m[10] = 1; h.m[15] = std::polar(1.0, th); h.cls = GC_DIAG2; break;
        case ARSO_GATE_SWAP:
            h.m[0] = 1; h.m[15] = 1; h.m[1 * 4 + 2] = 1; h.m[2 * 4 + 1] = 1; h.cls = GC_SWAP; break;
        case ARSO_GATE_U2:
            ARSO_REQUIRE(g.matrix != nullptr, "U2 gate needs a 4x4 matrix");
            for (int i = 0; i < 16; ++i) h.m[i] = cd(g.matrix[2 * i], g.matrix[2 * i + 1]);
            h.cls = GC_DENSE2;
            break;
        default: throw Error(ARSO_EINVAL, "unknown gate kind " + std::to_string(g.kind));
    }
    for (int i = 0; i < (h.arity == 1 ? 4 : 16); ++i)
        ARSO_REQUIRE(std::isfinite(h.m[i].real()) && std::isfinite(h.m[i].imag()), "non-finite gate matrix entry");
}

// gates [first, G) that a pass with tile set in_s would place (circuit order,
// blocked-qubit rule); returns their number and, when `out` is given, their indices
static size_t pass_closure(const arso_circuit *c, const std::vector<char> &done, size_t first,
                           const std::vector<char> &in_s, std::vector<uint32_t> *out) {
    const uint32_t n = c->n;
    std::vector<char> blocked(n, 0);
    uint32_t n_blocked = 0;
    size_t cnt = 0;
    for (size_t g = first; g < c->gates.size() && n_blocked < n; ++g) {
        if (done[g]) continue;
        const HostGate &h = c->gates[g];
        const uint32_t qs[2] = {h.q0, h.q1};
        bool ok = true;
        for (int j = 0; j < h.arity; ++j) ok &= !blocked[qs[j]] && in_s[qs[j]];
        if (ok) {
            ++cnt;
            if (out) out->push_back((uint32_t)g);
        } else {
            for (int j = 0; j < h.arity; ++j)
                if (!blocked[qs[j]]) blocked[qs[j]] = 1, ++n_blocked;
        }
    }
    return cnt;
}

static void schedule_streaming(arso_circuit *c) {
    const uint32_t n = c->n, t = c->tile_qubits, lowq = c->low_qubits;
    const size_t G = c->gates.size();
    std::vector<char> done(G, 0);
    size_t remaining = G, first = 0;
    c->passes.clear();
    c->perm.clear();
    do {
        std::vector<char> in_s(n, 0);
        uint32_t cnt = 0;
        auto add = [&](uint32_t q) {
            if (!in_s[q]) in_s[q] = 1, ++cnt;
        };
        for (uint32_t q = 0; q < lowq; ++q) add(q);
        if (first < G) {
            add(c->gates[first].q0);
            add(c->gates[first].q1);
        }
        size_t placed = pass_closure(c, done, first, in_s, nullptr);
        while (cnt < t) {
            size_t best = placed;
            uint32_t bq = n;
            for (uint32_t q = 0; q < n; ++q) {
                if (in_s[q]) continue;
                in_s[q] = 1;
                const size_t k = pass_closure(c, done, first, in_s, nullptr);
                in_s[q] = 0;
                if (k > best) best = k, bq = q;
            }
            if (bq < n) {
                add(bq);
                placed = best;
                continue;
            }
            // no single qubit places another gate: the earliest gate left out that fits
            std::vector<uint32_t> in_pass;
            pass_closure(c, done, first, in_s, &in_pass);
            std::vector<char> placed_g(G, 0);
            for (uint32_t g : in_pass) placed_g[g] = 1;
            bool grown = false;
            for (size_t g = first; g < G && !grown; ++g) {
                if (done[g] || placed_g[g]) continue;
                const HostGate &h = c->gates[g];
                const uint32_t fresh = (in_s[h.q0] ? 0u : 1u) + (h.arity == 2 && !in_s[h.q1] ? 1u : 0u);
                if (fresh && cnt + fresh <= t) {
                    add(h.q0);
                    add(h.q1);
                    grown = true;
                }
            }
            if (!grown) break;
            placed = pass_closure(c, done, first, in_s, nullptr);
        }
        // pad the tile to exactly t qubits (lowest unused qubits first)
        for (uint32_t q = 0; q < n && cnt < t; ++q) add(q);
        Pass p;
        p.gb = (uint32_t)c->perm.size();
        std::vector<uint32_t> in_pass;
        pass_closure(c, done, first, in_s, &in_pass);
        ARSO_REQUIRE(!in_pass.empty() || G == 0, "internal: the pass builder placed no gate");
        for (uint32_t g : in_pass) {
            done[g] = 1;
            --remaining;
            c->perm.push_back(g);
        }
        while (first < G && done[first]) ++first;
        for (uint32_t q = 0; q < n; ++q)
            if (in_s[q]) p.tile_qubits.push_back(q);
        p.ge = (uint32_t)c->perm.size();
        c->passes.push_back(std::move(p));
    } while (remaining > 0);
}

// Register-bit phases of each pass. A gate that mixes amplitudes needs its
// mixing qubit among the REG_BITS register bits (dense one-qubit gates and H:
// their qubit; CX: its target); diagonal gates, X, and the dense two-qubit
// gates and SWAP (run through shared memory) act on any bit. Tile bit 0 is a
// register bit in every phase (the register kernels pack amplitudes j and
// j|1 into one FP32x2 register pair).
//
// Within a pass the gates may run in any order that respects their qubit
// dependencies. The planner list-schedules them: with register set R it runs
// every ready gate whose need is in R, repeatedly; when none is left it picks
// the next R among all sets of tile bit 0 and four other tile bits by the
// weighted number of gates the closure under R would run. Passes start and
// end in the load/store mapping {0, t-4, t-3, t-2, t-1}, whose thread bits
// 1..t-5 keep global accesses contiguous.
static constexpr uint32_t NO_NEED = 0xFFFFFFFFu;

static uint32_t need_of(const HostGate &h, uint32_t lq0, uint32_t lq1) {
    switch (h.cls) {
        case GC_DENSE1: case GC_H: case GC_PROBE: return lq0;
        case GC_CX: return lq1;
        default: return NO_NEED;
    }
}

// relative cost of a gate in the register kernels (the planner's objective)
static double gate_weight(const HostGate &h) {
    switch (h.cls) {
        case GC_DENSE1: case GC_H: return 1.0;
        case GC_DENSE2: case GC_SWAP: return 2.0;
        case GC_DIAG1: case GC_OMEGA: return 0.5;
        default: return 0.25;
    }
}

namespace {
// Dependency DAG of one pass and a list scheduler with trial closures.
struct PassScheduler {
    uint32_t G;
    std::vector<uint32_t> need;    // tile bits that have to be register bits, as a mask
    std::vector<double> weight;
    std::vector<std::vector<uint32_t>> succ;
    std::vector<uint32_t> indeg;
    std::vector<uint32_t> ready;   // unscheduled gates whose predecessors are all scheduled, ascending (at most t:
                                   // they act on distinct qubits)
    std::vector<uint32_t> order;
    // Tensor-phase rules: a gate runs under R when all its qubits are in R (a
    // diagonal one always, another one while none of its qubits is frozen) or
    // when it is diagonal. A diagonal gate with qubits in and out of R freezes
    // its qubits in R that a non-diagonal gate of the phase already acted on.
    bool tensor = false;
    std::vector<uint8_t> diag;    // diagonal in the computational basis
    std::vector<uint32_t> qmask;  // tile-local qubits of the gate
    std::vector<uint32_t> undo, rd, blocked;  // working lists of closure

    bool runs(uint32_t g, uint32_t Rm, uint32_t frozen) const {
        if (!tensor) return (need[g] & ~Rm) == 0;
        if ((qmask[g] & ~Rm) == 0) return diag[g] || !(qmask[g] & frozen);
        return diag[g] != 0;
    }
    // Run every ready gate that runs under the register set Rm, lowest index first, repeatedly.
    // With `trial` the state is restored afterwards and only the weight is returned; without
    // tensor rules the gates that run do not depend on the order, and a trial takes them as they
    // come. A gate that does not run never does later under the same set: the frozen qubits only
    // grow. Planning the probe circuits of a 14-qubit circuit of 600 random gates, 1,482 gates: 11.0
    // ms with ordered sets and a scan from the first gate after every step, 2.3 ms so.
    double closure(uint32_t Rm, bool trial) {
        double w = 0.0;
        uint32_t started = 0, frozen = 0;
        const bool ordered = !trial || tensor;
        undo.clear();
        blocked.clear();
        rd.assign(ready.rbegin(), ready.rend());  // descending: the lowest is the last
        while (!rd.empty()) {
            const uint32_t g = rd.back();
            rd.pop_back();
            if (!runs(g, Rm, frozen)) {
                blocked.push_back(g);
                continue;
            }
            w += weight[g];
            if (tensor) {
                if ((qmask[g] & ~Rm) == 0) started |= diag[g] ? 0u : qmask[g];
                else frozen |= qmask[g] & Rm & started;
            }
            if (!trial) order.push_back(g);
            for (uint32_t s : succ[g]) {
                if (trial) undo.push_back(s);
                if (--indeg[s]) continue;
                if (ordered) rd.insert(std::upper_bound(rd.begin(), rd.end(), s, std::greater<uint32_t>()), s);
                else rd.push_back(s);
            }
        }
        if (trial) {
            for (uint32_t s : undo) ++indeg[s];
        } else {
            ready = blocked;
            std::sort(ready.begin(), ready.end());
        }
        return w;
    }
};
}  // namespace

// algorithmic FP32 flops per amplitude of one gate (see the tracing section of arso.h)
static double gate_flops(const HostGate &h) {
    switch (h.cls) {
        case GC_DENSE1: return 14.0;
        case GC_DENSE2: return 30.0;
        case GC_DIAG1: case GC_DIAG2: return 6.0;
        case GC_H: return 4.0;
        case GC_OMEGA: return (h.omega_k & 1u) ? 2.0 : 0.0;
        default: return 0.0;
    }
}

static bool is_diagonal(const HostGate &h) {
    switch (h.cls) {
        case GC_NOP: case GC_DIAG1: case GC_DIAG2: case GC_OMEGA: case GC_CZ: return true;
        default: return false;
    }
}

// U <- G U for gate h on register positions p0 (and p1) of the 32-dimensional
// register index (two-qubit matrices index bit(q0) + 2 bit(q1), row-major)
static void left_apply(std::vector<std::complex<double>> &U, const HostGate &h, uint32_t p0, uint32_t p1) {
    const uint32_t b0 = 1u << p0, b1 = 1u << p1;
    for (uint32_t col = 0; col < 32; ++col) {
        auto at = [&](uint32_t row) -> std::complex<double> & { return U[row * 32 + col]; };
        for (uint32_t l = 0; l < 32; ++l) {
            if (h.arity == 1) {
                if (l & b0) continue;
                const std::complex<double> x0 = at(l), x1 = at(l | b0);
                at(l) = h.m[0] * x0 + h.m[1] * x1;
                at(l | b0) = h.m[2] * x0 + h.m[3] * x1;
            } else {
                if (l & (b0 | b1)) continue;
                const uint32_t ix[4] = {l, l | b0, l | b1, l | b0 | b1};
                std::complex<double> x[4], y[4];
                for (int k = 0; k < 4; ++k) x[k] = at(ix[k]);
                for (int r = 0; r < 4; ++r) {
                    y[r] = 0;
                    for (int k = 0; k < 4; ++k) y[r] += h.m[4 * r + k] * x[k];
                }
                for (int k = 0; k < 4; ++k) at(ix[k]) = y[k];
            }
        }
    }
}

// Nearest binary16 value of x (ties to even; |x| < 65504), as bits; *v gets its value.
static uint16_t f16_bits(double x, double *v) {
    const double ax = std::fabs(x);
    const uint16_t sign = std::signbit(x) ? 0x8000u : 0u;
    if (ax == 0.0) {
        *v = 0.0;
        return sign;
    }
    int e;
    std::frexp(ax, &e);                      // ax in [2^(e-1), 2^e)
    const int E = std::max(e - 1, -14);      // below 2^-14 the spacing stays 2^-24 (subnormals)
    const double q = std::ldexp(1.0, E - 10);
    const double r = std::nearbyint(ax / q) * q;  // round to nearest, ties to even
    *v = sign ? -r : r;
    if (r < std::ldexp(1.0, -14)) return (uint16_t)(sign | (uint16_t)std::ldexp(r, 24));
    int er;
    const double fr = std::frexp(r, &er);    // r = fr 2^er, fr in [0.5, 1)
    const uint32_t mant = (uint32_t)std::ldexp(fr, 11) - 1024u;
    return (uint16_t)(sign | (uint16_t)((er - 1 + 15) << 10) | (uint16_t)mant);
}

// Roles of the records of phase ph (positions [gb, ge), tile-local qubits lq0/lq1
// indexed from pass_gb) and, when the phase qualifies, its operand images: the
// real 64 x 64 form of U in packed-register order on both sides (index 4p + 2c +
// lane for register 2p + lane, c = 0 real part, 1 imaginary part), B[n][k] with
// D[row][n] = sum_k A[row][k] B[n][k], scaled by 2^8 and split into the integer
// hi = rint(2^8 B) (|hi| <= 256, exact in fp16) and lo = fp16(2^8 B - hi).
static void tensor_phase(arso_circuit *c, uint32_t ph, uint32_t gb, uint32_t ge, uint32_t pass_gb,
                         const std::vector<uint32_t> &lq0, const std::vector<uint32_t> &lq1) {
    uint32_t R[REG_BITS], Rm = 0;
    int rp[32];
    std::fill(rp, rp + 32, -1);
    for (int b = 0; b < REG_BITS; ++b) {
        R[b] = (c->ph_R[ph] >> (5 * b)) & 31u;
        Rm |= 1u << R[b];
        rp[R[b]] = b;
    }
    std::vector<std::complex<double>> U(32 * 32, 0.0);
    for (int i = 0; i < 32; ++i) U[i * 33] = 1.0;
    uint32_t started = 0, frozen = 0;
    int dense = 0;
    bool ok = true;
    for (uint32_t pos = gb; pos < ge; ++pos) {
        const HostGate &h = c->gates[c->perm[pos]];
        const uint32_t a = lq0[pos - pass_gb], b = lq1[pos - pass_gb];
        const uint32_t qm = (1u << a) | (1u << b);
        const bool dg = is_diagonal(h);
        if ((qm & ~Rm) == 0) {
            c->role[pos] = TR_CORE;
            if (!dg) {
                ok &= (qm & frozen) == 0;
                started |= qm;
                ++dense;
            }
            left_apply(U, h, (uint32_t)rp[a], (uint32_t)rp[b]);
        } else {
            ok &= dg;
            const bool after = (qm & Rm & started) != 0;
            c->role[pos] = after ? TR_AFTER : TR_BEFORE;
            frozen |= qm & Rm & started;
        }
    }
    if (!ok || dense < TENSOR_MIN_DENSE) return;
    c->ph_t[ph] = (uint32_t)(c->tmats.size() / TENSOR_IMAGE_HALVES);
    const size_t base = c->tmats.size();
    c->tmats.resize(base + TENSOR_IMAGE_HALVES);
    uint16_t *hi = c->tmats.data() + base, *lo = hi + TENSOR_IMAGE_HALVES / 2;
    for (uint32_t n = 0; n < 64; ++n)
        for (uint32_t k = 0; k < 64; ++k) {
            const uint32_t j = 2 * (n >> 2) + (n & 1u), l = 2 * (k >> 2) + (k & 1u);
            const uint32_t co = (n >> 1) & 1u, ci = (k >> 1) & 1u;
            const std::complex<double> u = U[j * 32 + l];
            const double val = co == 0 ? (ci == 0 ? u.real() : -u.imag()) : (ci == 0 ? u.imag() : u.real());
            double vh, vl;
            const uint32_t off = ((n >> 3) * 1024 + (k >> 3) * 128 + (n & 7u) * 16 + (k & 7u) * 2) / 2;
            const double x = std::ldexp(val, 8), xi = std::nearbyint(x);
            hi[off] = f16_bits(xi, &vh);
            lo[off] = f16_bits(x - xi, &vl);
        }
}

static float2 f2(cd v) { return make_float2((float)v.real(), (float)v.imag()); }

// what to add to the real part of f, a constant rounded to FP32, for the exact modulus; next to
// the imaginary axis, where that would turn f more than its rounding did, for the exact real part
static float real_gap(cd exact, float2 f) {
    const double n = std::norm(exact), x = f.x;
    return (float)(8.0 * x * x > n ? (n - std::norm(cd(f.x, f.y))) / (2.0 * x) : exact.real() - x);
}

static cd omega(int k) {
    static const double s = std::sqrt(0.5);
    static const cd w[8] = {cd(1, 0), cd(s, s), cd(0, 1), cd(-s, s), cd(-1, 0), cd(-s, -s), cd(0, -1), cd(s, -s)};
    return w[k & 7];
}

// a unit phase: exactly omega^k when within rounding of it (k returned, else -1)
static int snap(cd &v) {
    v /= std::abs(v);
    for (int k = 0; k < 8; ++k)
        if (std::abs(v - omega(k)) < 1e-13) {
            v = omega(k);
            return k;
        }
    return -1;
}

// ------------------------------------------------------------ fused runs ---
// A run of gates on at most three qubits whose product is a permutation that flips one
// qubit c under a condition on the others, with phases that are a frame (RegOpCode) times
// signs; or, on two qubits, a diagonal. Toffoli networks, CX conjugations of rotations and
// H pairs around either are such runs: one conditional move (or one phase, or nothing)
// instead of some fifteen gates. Measured before and after: 16-rate sweep of the 12-qubit
// Grover circuit 122.6 -> 31.9 ms, 20-qubit adder 3.24 -> 1.87 ms, 32 uneven circuits
// 55.7 -> 48.7 ms.
struct FusedRun {
    uint32_t q[3];      // the qubits (global), n of them
    int n = 0;
    int c = -1;         // index of the flipped qubit in q; -1: none
    uint32_t f = 0;     // flip where bit x of f is set, x = the old values of the qubits
    cd d[8];            // |x> -> d[x] |x ^ flip>
};

// A run counts as such within RUN_TOL: above the rounding of a product of 40 matrices (a few
// 1e-15), and far below what FP32 amplitudes resolve of a small rotation's own amplitude. What
// was accepted is written with ten times that, so a value at the edge cannot fail there.
constexpr double RUN_TOL = 1e-13;

static uint32_t run_target(const FusedRun &r, uint32_t x) { return r.c >= 0 && (r.f >> x & 1) ? x ^ (1u << r.c) : x; }

// the phases of a run between the frames phi (in) and out: residual signs by new value y, or,
// without a flip and on two qubits, theta of one parity phase. False: neither.
static bool run_phases(const FusedRun &r, const cd *phi, cd &S, cd *out, uint32_t &signs, double &theta,
                       double tol = RUN_TOL) {
    const uint32_t N = 1u << r.n;
    cd e[8];
    for (uint32_t x = 0; x < N; ++x) {
        cd v = r.d[x];
        for (int k = 0; k < r.n; ++k)
            if (x >> k & 1) v *= phi[k];
        e[run_target(r, x)] = v;
    }
    S = e[0];
    for (int k = 0; k < r.n; ++k) {
        out[k] = e[1u << k] / e[0];
        snap(out[k]);
    }
    signs = 0;
    theta = 0.0;
    bool ok = true;
    cd res[8];
    for (uint32_t y = 0; y < N; ++y) {
        cd v = S;
        for (int k = 0; k < r.n; ++k)
            if (y >> k & 1) v *= out[k];
        res[y] = e[y] / v;
        if (std::abs(res[y] + 1.0) < tol) signs |= 1u << y;
        else ok &= std::abs(res[y] - 1.0) < tol;
    }
    if (ok) return true;
    if (r.c >= 0 || r.n != 2) return false;
    // e^{i theta ab} = e^{i theta a / 2} e^{i theta b / 2} e^{-i theta (a ^ b) / 2}
    signs = 0;
    theta = std::arg(res[3]);
    for (int k = 0; k < 2; ++k) out[k] *= std::polar(1.0, theta / 2);
    return true;
}

// The product of a run's gates so far: M[x] is the column of |x>, on the first n qubits of q.
struct RunMatrix {
    cd M[8][8];
    int n = 0;
    RunMatrix() { M[0][0] = 1.0; }
    // one more qubit, on which the product so far is the identity
    void widen() {
        const uint32_t N = 1u << n++;
        for (uint32_t x = 0; x < N; ++x)
            for (uint32_t y = 0; y < N; ++y) M[x + N][y + N] = M[x][y], M[x][y + N] = M[x + N][y] = 0.0;
    }
    // M <- h M, by what the gate does: CX moves entries, a diagonal matrix scales them
    void apply(const uint32_t *q, const HostGate &h) {
        int k0 = 0, k1 = 0;
        for (int k = 0; k < n; ++k) {
            if (q[k] == h.q0) k0 = k;
            if (q[k] == h.q1) k1 = k;
        }
        const uint32_t N = 1u << n, b0 = 1u << k0, b1 = 1u << k1;
        if (h.arity == 1) {
            const cd m0 = h.m[0], m1 = h.m[1], m2 = h.m[2], m3 = h.m[3];
            const bool diag = m1 == 0.0 && m2 == 0.0;
            for (uint32_t col = 0; col < N; ++col)
                for (uint32_t x = 0; x < N; ++x) {
                    if (x & b0) continue;
                    cd &a0 = M[col][x], &a1 = M[col][x | b0];
                    const cd v0 = a0, v1 = a1;
                    if (diag) a0 = m0 * v0, a1 = m3 * v1;
                    else a0 = m0 * v0 + m1 * v1, a1 = m2 * v0 + m3 * v1;
                }
        } else if (h.cls == GC_CX) {
            for (uint32_t col = 0; col < N; ++col)
                for (uint32_t x = 0; x < N; ++x)
                    if ((x & b0) && !(x & b1)) std::swap(M[col][x], M[col][x | b1]);
        } else {  // the other two-qubit gates of a run are diagonal (run_takes)
            for (uint32_t x = 0; x < N; ++x) {
                const cd d = h.m[5 * ((x & b0 ? 1 : 0) + (x & b1 ? 2 : 0))];
                if (d == 1.0) continue;
                for (uint32_t col = 0; col < N; ++col) M[col][x] *= d;
            }
        }
    }
};

// the gates as a fused run; false when their product is none
static bool run_of(const RunMatrix &P, FusedRun &r, double tol = RUN_TOL) {
    const cd(*M)[8] = P.M;
    const uint32_t N = 1u << r.n;
    uint32_t to[8];
    for (uint32_t x = 0; x < N; ++x) {
        int hit = -1;
        for (uint32_t y = 0; y < N; ++y) {
            const double a = std::norm(M[x][y]);
            if (a > 0.25) hit = hit < 0 ? (int)y : 8;
            else if (a > tol * tol) return false;
        }
        if (hit < 0 || hit >= 8 || std::abs(std::abs(M[x][hit]) - 1.0) > tol) return false;
        to[x] = (uint32_t)hit;
        r.d[x] = M[x][hit];
        snap(r.d[x]);
    }
    uint32_t moved = 0;
    r.f = 0;
    for (uint32_t x = 0; x < N; ++x) {
        moved |= x ^ to[x];
        if (x != to[x]) r.f |= 1u << x;
    }
    if (moved & (moved - 1)) return false;  // more than one qubit flips
    r.c = moved ? (moved == 1 ? 0 : moved == 2 ? 1 : 2) : -1;
    const cd one[3] = {1.0, 1.0, 1.0};
    cd S, out[3];
    uint32_t signs;
    double theta;
    return run_phases(r, one, S, out, signs, theta, tol);
}

// what a gate costs the kernels: 2 when it is dispatched, 1 when it may be (a phase that has
// to be applied before a later gate)
static int run_cost(const HostGate &h) {
    switch (h.cls) {
        case GC_H: case GC_DENSE1: case GC_CX: case GC_CZ: case GC_DIAG2: return 2;
        case GC_DIAG1: return 1;
        case GC_OMEGA: return (int)(h.omega_k & 1u);
        default: return 0;
    }
}
// gates that no run takes: measurements, and those that run through shared memory
static bool run_takes(const HostGate &h) { return h.cls != GC_PROBE && h.cls != GC_DENSE2 && h.cls != GC_SWAP; }

// the run that find_units accepted, from its gates
static bool product_of(const std::vector<const HostGate *> &gs, FusedRun &r) {
    r.n = 0;
    for (const HostGate *h : gs)
        for (uint32_t q : {h->q0, h->q1})
            if (std::find(r.q, r.q + r.n, q) == r.q + r.n) r.q[r.n++] = q;
    RunMatrix M;
    for (int k = 0; k < r.n; ++k) M.widen();
    for (const HostGate *h : gs) M.apply(r.q, *h);
    return run_of(M, r, 10 * RUN_TOL);
}

// The pass's gates (indices from its first position) as units in an order that keeps the
// circuit's dependencies: fused runs, and single gates. From each gate on, the run takes
// every gate it can while it stays on three qubits, passing over gates on other qubits,
// and ends after the longest prefix that is a fused run and saves more than it leaves to do
// (at least two dispatched gates, and something besides when an op remains). Planning the 32
// uneven circuits of a batch takes 82 ms of one core; the products on three qubits from the
// first gate on and the scheduler's ordered sets took it to 185, 120 without fused runs.
static std::vector<std::vector<uint32_t>> find_units(const arso_circuit *c, const Pass &ps, bool fuse) {
    const uint32_t G = ps.ge - ps.gb;
    std::vector<std::pair<uint32_t, std::vector<uint32_t>>> units;  // (last gate, gates)
    std::vector<char> taken(G, 0);
    constexpr uint32_t MAX_RUN = 40, MAX_SCAN = 256;
    std::vector<uint32_t> run;
    for (uint32_t i = 0; i < G; ++i) {
        if (taken[i]) continue;
        run.assign(1, i);
        size_t keep = 1;
        auto gate = [&](uint32_t k) -> const HostGate & { return c->gates[c->perm[ps.gb + k]]; };
        if (fuse && run_takes(gate(i))) {
            FusedRun r;
            RunMatrix M;
            int costs = 0, dispatched = 0;
            uint32_t in = 0, closed = 0;  // qubits of the run; of gates that other runs have taken
            auto add = [&](const HostGate &h) {
                for (uint32_t q : {h.q0, h.q1})
                    if (!(in >> q & 1)) in |= 1u << q, r.q[r.n++] = q, M.widen();
                M.apply(r.q, h);
                costs += run_cost(h);
                dispatched += run_cost(h) == 2;
            };
            add(gate(i));
            for (uint32_t j = i + 1; j < G && j < i + MAX_SCAN && run.size() < MAX_RUN; ++j) {
                const HostGate &h = gate(j);
                const uint32_t qs = 1u << h.q0 | 1u << h.q1;
                if (!(qs & in)) {
                    if (taken[j]) closed |= qs;
                    continue;
                }
                if (taken[j] || !run_takes(h) || (qs & ~in & closed) || r.n + __builtin_popcount(qs & ~in) > 3) break;
                add(h);
                run.push_back(j);
                if (dispatched < 2) continue;
                FusedRun t = r;
                if (run_of(M, t)) {
                    cd S, out[3];
                    const cd one[3] = {1.0, 1.0, 1.0};
                    uint32_t signs = 0;
                    double theta = 0.0;
                    run_phases(t, one, S, out, signs, theta);
                    if (costs >= 5 || (t.c < 0 && !signs && theta == 0.0)) keep = run.size();
                }
            }
        }
        run.resize(keep);
        for (uint32_t k : run) taken[k] = 1;
        units.emplace_back(run.back(), run);
    }
    std::sort(units.begin(), units.end());
    std::vector<std::vector<uint32_t>> out;
    for (auto &u : units) out.push_back(std::move(u.second));
    return out;
}

// most units of the register program (ProgWriter) that a gate takes in its phase, now or as
// the phase it leaves to apply later; qubits can bring a phase each into it (phase_units)
static uint32_t max_units(const HostGate &h) {
    switch (h.cls) {
        case GC_DENSE1: return 4;
        case GC_OMEGA: case GC_X: case GC_NOP: return 1;
        default: return 2;
    }
}
static uint32_t phase_units(uint32_t t) { return 2 * t + 1; }

static void plan_phases(arso_circuit *c) {
    const uint32_t t = c->tile_qubits;
    c->reg_blocked = c->precision == ARSO_C64 && t >= (uint32_t)RB_MIN_TILE;
    c->ph_gb.clear();
    c->ph_R.clear();
    c->rpos.assign(c->perm.size(), 0xFF);
    c->tensor = c->reg_blocked && c->engine == 1 && t >= 12 && (c->flags & ARSO_OPT_TENSOR_PHASES);
    c->ph_t.clear();
    c->tmats.clear();
    c->role.assign(c->perm.size(), (uint8_t)TR_CORE);
    if (!c->reg_blocked) return;
    const std::vector<uint32_t> load_map = {0, t - 4, t - 3, t - 2, t - 1};
    c->blocks.clear();
    for (Pass &ps : c->passes) {
        std::vector<int> local(c->n, -1);
        for (size_t i = 0; i < ps.tile_qubits.size(); ++i) local[ps.tile_qubits[i]] = (int)i;
        // what is scheduled: single gates and fused runs of them
        const std::vector<std::vector<uint32_t>> units = find_units(c, ps, !c->tensor && c->probe_loc.empty());
        const uint32_t G = (uint32_t)units.size();
        PassScheduler S;
        S.G = G;
        S.tensor = c->tensor;
        S.diag.resize(G);
        S.qmask.assign(G, 0);
        S.need.assign(G, 0);
        S.weight.assign(G, 0.0);
        S.succ.assign(G, {});
        S.indeg.assign(G, 0);
        std::vector<int> last(t, -1);
        for (uint32_t i = 0; i < G; ++i) {
            for (uint32_t k : units[i]) {
                const HostGate &h = c->gates[c->perm[ps.gb + k]];
                const uint32_t a = (uint32_t)local[h.q0], b = (uint32_t)local[h.q1], need = need_of(h, a, b);
                if (need != NO_NEED) S.need[i] |= 1u << need;
                S.weight[i] = units[i].size() > 1 ? 2.0 : gate_weight(h);
                S.diag[i] = is_diagonal(h) ? 1 : 0;
                S.qmask[i] |= (1u << a) | (1u << b);
            }
            std::set<int> before;
            for (uint32_t q = 0; q < t; ++q) {
                if (!(S.qmask[i] >> q & 1)) continue;
                if (last[q] >= 0) before.insert(last[q]);
                last[q] = (int)i;
            }
            for (int p : before) S.succ[p].push_back(i), ++S.indeg[i];
        }
        for (uint32_t i = 0; i < G; ++i)
            if (!S.indeg[i]) S.ready.push_back(i);
        ps.pb = (uint32_t)c->ph_R.size();
        std::vector<uint32_t> cur = load_map;
        std::vector<std::pair<uint32_t, std::vector<uint32_t>>> phases;  // (start in order, R)
        for (;;) {
            const size_t before = S.order.size();
            uint32_t cm = 0;
            for (uint32_t q : cur) cm |= 1u << q;
            S.closure(cm, false);
            if (S.order.size() > before) phases.emplace_back((uint32_t)before, cur);
            if (S.order.size() == G) break;
            // next register set: tile bit 0 and the 4 other tile bits whose closure runs
            // the largest weight of gates (all C(t-1, 4) sets are tried; ties keep the first)
            std::vector<uint32_t> R{0, 1, 2, 3, 4}, best;
            double best_w = -1.0;
            for (uint32_t a = 1; a < t; ++a)
                for (uint32_t b = a + 1; b < t; ++b)
                    for (uint32_t d = b + 1; d < t; ++d)
                        for (uint32_t e = d + 1; e < t; ++e) {
                            R[1] = a, R[2] = b, R[3] = d, R[4] = e;
                            const double w = S.closure(1u | 1u << a | 1u << b | 1u << d | 1u << e, true);
                            if (w > best_w + 1e-12) best_w = w, best = R;
                        }
            R = best;
            std::sort(R.begin(), R.end());
            // tensor rules: a new phase under the same set starts with nothing frozen
            ARSO_REQUIRE(best_w > 0.0 && (R != cur || S.tensor), "internal: the phase planner made no progress");
            cur = R;
        }
        if (phases.empty()) phases.emplace_back(0u, load_map);
        if (!c->tensor) {
            // within a phase: all ready two-qubit gates, then a layer of ready one-qubit gates,
            // one per qubit, in turn (reg_program gives a layer one dispatch)
            std::vector<uint32_t> where(G, 0), deg(G, 0), ord;
            for (size_t k = 0; k < phases.size(); ++k) {
                const uint32_t b = phases[k].first, e = k + 1 < phases.size() ? phases[k + 1].first : G;
                std::set<uint32_t> one, two;
                auto ready = [&](uint32_t g) {
                    (units[g].size() == 1 && c->gates[c->perm[ps.gb + units[g][0]]].arity == 1 ? one : two).insert(g);
                };
                for (uint32_t i = b; i < e; ++i) where[S.order[i]] = (uint32_t)k + 1, deg[S.order[i]] = 0;
                for (uint32_t i = b; i < e; ++i)
                    for (uint32_t x : S.succ[S.order[i]])
                        if (where[x] == k + 1) ++deg[x];
                for (uint32_t i = b; i < e; ++i)
                    if (!deg[S.order[i]]) ready(S.order[i]);
                auto emit = [&](uint32_t g) {
                    ord.push_back(g);
                    for (uint32_t x : S.succ[g])
                        if (where[x] == k + 1 && --deg[x] == 0) ready(x);
                };
                while (!one.empty() || !two.empty()) {
                    while (!two.empty()) {
                        const uint32_t g = *two.begin();
                        two.erase(two.begin());
                        emit(g);
                    }
                    const std::set<uint32_t> now = one;
                    one.clear();
                    for (int probes = 1; probes >= 0; --probes)
                        for (uint32_t g : now)
                            if ((c->gates[c->perm[ps.gb + units[g][0]]].cls == GC_PROBE) == (probes == 1)) emit(g);
                }
            }
            S.order = ord;
        }
        // the pass's new engine order; a phase longer than its staging buffer continues with the
        // same register set, a fused run staying in one piece
        const uint32_t n_gates = ps.ge - ps.gb;
        std::vector<uint32_t> perm_new;
        for (size_t k = 0; k < phases.size(); ++k) {
            ARSO_REQUIRE(phases[k].second[0] == 0, "internal: a register set without tile bit 0");
            const uint32_t end = k + 1 < phases.size() ? phases[k + 1].first : G;
            const uint32_t limit = c->tensor ? 2u * MAX_PHASE_OPS : (uint32_t)MAX_PHASE_UNITS - phase_units(t);
            uint32_t used = 0;
            c->ph_gb.push_back(ps.gb + (uint32_t)perm_new.size());
            c->ph_R.push_back(pack_rbits(phases[k].second.data()));
            for (uint32_t u = phases[k].first; u < end; ++u) {
                const std::vector<uint32_t> &unit = units[S.order[u]];
                uint32_t size = unit.size() > 1 ? 20 : 0;  // header, fused op, flush, frame repair, phases it leaves, an empty layer
                for (uint32_t i : unit) size += max_units(c->gates[c->perm[ps.gb + i]]);
                if (c->tensor) size = 2;
                if (used + size > limit) {
                    c->ph_gb.push_back(ps.gb + (uint32_t)perm_new.size());
                    c->ph_R.push_back(pack_rbits(phases[k].second.data()));
                    used = 0;
                }
                used += size;
                const uint32_t p0 = ps.gb + (uint32_t)perm_new.size();
                for (uint32_t i : unit) perm_new.push_back(c->perm[ps.gb + i]);
                if (unit.size() > 1) c->blocks.emplace_back(p0, ps.gb + (uint32_t)perm_new.size());
            }
        }
        std::copy(perm_new.begin(), perm_new.end(), c->perm.begin() + ps.gb);
        std::vector<uint32_t> lq0(n_gates), lq1(n_gates);
        for (uint32_t i = 0; i < n_gates; ++i) {
            const HostGate &h = c->gates[c->perm[ps.gb + i]];
            lq0[i] = (uint32_t)local[h.q0];
            lq1[i] = (uint32_t)local[h.q1];
        }
        ps.pe = (uint32_t)c->ph_R.size();
        // register positions of each gate's qubits within its phase
        for (uint32_t ph = ps.pb; ph < ps.pe; ++ph) {
            uint32_t R[REG_BITS];
            for (int b = 0; b < REG_BITS; ++b) R[b] = (c->ph_R[ph] >> (5 * b)) & 31u;
            const uint32_t ge = ph + 1 < ps.pe ? c->ph_gb[ph + 1] : ps.ge;
            for (uint32_t pos = c->ph_gb[ph]; pos < ge; ++pos) {
                uint32_t p0 = 15, p1 = 15;
                for (int b = 0; b < REG_BITS; ++b) {
                    if (R[b] == lq0[pos - ps.gb]) p0 = (uint32_t)b;
                    if (R[b] == lq1[pos - ps.gb]) p1 = (uint32_t)b;
                }
                c->rpos[pos] = (uint8_t)(p0 | (p1 << 4));
            }
        }
        if (c->tensor) {
            c->ph_t.resize(ps.pe, NO_TENSOR);
            for (uint32_t ph = ps.pb; ph < ps.pe; ++ph)
                tensor_phase(c, ph, c->ph_gb[ph], ph + 1 < ps.pe ? c->ph_gb[ph + 1] : ps.ge, ps.gb, lq0, lq1);
        }
    }
    for (Pass &ps : c->passes) {
        ps.flops_per_amp = 0.0;
        for (uint32_t pos = ps.gb; pos < ps.ge; ++pos) ps.flops_per_amp += gate_flops(c->gates[c->perm[pos]]);
        // shared-memory transposes of one sweep: every change of register set, from the load layout
        const uint32_t load_packed = pack_rbits(load_map.data());
        uint32_t prev = load_packed;
        ps.remaps = 0;
        for (uint32_t ph = ps.pb; ph < ps.pe; ++ph) {
            ps.remaps += c->ph_R[ph] != prev;
            prev = c->ph_R[ph];
        }
        ps.end_remap = prev != load_packed;
    }
    c->chg_prefix.assign(c->ph_R.size() + 1, 0);
    for (size_t ph = 0; ph < c->ph_R.size(); ++ph)
        c->chg_prefix[ph + 1] = c->chg_prefix[ph] + (ph > 0 && c->ph_R[ph] != c->ph_R[ph - 1]);
    c->ph_gb.push_back(c->passes.empty() ? 0 : c->passes.back().ge);  // sentinel
    c->phase_of_pos.assign(c->perm.size(), 0);
    for (size_t ph = 0; ph + 1 < c->ph_gb.size(); ++ph)
        for (uint32_t pos = c->ph_gb[ph]; pos < c->ph_gb[ph + 1]; ++pos) c->phase_of_pos[pos] = (uint32_t)ph;
}

// ------------------------------------------------------ register program ---
// op code and mask-adjustment fields of a register-kernel gate record
static uint32_t reg_opcode(uint32_t cls, uint32_t p0, uint32_t p1) {
    auto enc = [](uint32_t opc, uint32_t sa, uint32_t sb, uint32_t xa, uint32_t xb) {
        return opc | sa << 8 | sb << 10 | xa << 12 | xb << 13;
    };
    const uint32_t R = (uint32_t)REG_BITS;
    switch (cls) {
        case GC_SU2: return enc(OP_SU2 + p0, 0, 0, 0, 0);
        case GC_DENSE1: return enc(OP_DENSE1 + p0, 0, 0, 0, 0);
        case GC_H: return enc(OP_H + 2 * p0, 1, 0, 0, 0);  // + flip = bit q0 of m
        case GC_CZ: {
            if (p0 < R && p1 < R) {
                const uint32_t lo = std::min(p0, p1), hi = std::max(p0, p1);
                const uint32_t pp = lo == 0 ? hi - 1 : lo == 1 ? hi + 2 : lo == 2 ? hi + 4 : 9;
                // want = 1 ^ mask bit; the lower position carries weight 2
                return p0 < p1 ? enc(OP_CZ_RR + 4 * pp, 2, 1, 1, 1) : enc(OP_CZ_RR + 4 * pp, 1, 2, 1, 1);
            }
            if (p0 < R) return enc(OP_CZ_RT + 2 * p0, 1, 0, 1, 0);
            if (p1 < R) return enc(OP_CZ_RT + 2 * p1, 0, 1, 0, 1);
            return enc(OP_CZ_TT, 0, 0, 0, 0);
        }
        case GC_X: return enc(OP_X, 0, 0, 0, 0);
        case GC_OMEGA: return enc(OP_OMEGA, 0, 0, 0, 0);
        case GC_DIAG1: return enc(OP_DIAG1, 0, 0, 0, 0);
        case GC_DIAG2: return enc(OP_CP, 0, 0, 0, 0);
        case GC_CX: return enc(OP_CX + std::min(p1, R - 1), 0, 0, 0, 0);
        case GC_DENSE2: return enc(OP_DENSE2, 0, 0, 0, 0);
        case GC_SWAP: return enc(OP_SWAP, 0, 0, 0, 0);
        default: return enc(OP_NOP, 0, 0, 0, 0);
    }
}

// The frame of a tile: scalar S and phases phi (see RegOpCode in internal.h).
struct Frame {
    std::vector<cd> f;  // f[0] = S, f[1 + q] = phi of tile bit q
    explicit Frame(uint32_t t) : f(1 + t, cd(1, 0)) {}
    cd &S() { return f[0]; }
    cd &phi(uint32_t q) { return f[1 + q]; }
};

// Largest growth of the stored state over the true one before a gate restores its
// scale with a full matrix: G(x) grows a state by sqrt(1 + |x|^2) <= sqrt 2, so FP32's
// range would end after some 250 gates; 2^40 keeps 2^86 of headroom above it.
constexpr double FRAME_GROWTH = 1.0 / (1ull << 40);
// A matrix has a frame form when it is a unitary one times a scale: rows of one norm within
// UNITARY_TOL, orthogonal within ORTHO_TOL of the smaller entry (the form derives the second
// row from the first, so that a tiny rotation keeps its own amplitude). The scale goes into S.
// It differs from 1 by the rounding of a matrix given in 32 bits: [[a, b], [-conj b, conj a]]
// keeps its form whatever the rounding, and the frame form is what it ran as before there
// were frames (18-qubit brickwork from complex64 matrices, 500 trajectories: 8.34 ms as full
// matrices, 2.59 so, 4.78 before frames). An entry counts as zero within the rounding of the sine or cosine of
// a right angle.
constexpr double UNITARY_TOL = 1e-12, ORTHO_TOL = 1e-9, ZERO_TOL = 4.5e-16, SCALE_TOL = 1e-5;

// What a one-qubit gate becomes in a frame.
struct FrameGate {
    enum { NOP, FLIP, GIV, FULL } kind = NOP;
    bool flip = false;   // GIV: an index flip X first
    float2 x{};          // GIV
    cd m[4];             // FULL: the matrix
};

// U on a qubit with frame phase phi: what remains of it, and the frame after it
static FrameGate frame_dense(Frame &F, uint32_t q, const cd *u) {
    const cd phi = F.phi(q);
    cd u00 = u[0], u01 = u[1] * phi, u10 = u[2], u11 = u[3] * phi;
    if (std::abs(u01) < ZERO_TOL && std::abs(u10) < ZERO_TOL) u01 = u10 = 0;
    if (std::abs(u00) < ZERO_TOL && std::abs(u11) < ZERO_TOL) u00 = u11 = 0;
    const double a = std::abs(u00), b = std::abs(u01);
    const double scale2 = a * a + b * b;
    const bool unitary = std::abs(scale2 - 1.0) < SCALE_TOL && std::abs(std::norm(u10) + std::norm(u11) - scale2) < UNITARY_TOL &&
                         std::abs(u00 * std::conj(u10) + u01 * std::conj(u11)) <= ORTHO_TOL * std::min(a, b);
    FrameGate g;
    auto full = [&](cd m00, cd m01, cd m10, cd m11) {
        g.kind = FrameGate::FULL;
        g.m[0] = m00, g.m[1] = m01, g.m[2] = m10, g.m[3] = m11;
    };
    if (!unitary) {  // any matrix as it is; the frame phase goes into its columns
        full(u00, u01, u10, u11);
        F.phi(q) = 1;
        return g;
    }
    if (b == 0.0) {  // diagonal
        F.S() *= u00;
        F.phi(q) = u11 / u00;
        snap(F.phi(q));
        return g;
    }
    if (a == 0.0) {  // diag(u01, u10) X
        F.S() *= u01;
        F.phi(q) = u10 / u01;
        snap(F.phi(q));
        g.kind = FrameGate::FLIP;
        return g;
    }
    // U'' = diag(d0, d1) G(x) X^flip, the larger entry of the first row as d0
    g.flip = a < b;
    const cd d0 = g.flip ? u01 : u00, d1 = g.flip ? u10 : u11;
    float2 x = f2((g.flip ? u00 : u01) / d0);
    if (std::abs(x.x) < 1e-16f) x.x = 0.f;  // the sine and cosine of a right angle's rounding
    if (std::abs(x.y) < 1e-16f) x.y = 0.f;
    const double sc = std::sqrt(scale2 / (1.0 + (double)x.x * x.x + (double)x.y * x.y));  // exact scale of the rounded x
    F.S() *= d0 / std::abs(d0) * sc;
    F.phi(q) = d1 / d0;
    snap(F.phi(q));
    if (std::abs(F.S()) < FRAME_GROWTH) {  // rescale: G(x) X^flip times a power of two near |S|, exactly
        const double s = std::exp2(std::floor(std::log2(std::abs(F.S()))));
        const cd xs(x.x, x.y), o1(s, 0);
        if (g.flip) full(xs * s, o1, o1, -std::conj(xs) * s);
        else full(o1, xs * s, -std::conj(xs) * s, o1);
        F.S() /= s;
        return g;
    }
    g.kind = FrameGate::GIV;
    g.x = x;
    return g;
}

// Macro-ops of one phase, built gate by gate.
struct ProgWriter {
    std::vector<uint4> &out;
    size_t first;                    // first unit of the phase
    size_t last = SIZE_MAX;          // header of the last macro-op written in the phase
    bool open = false;               // a layer being collected
    uint32_t active = 0, real = 0, flips = 0, used = 0, end = 0;
    float2 x[REG_BITS];
    uint32_t probes = 0;             // register positions being measured (open is false then)
    ProbeSlot probe[REG_BITS];
    std::vector<ProbeSlot> *slots = nullptr;
    explicit ProgWriter(std::vector<uint4> &o) : out(o), first(o.size()) {}
    void close() {
        if (probes) {
            last = out.size();
            out.push_back(make_uint4(OP_PROBE | probes << 8 | 1u << 24, end, (uint32_t)slots->size(), 0));
            for (int p = 0; p < REG_BITS; ++p)
                if (probes >> p & 1) slots->push_back(probe[p]);
            probes = 0;
        }
        if (!open) return;
        open = false;
        uint32_t n = 1;
        for (int p = 0; p < REG_BITS; ++p) n += active >> p & 1;
        last = out.size();
        out.push_back(make_uint4(OP_LAYER | active << 8 | real << 13 | n << 24, end, 0, flips));
        for (int p = 0; p < REG_BITS; ++p) {
            if (!(active >> p & 1)) continue;
            const float v[4] = {x[p].x, p ? x[p].x : -x[p].x, x[p].y, x[p].y};
            uint32_t b[4];
            std::memcpy(b, v, 16);
            out.push_back(make_uint4(b[0], b[1], b[2], b[3]));
        }
    }
    void start(uint32_t tile_bit) {  // a layer that has no gate on tile_bit yet
        if (probes || (open && (used >> tile_bit & 1))) close();
        if (!open) open = true, active = real = flips = used = 0;
        used |= 1u << tile_bit;
    }
    void nop(uint32_t tile_bit, uint32_t pos) {  // absorbed: only its events are left
        if (open || probes) used |= 1u << tile_bit, end = pos + 1;
        else if (last != SIZE_MAX) out[last].y = pos + 1;
        else start(tile_bit), end = pos + 1;
    }
    void flip(uint32_t tile_bit, uint32_t pos) {
        start(tile_bit);
        flips |= 1u << tile_bit;
        end = pos + 1;
    }
    void giv(uint32_t tile_bit, uint32_t p, const FrameGate &g, uint32_t pos) {
        start(tile_bit);
        active |= 1u << p;
        if (g.x.y == 0.f) real |= 1u << p;
        if (g.flip) flips |= 1u << tile_bit;
        x[p] = g.x;
        end = pos + 1;
    }
    void cz(uint32_t q0, uint32_t q1, uint32_t p0, uint32_t p1, uint32_t pos) {
        if (p0 > p1) std::swap(p0, p1), std::swap(q0, q1);
        const uint32_t R = REG_BITS;
        const uint32_t pair = p0 == 0 ? p1 - 1 : p0 == 1 ? p1 + 2 : p0 == 2 ? p1 + 4 : 9;
        op(p1 < R ? OP_CZ_RR + pair : p0 < R ? OP_CZ_RT + p0 : (uint32_t)OP_CZ_TT, pos + 1, q0 | q1 << 8);
    }
    // conditional flip of c (register position pc) and signs: terms (internal.h) over a, b, c
    void flip_if(uint32_t a, uint32_t pa, uint32_t b, uint32_t pb, uint32_t cq, uint32_t pc, uint32_t terms,
                 uint32_t flips_, uint32_t pos_end) {
        close();
        last = out.size();
        out.push_back(make_uint4(((terms & 7u) ? OP_CX + std::min(pc, REG_BITS - 1u) : (uint32_t)OP_SIGN) | 2u << 24, pos_end,
                                 0, flips_));
        out.push_back(make_uint4(reg_bits(pa), reg_bits(pb),
                                 (31 - a) | (31 - b) << 8 | (31 - cq) << 16 | pc << 24, terms));
    }
    static uint32_t reg_bits(uint32_t p) {
        static const uint32_t pat[5] = {0xAAAAAAAAu, 0xCCCCCCCCu, 0xF0F0F0F0u, 0xFF00FF00u, 0xFFFF0000u};
        return p < 5 ? pat[p] : 0u;
    }
    void measure(Frame &F, uint32_t tile_bit, uint32_t p, uint32_t loc, uint32_t pos) {
        if (open || (probes && (used >> tile_bit & 1))) close();
        if (!probes) used = 0;
        used |= 1u << tile_bit;
        probes |= 1u << p;
        probe[p] = {loc, F.phi(tile_bit), std::norm(F.S())};
        end = pos + 1;
    }
    // any other op, after the open layer; `before`: it may precede the open layer
    void op(uint32_t code, uint32_t pos_end, uint32_t z, const uint32_t *c = nullptr, bool before = false) {
        if (!before) close();
        last = out.size();
        out.push_back(make_uint4(code | (c ? 2u : 1u) << 24, pos_end, z, 0));
        if (c) out.push_back(make_uint4(c[0], c[1], 0, 0));
    }
    // the frame phase of q applied to the state, before the gate at `pos`
    void flush(Frame &F, uint32_t q, uint32_t p, uint32_t pos) {
        const int k = snap(F.phi(q));
        if (k == 0) return;
        const bool before = open && !(used >> q & 1);
        if (!before) close();
        if (k > 0) {
            op(OP_OMEGA | (uint32_t)k << 20, before ? 0 : pos, q | p << 16, nullptr, true);
        } else {
            // diag(1, phi) = h diag(conj h, h), h^2 = phi: the rounded h scales both halves alike, and
            // the host takes that scale out (a rounded phi would scale one half of the state)
            const cd h = std::sqrt(F.phi(q));
            const float2 hf = f2(h);
            uint32_t c[2];
            std::memcpy(c, &hf, 8);
            op(OP_PHASE, before ? 0 : pos, q | p << 16, c, true);
            F.S() *= h / std::abs(cd(hf.x, hf.y));
        }
        F.phi(q) = 1;
    }
};

// Records of a circuit with tensor phases: each gate's own matrix.
static void tensor_records(arso_circuit *c) {
    c->rops.resize(c->perm.size());
    for (const Pass &ps : c->passes) {
        std::vector<int> local(c->n, -1);
        for (size_t i = 0; i < ps.tile_qubits.size(); ++i) local[ps.tile_qubits[i]] = (int)i;
        for (uint32_t pos = ps.gb; pos < ps.ge; ++pos) {
            const HostGate &h = c->gates[c->perm[pos]];
            const uint32_t p0 = c->rpos[pos] & 15u, p1 = c->rpos[pos] >> 4;
            RegOp &o = c->rops[pos];
            o = RegOp{};
            uint8_t cls = h.cls;
            o.aux = cls == GC_OMEGA ? h.omega_k : (uint32_t)c->rmats.size();
            if (cls == GC_DENSE1) {
                // a dense gate whose complex64 entries have the special unitary form
                // [[a, b], [-conj b, conj a]] exactly runs on a and b alone
                for (int i = 0; i < 4; ++i) c->rmats.push_back(f2(h.m[i]));
                const float2 *m = c->rmats.data() + o.aux;
                if (m[2].x == -m[1].x && m[2].y == m[1].y && m[3].x == m[0].x && m[3].y == -m[0].y) {
                    cls = GC_SU2;
                    o.c0 = m[0];
                    o.c1 = m[1];
                }
            } else if (cls == GC_DENSE2) {
                for (int i = 0; i < 16; ++i) c->rmats.push_back(f2(h.m[i]));
            } else if (cls == GC_DIAG1) {
                o.c0 = f2(h.m[0]);
                o.c1 = f2(h.m[3]);
            } else if (cls == GC_DIAG2) {
                o.c0 = f2(h.m[15]);
            }
            o.pad[0] = reg_opcode(cls, p0, p1);
            o.pad[1] = (uint32_t)c->role[pos];
            o.w0 = (uint32_t)cls | p0 << 8 | p1 << 12 | (uint32_t)local[h.q0] << 16 | (uint32_t)local[h.q1] << 24;
        }
    }
}

// A fused run at positions [pos, end): the block header, its fused macro-op, and the gates
// one by one (written by `gate`) with the ops that bring them to the fused op's frame.
template <class Gate>
static void emit_run(arso_circuit *c, ProgWriter &W, Frame &F, const std::vector<int> &local, uint32_t pos, uint32_t end,
                     Gate &&gate) {
    std::vector<const HostGate *> gs;
    for (uint32_t p = pos; p < end; ++p) gs.push_back(&c->gates[c->perm[p]]);
    FusedRun r;
    ARSO_REQUIRE(product_of(gs, r), "internal: a fused run that is none");
    uint32_t q[3] = {0, 0, 0}, p[3] = {15, 15, 15};  // tile bits and register positions
    for (int k = 0; k < r.n; ++k) q[k] = (uint32_t)local[r.q[k]];
    for (uint32_t i = pos; i < end; ++i) {
        const HostGate &h = c->gates[c->perm[i]];
        for (int k = 0; k < r.n; ++k) {
            if (r.q[k] == h.q0) p[k] = c->rpos[i] & 15u;
            if (r.q[k] == h.q1) p[k] = c->rpos[i] >> 4;
        }
    }
    // the flipped qubit's frame phase cannot stay, unless it is a sign
    if (r.c >= 0 && snap(F.phi(q[r.c])) != 4) W.flush(F, q[r.c], p[r.c], pos);
    cd phi[3], out[3], S;
    for (int k = 0; k < r.n; ++k) phi[k] = F.phi(q[k]);
    uint32_t signs = 0;
    double theta = 0.0;
    ARSO_REQUIRE(run_phases(r, phi, S, out, signs, theta, 10 * RUN_TOL), "internal: a fused run's phases");
    // terms of the flip over (a, b), the other two qubits, and of the signs over (a, b, c)
    const int ci = r.c >= 0 ? r.c : r.n - 1;
    int ab[2] = {ci, ci}, m = 0;
    for (int k = 0; k < r.n; ++k)
        if (k != ci) ab[m++] = k;
    auto at = [&](uint32_t bits, int a, int b, int cc) {  // value of a truth table at chosen qubits
        uint32_t x = 0;
        if (a) x |= 1u << ab[0];
        if (b && m > 1) x |= 1u << ab[1];
        if (cc) x |= 1u << ci;
        return bits >> x & 1u;
    };
    uint32_t terms = 0, flip0 = 0;
    if (r.c >= 0) {
        const uint32_t f0 = at(r.f, 0, 0, 0), fa = at(r.f, 1, 0, 0), fb = m > 1 ? at(r.f, 0, 1, 0) : f0,
                       fab = m > 1 ? at(r.f, 1, 1, 0) : fa;
        flip0 = f0;
        terms |= (f0 ^ fa) | (f0 ^ fb) << 1 | (f0 ^ fa ^ fb ^ fab) << 2;
    }
    {   // signs: no constant or linear terms (those are the frame)
        const uint32_t a = m > 0, b = m > 1;
        const uint32_t sab = a && b ? at(signs, 1, 1, 0) : 0, sac = a ? at(signs, 1, 0, 1) : 0,
                       sbc = b ? at(signs, 0, 1, 1) : 0, sabc = a && b ? at(signs, 1, 1, 1) : 0;
        terms |= sab << 3 | sac << 4 | sbc << 5 | (a && b ? (sab ^ sac ^ sbc ^ sabc) << 6 : 0u);
    }
    cd scale(1, 0);
    float2 h{};
    if (theta != 0.0) {  // the parity phase e^{-i theta (a ^ b) / 2} = g diag(conj g, g), g = e^{-i theta / 4}
        const cd g = std::polar(1.0, -theta / 4);
        h = f2(g);
        scale = g / std::abs(cd(h.x, h.y));
    }
    W.close();
    const size_t head = W.out.size();
    W.out.push_back(make_uint4(OP_BLOCK | 1u << 24, end, 0, 0));
    if (theta != 0.0) {
        uint32_t cst[2];
        std::memcpy(cst, &h, 8);
        W.op(OP_PARITY, 0, q[0] | q[1] << 8 | p[0] << 16 | p[1] << 20, cst);
    } else {
        W.flip_if(q[ab[0]], p[ab[0]], q[ab[1]], p[ab[1]], q[ci], p[ci], terms, flip0 << q[ci], 0);
    }
    const size_t slow = W.out.size();
    W.last = SIZE_MAX;  // a gate that leaves nothing to do must not end in the fused macro-op
    Frame fused = F;
    fused.S() *= S * scale;
    for (int k = 0; k < r.n; ++k) {
        fused.phi(q[k]) = out[k];
        snap(fused.phi(q[k]));
    }
    for (uint32_t i = pos; i < end; ++i) gate(i);
    W.close();
    // the gates' frame into the fused one: the ratio of the two, phase by phase and as a scalar
    for (int k = 0; k < r.n; ++k) {
        const cd want = fused.phi(q[k]);
        F.phi(q[k]) /= want;
        W.flush(F, q[k], p[k], end);
    }
    const cd ratio = F.S() / fused.S();
    if (std::abs(ratio - 1.0) > 1e-14) {
        const float2 f = f2(ratio);
        const float d = real_gap(ratio, f);
        uint32_t cst[2];
        std::memcpy(cst, &f, 8);
        W.op(OP_SCALE, end, 0, cst);
        std::memcpy(&W.out.back().z, &d, 4);
    }
    W.out[head].z = (uint32_t)(W.out.size() - slow);
    W.last = SIZE_MAX;  // nor a later one in a macro-op that the fused path passes over
    F = fused;
}

// The register program of every phase (internal.h), its event table and frames: the
// frames start from the identity in every pass (streaming) or once (resident, recorded at
// every phase boundary). The scalar alone goes on from pass to pass: what the rounding of a
// pass's table takes from it is in the next pass's, so that a state is off by one rounding of
// it, not by one a pass (the same for all amplitudes, those would add up: norm of a 14-qubit
// Clifford+T circuit of 600 gates on five passes, 2.6e-7 short, 1.7e-8 so).
static void reg_program(arso_circuit *c) {
    c->frames = c->reg_blocked && !c->tensor;
    c->rops.clear();
    c->prog.clear();
    c->ph_pg.clear();
    c->rmats.clear();
    c->evs.clear();
    c->frame.clear();
    if (!c->reg_blocked) return;
    if (!c->frames) return tensor_records(c);
    c->probe_slots.clear();
    c->probe_first.clear();
    c->evs.resize(2 * c->perm.size());
    size_t blk = 0;  // next fused run (they are in engine order)
    cd carry = 1.0;  // what the last pass's table, rounded to FP32, left of its scalar
    std::vector<float2> table;
    for (Pass &ps : c->passes) {
        std::vector<int> local(c->n, -1);
        for (size_t i = 0; i < ps.tile_qubits.size(); ++i) local[ps.tile_qubits[i]] = (int)i;
        Frame F(c->tile_qubits);
        F.S() = carry;
        ps.full = 0;
        for (uint32_t ph = ps.pb; ph < ps.pe; ++ph) {
            if (c->engine == 0) c->frame.push_back(F.f);
            c->ph_pg.push_back((uint32_t)c->prog.size());
            c->probe_first.push_back((uint32_t)c->probe_slots.size());
            ProgWriter W(c->prog);
            W.slots = &c->probe_slots;
            auto gate = [&](uint32_t pos) {
                const HostGate &h = c->gates[c->perm[pos]];
                const uint32_t q0 = (uint32_t)local[h.q0], q1 = (uint32_t)local[h.q1];
                const uint32_t p0 = c->rpos[pos] & 15u, p1 = c->rpos[pos] >> 4;
                const uint32_t z = q0 | q1 << 8 | p0 << 16 | p1 << 20, code = reg_opcode(h.cls, p0, p1);
                switch (h.cls) {
                    case GC_H: {
                        // an odd power of omega would make x a rounded constant: the same rounding
                        // in every such gate of a Clifford+T circuit, so it is applied (compensated) first
                        const int k = snap(F.phi(q0));
                        if (k > 0 && (k & 1)) W.flush(F, q0, p0, pos);
                    }  // fall through
                    case GC_DENSE1: {
                        const FrameGate g = frame_dense(F, q0, h.m);
                        if (g.kind == FrameGate::NOP) {
                            W.nop(q0, pos);
                        } else if (g.kind == FrameGate::FLIP) {
                            W.flip(q0, pos);
                        } else if (g.kind == FrameGate::GIV) {
                            W.giv(q0, p0, g, pos);
                        } else {
                            const uint32_t aux[2] = {(uint32_t)c->rmats.size(), 0};
                            for (const cd &v : g.m) c->rmats.push_back(f2(v));
                            W.op(reg_opcode(GC_DENSE1, p0, p1), pos + 1, z, aux);
                            ++ps.full;
                        }
                        break;
                    }
                    case GC_DIAG1:
                    case GC_OMEGA:
                        F.S() *= h.m[0];
                        F.phi(q0) *= h.m[3] / h.m[0];
                        snap(F.phi(q0));
                        W.nop(q0, pos);
                        break;
                    case GC_X:  // X diag(1, phi) X = phi diag(1, conj phi)
                        F.S() *= F.phi(q0);
                        F.phi(q0) = std::conj(F.phi(q0));
                        W.flip(q0, pos);
                        break;
                    case GC_CX:
                        if (snap(F.phi(q1)) == 4) F.phi(q0) = -F.phi(q0);  // CX Z_t = Z_c Z_t CX
                        else W.flush(F, q1, p1, pos);
                        W.flip_if(q0, p0, q0, p0, q1, p1, 1u, 0, pos + 1);
                        break;
                    case GC_SWAP:
                        std::swap(F.phi(q0), F.phi(q1));
                        W.op(code, pos + 1, z);
                        break;
                    case GC_DENSE2: {
                        const uint32_t aux[2] = {(uint32_t)c->rmats.size(), 0};
                        const cd col[4] = {1.0, F.phi(q0), F.phi(q1), F.phi(q0) * F.phi(q1)};
                        for (int i = 0; i < 16; ++i) c->rmats.push_back(f2(h.m[i] * col[i & 3]));
                        F.phi(q0) = F.phi(q1) = 1;
                        W.op(code, pos + 1, z, aux);
                        break;
                    }
                    case GC_DIAG2: {  // commutes with the frame
                        const float2 f = f2(h.m[15]);
                        uint32_t cst[2];
                        std::memcpy(cst, &f, 8);
                        W.op(code, pos + 1, z, cst);
                        break;
                    }
                    case GC_CZ: W.cz(q0, q1, p0, p1, pos); break;
                    case GC_PROBE: W.measure(F, q0, p0, c->probe_loc[c->perm[pos]], pos); break;
                    default: W.nop(q0, pos); break;
                }
                auto slot = [&](uint32_t q) {
                    const float2 f = f2(F.phi(q));
                    return EvSlot{f, q, real_gap(F.phi(q), f)};
                };
                c->evs[2 * pos] = slot(q0);
                c->evs[2 * pos + 1] = slot(q1);
            };
            for (uint32_t pos = c->ph_gb[ph]; pos < c->ph_gb[ph + 1];) {
                if (blk < c->blocks.size() && c->blocks[blk].first == pos) {
                    const uint32_t end = c->blocks[blk++].second;
                    emit_run(c, W, F, local, pos, end, gate);
                    pos = end;
                } else {
                    gate(pos++);
                }
            }
            if (ph + 1 == ps.pe)  // odd powers of omega do not go into a rounded table: they are applied, compensated
                for (uint32_t q = 0; q < c->tile_qubits; ++q)
                    if (const int k = snap(F.phi(q)); k > 0 && (k & 1)) {
                        uint32_t p = 15;
                        for (int b = 0; b < REG_BITS; ++b)
                            if ((c->ph_R[ph] >> (5 * b) & 31u) == q) p = (uint32_t)b;
                        W.flush(F, q, p, c->ph_gb[ph + 1]);
                    }
            W.close();
            ARSO_REQUIRE(c->prog.size() - c->ph_pg.back() <= (size_t)MAX_PHASE_UNITS, "internal: a phase's program is too long");
        }
        c->frame.push_back(F.f);  // streaming: the pass's end; resident: the circuit's
        if (c->engine == 1) {
            table.resize(frame_floats2((int)c->tile_qubits));
            carry = 1.0 / frame_table(F.f, (int)c->tile_qubits, table.data());
        }
    }
    c->ph_pg.push_back((uint32_t)c->prog.size());
    c->probe_first.push_back((uint32_t)c->probe_slots.size());
}

// The circuit that the single-error analysis of a streaming complex64 circuit runs: its
// gates with a measurement of each error location's qubit right after the location's gate.
// dual: the adjoint gates in reverse order, each after the measurements of its locations,
// on one more qubit, 0, that no gate touches: it tells psi (0) from phi (1), so their
// amplitudes are neighbours and the two lanes of every packed register.
std::unique_ptr<arso_circuit> build_probe(const arso_circuit *c, bool dual) {
    std::unique_ptr<arso_circuit> P(new arso_circuit());
    const size_t G = c->gates.size();
    std::vector<uint32_t> first(G + 1, 0);  // first location of each gate
    for (size_t g = 0; g < G; ++g) first[g + 1] = first[g] + (uint32_t)c->gates[g].arity;
    P->n = c->n + (dual ? 1 : 0);
    P->engine = 1;
    // the forward circuit's own passes where they are register-blocked
    const bool own = !dual && c->reg_blocked && !c->tensor;
    P->tile_qubits = own ? c->tile_qubits : std::min(13u, P->n);
    P->low_qubits = own ? c->low_qubits : 4u;
    std::vector<uint32_t> order;  // gate of each position of the passes
    if (own) {
        P->passes = c->passes;
        order = c->perm;
    } else {
        arso_circuit T;
        T.n = P->n;
        T.tile_qubits = P->tile_qubits;
        T.low_qubits = P->low_qubits;
        T.gates.resize(G);
        for (size_t k = 0; k < G; ++k) {
            T.gates[k] = c->gates[dual ? G - 1 - k : k];
            T.gates[k].q0 += dual;
            T.gates[k].q1 += dual;
        }
        schedule_streaming(&T);
        P->passes = T.passes;
        for (uint32_t k : T.perm) order.push_back(dual ? (uint32_t)(G - 1 - k) : k);
    }
    for (Pass &ps : P->passes) {
        const uint32_t gb = (uint32_t)P->gates.size();
        for (uint32_t pos = ps.gb; pos < ps.ge; ++pos) {
            HostGate h = c->gates[order[pos]];
            h.q0 += dual;
            h.q1 += dual;
            if (dual) {  // adjoint
                const int dim = h.arity == 1 ? 2 : 4;
                HostGate a = h;
                for (int r = 0; r < dim; ++r)
                    for (int k = 0; k < dim; ++k) a.m[r * dim + k] = std::conj(h.m[k * dim + r]);
                a.omega_k = (8u - h.omega_k) & 7u;
                h = a;
            } else {
                P->gates.push_back(h);
                P->probe_loc.push_back(0);
            }
            for (int j = 0; j < h.arity; ++j) {
                HostGate m{};
                m.arity = 1;
                m.cls = GC_PROBE;
                m.q0 = m.q1 = j ? h.q1 : h.q0;
                P->gates.push_back(m);
                P->probe_loc.push_back(first[order[pos]] + j);
            }
            if (dual) {
                P->gates.push_back(h);
                P->probe_loc.push_back(0);
            }
        }
        ps.gb = gb;
        ps.ge = (uint32_t)P->gates.size();
    }
    P->perm.resize(P->gates.size());
    for (size_t i = 0; i < P->perm.size(); ++i) P->perm[i] = (uint32_t)i;
    plan_phases(P.get());
    reg_program(P.get());
    P->pos_of.assign(P->gates.size(), 0);
    for (size_t pos = 0; pos < P->perm.size(); ++pos) P->pos_of[P->perm[pos]] = (uint32_t)pos;
    return P;
}

// The kernels' table of frame f (internal.h), in the load/store mapping {0, t-4, ..., t-1}.
// Returns the mean of its factors over the exact ones: what the rounding of the table does to
// the state as a whole.
cd frame_table(const std::vector<cd> &f, int t, float2 *out) {
    const int nt = 1 << (t - REG_BITS);
    // the products of the phases of the bits set in i, S in the first
    auto products = [&](cd *v, cd first, int bits, auto phi) {
        v[0] = first;
        for (int b = 0; b < bits; ++b)
            for (int i = 0; i < 1 << b; ++i) v[(1 << b) + i] = v[i] * phi(b);
    };
    auto rounded = [](cd v, float2 &o) {
        o = f2(v);
        return cd(o.x, o.y) * std::conj(v) / std::norm(v);
    };
    cd thread[1 << (MAX_TILE_QUBITS - REG_BITS)], reg[32], rt = 0.0, rr = 0.0;
    float2 r[32];
    products(thread, f[0], t - REG_BITS, [&](int b) { return f[2 + b]; });
    products(reg, 1.0, REG_BITS, [&](int b) { return b ? f[t - 4 + b] : f[1]; });
    for (int i = 0; i < nt; ++i) rt += rounded(thread[i], out[i]);
    for (int k = 0; k < 32; ++k) rr += rounded(reg[k], r[k]);
    for (int k = 0; k < 16; ++k) {
        out[nt + 2 * k] = make_float2(r[2 * k].x, r[2 * k + 1].x);
        out[nt + 2 * k + 1] = make_float2(r[2 * k].y, r[2 * k + 1].y);
    }
    return rt / (double)nt * (rr / 32.0);
}

void build_circuit(arso_circuit *c, uint32_t n, const arso_gate *gates, size_t n_gates,
                   const arso_compile_opts *opts) {
    ARSO_REQUIRE(n >= 1 && n <= 30, "n_qubits must be in [1, 30]");
    ARSO_REQUIRE(n_gates == 0 || gates != nullptr, "gates is NULL");
    ARSO_REQUIRE(n_gates < (1u << 28), "too many gates");
    c->n = n;
    c->precision = opts ? (int)opts->precision : ARSO_C64;
    ARSO_REQUIRE(c->precision == ARSO_C64 || c->precision == ARSO_C128, "bad precision");
    c->gates.resize(n_gates);
    c->k = c->m = 0;
    for (size_t i = 0; i < n_gates; ++i) {
        const arso_gate &g = gates[i];
        HostGate &h = c->gates[i];
        h.kind = g.kind;
        h.arity = g.kind >= ARSO_GATE_CX ? 2 : 1;
        h.q0 = g.q[0];
        h.q1 = h.arity == 2 ? g.q[1] : g.q[0];
        ARSO_REQUIRE(h.q0 < n && h.q1 < n, "gate " + std::to_string(i) + ": qubit out of range");
        ARSO_REQUIRE(h.arity == 1 || h.q0 != h.q1, "gate " + std::to_string(i) + ": repeated qubit");
        matrix_for(g, h);
        if (h.arity == 1) ++c->k; else ++c->m;
    }
    c->L = c->k + 2 * c->m;
    ARSO_REQUIRE(c->L < (1ull << 29), "too many error locations");
    c->loc_gate.clear();
    c->loc_gate.reserve(c->L);
    for (size_t i = 0; i < n_gates; ++i)
        for (int j = 0; j < c->gates[i].arity; ++j) c->loc_gate.push_back((uint32_t)i);

    const int rmax = c->precision == ARSO_C128 ? RESIDENT_MAX_N_C128 : RESIDENT_MAX_N_C64;
    c->engine = (int)n <= rmax ? 0 : 1;
    uint32_t tq = opts && opts->tile_qubits ? opts->tile_qubits : (c->precision == ARSO_C128 ? 12u : 13u);
    uint32_t lq = opts && opts->low_qubits ? opts->low_qubits : 4u;
    c->max_batch = opts ? opts->max_batch : 0;
    c->flags = opts ? opts->flags : 0;
    c->cache_budget = opts && opts->cache_bytes ? opts->cache_bytes : (uint64_t)16 << 30;
    if (c->engine == 0) {
        c->tile_qubits = n;
        c->low_qubits = n;
        c->perm.resize(n_gates);
        for (size_t i = 0; i < n_gates; ++i) c->perm[i] = (uint32_t)i;
        Pass p;
        p.gb = 0;
        p.ge = (uint32_t)n_gates;
        for (uint32_t q = 0; q < n; ++q) p.tile_qubits.push_back(q);
        c->passes.assign(1, p);
    } else {
        const uint32_t tmax = c->precision == ARSO_C128 ? 13u : (uint32_t)MAX_TILE_QUBITS;
        ARSO_REQUIRE(tq >= 6 && tq <= tmax, "tile_qubits out of range");
        tq = std::min(tq, n);
        lq = std::min(std::max(lq, 1u), tq);
        c->tile_qubits = tq;
        c->low_qubits = lq;
        schedule_streaming(c);
    }
    plan_phases(c);  // may reorder gates within a pass
    reg_program(c);
    c->flops_prefix.assign(n_gates + 1, 0.0);
    for (size_t pos = 0; pos < n_gates; ++pos) c->flops_prefix[pos + 1] = c->flops_prefix[pos] + gate_flops(c->gates[c->perm[pos]]);
    c->pos_of.assign(n_gates, 0);
    for (size_t pos = 0; pos < c->perm.size(); ++pos) c->pos_of[c->perm[pos]] = (uint32_t)pos;
    c->pass_of_pos.assign(n_gates, 0);
    for (size_t p = 0; p < c->passes.size(); ++p)
        for (uint32_t pos = c->passes[p].gb; pos < c->passes[p].ge; ++pos) c->pass_of_pos[pos] = (uint32_t)p;
}

}  // namespace arso

namespace arso {

// 32 surrogate features: n, G, L, k, m, depth, two-qubit layers, log10 L,
// log10 G, two-qubit fraction, counts per gate kind (18), criterion one-hot (4).
std::vector<float> circuit_features(const arso_circuit *c, const arso_criterion *crit) {
    std::vector<float> f(ARSO_N_FEATURES, 0.f);
    const size_t G = c->gates.size();
    std::vector<uint32_t> level(c->n, 0);
    uint32_t depth = 0;
    std::vector<char> layer_has_2q;
    static const uint32_t kinds[18] = {ARSO_GATE_H, ARSO_GATE_X, ARSO_GATE_Y, ARSO_GATE_Z, ARSO_GATE_S,
                                       ARSO_GATE_SDG, ARSO_GATE_T, ARSO_GATE_TDG, ARSO_GATE_RX, ARSO_GATE_RY,
                                       ARSO_GATE_RZ, ARSO_GATE_P, ARSO_GATE_U, ARSO_GATE_CX, ARSO_GATE_CZ,
                                       ARSO_GATE_CP, ARSO_GATE_SWAP, ARSO_GATE_U2};
    float counts[18] = {0};
    for (const HostGate &h : c->gates) {
        uint32_t lv = level[h.q0];
        if (h.arity == 2) lv = std::max(lv, level[h.q1]);
        lv += 1;
        level[h.q0] = lv;
        if (h.arity == 2) level[h.q1] = lv;
        depth = std::max(depth, lv);
        if (layer_has_2q.size() < lv + 1) layer_has_2q.resize(lv + 1, 0);
        if (h.arity == 2) layer_has_2q[lv] = 1;
        for (int i = 0; i < 18; ++i)
            if (kinds[i] == h.kind) counts[i] += 1.f;
    }
    uint32_t layers2 = 0;
    for (char b : layer_has_2q) layers2 += b ? 1 : 0;
    f[0] = (float)c->n;
    f[1] = (float)G;
    f[2] = (float)c->L;
    f[3] = (float)c->k;
    f[4] = (float)c->m;
    f[5] = (float)depth;
    f[6] = (float)layers2;
    f[7] = (float)std::log10(std::max<double>(1.0, (double)c->L));
    f[8] = (float)std::log10(std::max<double>(1.0, (double)G));
    f[9] = G ? (float)c->m / (float)G : 0.f;
    for (int i = 0; i < 18; ++i) f[10 + i] = counts[i];
    if (crit && crit->kind <= ARSO_CRIT_ARGMAX) f[28 + crit->kind] = 1.f;
    return f;
}

}  // namespace arso
