// Runs the register programs of a circuit (internal.h) in FP64 with the constants they hold, on
// the CPU: what the kernels compute but for the rounding of their arithmetic. The frame tables
// are applied in FP32 products as the kernels form them.
//   program_emulator < "n tile seed events", then "kind q0 q1 param count m..." a gate
// prints "dense <full one-qubit matrices> norm <||psi|| - 1> error <||psi - psi_64||> phases <n>"
// of a trajectory with the given number of random error events.
#include "../paper_2301_07264_gb300/csrc/circuit.cpp"

#include <cstdio>
#include <random>

namespace arso {
void *pool_alloc(size_t, cudaStream_t) { return nullptr; }
void *pool_alloc_list(size_t, cudaStream_t, ContextPools *&) { return nullptr; }
void *pool_alloc_now(size_t, ContextPools *&) { return nullptr; }
void pool_free(void *, ContextPools *, bool) noexcept {}
void set_last_error(const std::string &) {}
}  // namespace arso
using namespace arso;

static cd c2(uint32_t a, uint32_t b) {
    float x, y;
    std::memcpy(&x, &a, 4), std::memcpy(&y, &b, 4);
    return cd(x, y);
}
static cd c2(float2 v) { return cd(v.x, v.y); }

struct Event { uint32_t pos, slot, code; };

struct Machine {
    const arso_circuit &c;
    uint32_t N, m = 0;                // m: index mask over global qubits
    cd phase = 1.0;                   // i^gp and the scale that the kernels apply with it
    std::vector<cd> s;
    std::vector<uint32_t> g;          // global qubit of each tile bit
    uint32_t dense = 0;
    explicit Machine(const arso_circuit &k) : c(k), N(1u << k.n), s(N, 0.0) { s[0] = 1.0; }
    uint32_t bit(uint32_t j, uint32_t q) const { return ((j ^ m) >> g[q]) & 1u; }
    void pair(uint32_t q, cd m00, cd m01, cd m10, cd m11) {
        for (uint32_t x = 0; x < N; ++x) {
            if (x >> g[q] & 1) continue;
            const uint32_t a = x ^ (m & 1u << g[q]), b = a ^ 1u << g[q];
            const cd u = s[a], v = s[b];
            s[a] = m00 * u + m01 * v, s[b] = m10 * u + m11 * v;
        }
    }
    void error(const Event &e) {
        const EvSlot &v = c.evs[2 * e.pos + e.slot];
        if (e.code & 2)
            for (uint32_t j = 0; j < N; ++j)
                if (bit(j, v.q)) s[j] = -s[j];
        if (e.code & 1) m ^= 1u << g[v.q];
        if (e.code == 3) phase *= cd(0, 1);
        if ((e.code & 1) && (v.phi.x != 1.f || v.phi.y != 0.f)) {
            const cd f = c2(v.phi) + (double)v.d;
            for (uint32_t j = 0; j < N; ++j) s[j] *= bit(j, v.q) ? std::conj(f) : f;
        }
    }
    void run(uint32_t ph, const std::vector<Event> &ev, size_t &next) {
        uint32_t R[5];
        for (int b = 0; b < 5; ++b) R[b] = c.ph_R[ph] >> (5 * b) & 31u;
        uint32_t skip = 0;
        for (size_t u = c.ph_pg[ph], ue = c.ph_pg[ph + 1]; u < ue;) {
            const uint4 h = c.prog[u];
            const uint32_t code = h.x & 255u;
            if (code == OP_BLOCK) {
                if (next < ev.size() && ev[next].pos < h.y) u += 1 + (c.prog[u + 1].x >> 24);
                else ++u, skip = h.z;
                continue;
            }
            const uint4 k = u + 1 < c.prog.size() ? c.prog[u + 1] : uint4{};
            const uint32_t q0 = h.z & 255u, q1 = h.z >> 8 & 255u;
            auto flip = [&](uint32_t w) {
                for (uint32_t q = 0; q < g.size(); ++q)
                    if (w >> q & 1) m ^= 1u << g[q];
            };
            if (code == OP_LAYER) {
                flip(h.w);
                size_t v = u + 1;
                for (int p = 0; p < 5; ++p)
                    if (h.x >> (8 + p) & 1) {
                        const cd x = c2(c.prog[v].x, c.prog[v].z);
                        pair(R[p], 1.0, x, -std::conj(x), 1.0);
                        ++v;
                    }
            } else if ((code >= OP_CX && code < OP_CX + 5) || code == OP_SIGN) {
                const uint32_t a = 31 - (k.z & 31), b = 31 - (k.z >> 8 & 31), t = 31 - (k.z >> 16 & 31);
                if (code != OP_SIGN)
                    for (uint32_t j = 0; j < N; ++j) {
                        const uint32_t A = bit(j, a), B = bit(j, b);
                        if (!(j >> g[t] & 1) && ((k.w & A) ^ (k.w >> 1 & B) ^ (k.w >> 2 & A & B)) & 1) std::swap(s[j], s[j | 1u << g[t]]);
                    }
                flip(h.w);
                for (uint32_t j = 0; j < N; ++j) {
                    const uint32_t A = bit(j, a), B = bit(j, b), T = bit(j, t);
                    if (((k.w >> 3 & A & B) ^ (k.w >> 4 & A & T) ^ (k.w >> 5 & B & T) ^ (k.w >> 6 & A & B & T)) & 1) s[j] = -s[j];
                }
            } else if ((code >= OP_CZ_RR && code < OP_CZ_RR + 10) || (code >= OP_CZ_RT && code < OP_CZ_RT + 5) || code == OP_CZ_TT) {
                for (uint32_t j = 0; j < N; ++j)
                    if (bit(j, q0) && bit(j, q1)) s[j] = -s[j];
            } else if (code == OP_OMEGA) {
                for (uint32_t j = 0; j < N; ++j)
                    if (bit(j, q0)) s[j] *= omega(h.x >> 20 & 7);
            } else if (code == OP_PHASE || code == OP_PARITY) {
                const cd f = c2(k.x, k.y);
                for (uint32_t j = 0; j < N; ++j) s[j] *= (code == OP_PHASE ? bit(j, q0) : bit(j, q0) ^ bit(j, q1)) ? f : std::conj(f);
            } else if (code == OP_CP) {
                for (uint32_t j = 0; j < N; ++j)
                    if (bit(j, q0) && bit(j, q1)) s[j] *= c2(k.x, k.y);
            } else if (code == OP_SCALE) {
                for (cd &x : s) x *= c2(k.x, k.y) + c2(k.z, 0).real();
            } else if (code >= OP_DENSE1 && code < OP_DENSE1 + 5) {
                const float2 *M = c.rmats.data() + k.x;
                pair(R[code - OP_DENSE1], c2(M[0]), c2(M[1]), c2(M[2]), c2(M[3]));
                ++dense;
            } else if (code == OP_DENSE2) {
                const float2 *M = c.rmats.data() + k.x;
                for (uint32_t x = 0; x < N; ++x) {
                    if ((x >> g[q0] & 1) || (x >> g[q1] & 1)) continue;
                    uint32_t ix[4];
                    cd v[4];
                    for (uint32_t i = 0; i < 4; ++i) ix[i] = (x | (i & 1) << g[q0] | (i >> 1) << g[q1]) ^ m, v[i] = s[ix[i]];
                    for (int i = 0; i < 4; ++i) {
                        s[ix[i]] = 0;
                        for (int l = 0; l < 4; ++l) s[ix[i]] += c2(M[4 * i + l]) * v[l];
                    }
                }
            } else if (code == OP_SWAP) {
                std::vector<cd> o(s);
                for (uint32_t j = 0; j < N; ++j) {
                    const uint32_t x = j ^ m, a = x >> g[q0] & 1, b = x >> g[q1] & 1;
                    s[((x & ~(1u << g[q0] | 1u << g[q1])) | b << g[q0] | a << g[q1]) ^ m] = o[j];
                }
            } else {
                std::printf("unknown op %u\n", code);
                std::exit(1);
            }
            u += (h.x >> 24) + skip;
            skip = 0;
            while (next < ev.size() && ev[next].pos < h.y) error(ev[next++]);
        }
    }
    // the frame's table and what is left of the masks and the phase
    void end(const std::vector<cd> &f) {
        const int t = (int)c.tile_qubits, nt = 1 << (t - REG_BITS);
        std::vector<float2> tab(frame_floats2(t));
        frame_table(f, t, tab.data());
        std::vector<cd> o(N);
        for (uint32_t j = 0; j < N; ++j) {
            uint32_t x = 0;
            for (int q = 0; q < t; ++q) x |= bit(j, q) << q;
            const float2 F = tab[(x >> 1) & (nt - 1)];
            const float *r = reinterpret_cast<const float *>(tab.data() + nt) + 4 * (x >> (t - 4)) + (x & 1);
            const float gr = std::fma(-F.y, r[2], F.x * r[0]), gi = std::fma(F.y, r[0], F.x * r[2]);
            o[j ^ m] = s[j] * cd(gr, gi) * phase;
        }
        s = o;
        m = 0;
        phase = 1.0;
    }
};

int main() {
    unsigned n, tile, seed, events, kind, q0, q1;
    if (std::scanf("%u %u %u %u", &n, &tile, &seed, &events) != 4) return 1;
    std::vector<arso_gate> gates;
    std::vector<std::vector<double>> mats;
    double param;
    int cnt;
    while (std::scanf("%u %u %u %lf %d", &kind, &q0, &q1, &param, &cnt) == 5) {
        arso_gate x{};
        x.kind = kind, x.q[0] = q0, x.q[1] = q1, x.param = param;
        mats.emplace_back(cnt);
        for (double &v : mats.back())
            if (std::scanf("%lf", &v) != 1) return 1;
        gates.push_back(x);
    }
    for (size_t i = 0; i < gates.size(); ++i) gates[i].matrix = mats[i].empty() ? nullptr : mats[i].data();
    arso_compile_opts o{};
    o.tile_qubits = tile;
    arso_circuit c;
    build_circuit(&c, n, gates.data(), gates.size(), &o);
    if (!c.frames) return 1;
    // events in engine order, the same in the order of the gates for the FP64 run
    std::mt19937 rng(seed);
    std::set<std::pair<uint32_t, uint32_t>> at;
    while (at.size() < events) {
        const uint32_t pos = rng() % gates.size();
        at.insert({pos, rng() % (uint32_t)c.gates[c.perm[pos]].arity});
    }
    std::vector<Event> ev;
    for (auto &p : at) ev.push_back({p.first, p.second, 1 + rng() % 3});

    Machine M(c);
    size_t next = 0;
    for (size_t p = 0; p < c.passes.size(); ++p) {
        M.g = c.passes[p].tile_qubits;
        for (uint32_t ph = c.passes[p].pb; ph < c.passes[p].pe; ++ph) M.run(ph, ev, next);
        M.end(c.engine == 1 ? c.frame[p] : c.frame.back());
    }
    std::vector<cd> w(M.N, 0.0);
    w[0] = 1.0;
    next = 0;
    for (uint32_t pos = 0; pos < c.perm.size(); ++pos) {
        const HostGate &h = c.gates[c.perm[pos]];
        const uint32_t b0 = 1u << h.q0, b1 = 1u << h.q1;
        for (uint32_t x = 0; x < M.N; ++x) {
            if ((x & b0) || (h.arity == 2 && (x & b1))) continue;
            const int d = h.arity == 1 ? 2 : 4;
            uint32_t ix[4] = {x, x | b0, x | b1, x | b0 | b1};
            cd v[4];
            for (int i = 0; i < d; ++i) v[i] = w[ix[i]];
            for (int i = 0; i < d; ++i) {
                w[ix[i]] = 0;
                for (int l = 0; l < d; ++l) w[ix[i]] += h.m[d * i + l] * v[l];
            }
        }
        for (; next < ev.size() && ev[next].pos == pos; ++next) {
            const uint32_t b = ev[next].slot ? b1 : b0, code = ev[next].code;
            for (uint32_t x = 0; x < M.N; ++x) {
                if (x & b) continue;
                cd &a0 = w[x], &a1 = w[x | b];
                const cd u = a0, v = a1;
                if (code == 1) a0 = v, a1 = u;
                if (code == 2) a1 = -v;
                if (code == 3) a0 = cd(0, -1) * v, a1 = cd(0, 1) * u;  // Eq. (2)
            }
        }
    }
    double n1 = 0, n2 = 0, d = 0;
    for (uint32_t j = 0; j < M.N; ++j) n1 += std::norm(M.s[j]), n2 += std::norm(w[j]), d += std::norm(M.s[j] - w[j]);
    std::printf("dense %u norm %.3e error %.3e phases %zu\n", M.dense, std::sqrt(n1) - std::sqrt(n2), std::sqrt(d), c.ph_R.size());
    return 0;
}
