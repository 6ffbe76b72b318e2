// qs_jit.cu -- tile passes generated for their exact shape and compiled at run time (NVRTC).
//
// What a generated kernel computes is what k_tile_pass computes for the same TilePass, groups
// and gates (the same tile map, swizzle, register groups, folded exchanges, predicates and
// pair updates, Section III Eq. 2 per selected pair); only the per-gate interpretation is
// gone. See qs_jit.cuh.
#include <nvrtc.h>
#include <sys/stat.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "k_tile.cuh"
#include "qs_jit.cuh"

namespace qs {

int device_sm_count();
void *debug_state_address();

#ifdef QS_DEBUG_CHECKS
constexpr bool kDebugBuild = true;
#else
constexpr bool kDebugBuild = false;
#endif

namespace {

struct Out {
    std::string s;
    void f(const char *fmt, ...) {
        char buf[1024];
        va_list ap;
        va_start(ap, fmt);
        const int m = std::vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        if (m < (int)sizeof(buf)) {
            s += buf;
        } else {
            std::vector<char> big((size_t)m + 1);
            va_start(ap, fmt);
            std::vsnprintf(big.data(), big.size(), fmt, ap);
            va_end(ap);
            s += big.data();
        }
    }
};

// Local tile offset o -> global amplitude offset (the pass's runs of consecutive local bits).
uint64_t scatter_host(const TilePass &P, uint32_t o) {
    uint64_t g = 0;
    for (int r = 0; r < P.nruns; ++r)
        g |= (uint64_t)((o >> P.run_src[r]) & ((1u << P.run_len[r]) - 1u)) << P.run_dst[r];
    return g;
}

// Types, copies and pair updates shared by every generated kernel (one precision).
void preamble(Out &o, bool dbl) {
    o.f("typedef unsigned int u32;\ntypedef unsigned long long u64;\n");
    if (dbl) {
        o.f("typedef double R;\nstruct alignas(16) T2 { double x, y; };\n");
        o.f("__device__ __forceinline__ R F(R a, R b, R c) { return __fma_rn(a, b, c); }\n");
    } else {
        o.f("typedef float R;\nstruct alignas(8) T2 { float x, y; };\nstruct alignas(16) T4 { float x, y, z, w; };\n");
        o.f("__device__ __forceinline__ R F(R a, R b, R c) { return __fmaf_rn(a, b, c); }\n");
    }
    // the same operation order as the interpreted pass (k_gate.cuh cmac / cmul / pair_update)
    if (dbl) {
        o.f("__device__ __forceinline__ void u_gen(T2 &x, T2 &y, const R *m) {\n"
            "  T2 a, b;\n"
            "  a.x = F(m[0], x.x, F(-m[1], x.y, F(m[2], y.x, -m[3] * y.y)));\n"
            "  a.y = F(m[0], x.y, F(m[1], x.x, F(m[2], y.y, m[3] * y.x)));\n"
            "  b.x = F(m[4], x.x, F(-m[5], x.y, F(m[6], y.x, -m[7] * y.y)));\n"
            "  b.y = F(m[4], x.y, F(m[5], x.x, F(m[6], y.y, m[7] * y.x)));\n"
            "  x = a; y = b;\n}\n");
        o.f("__device__ __forceinline__ void u_real(T2 &x, T2 &y, const R *m) {\n"
            "  T2 a, b;\n"
            "  a.x = F(m[0], x.x, m[2] * y.x); a.y = F(m[0], x.y, m[2] * y.y);\n"
            "  b.x = F(m[4], x.x, m[6] * y.x); b.y = F(m[4], x.y, m[6] * y.y);\n"
            "  x = a; y = b;\n}\n");
    } else {
        // float32: the real-matrix update takes the real and imaginary parts of a pair through
        // one packed two-lane instruction (fma.rn.f32x2 / mul.rn.f32x2, each lane rounded like
        // the scalar operation): the same results, half the instructions. (The general update
        // stays scalar: packed, it saves a quarter of its instructions but makes the register
        // allocation of long passes take minutes to compile.)
        o.f("__device__ __forceinline__ u64 pk(float a, float b) { u64 r; asm(\"mov.b64 %%0, {%%1, %%2};\" : \"=l\"(r) : "
            "\"f\"(a), \"f\"(b)); return r; }\n");
        o.f("__device__ __forceinline__ T2 upk(u64 r) { T2 a; asm(\"mov.b64 {%%0, %%1}, %%2;\" : \"=f\"(a.x), \"=f\"(a.y) : "
            "\"l\"(r)); return a; }\n");
        o.f("__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) { u64 d; asm(\"fma.rn.f32x2 %%0, %%1, %%2, %%3;\" : "
            "\"=l\"(d) : \"l\"(a), \"l\"(b), \"l\"(c)); return d; }\n");
        o.f("__device__ __forceinline__ u64 mul2(u64 a, u64 b) { u64 d; asm(\"mul.rn.f32x2 %%0, %%1, %%2;\" : \"=l\"(d) : "
            "\"l\"(a), \"l\"(b)); return d; }\n");
        o.f("__device__ __forceinline__ void u_gen(T2 &x, T2 &y, const R *m) {\n"
            "  T2 a, b;\n"
            "  a.x = F(m[0], x.x, F(-m[1], x.y, F(m[2], y.x, -m[3] * y.y)));\n"
            "  a.y = F(m[0], x.y, F(m[1], x.x, F(m[2], y.y, m[3] * y.x)));\n"
            "  b.x = F(m[4], x.x, F(-m[5], x.y, F(m[6], y.x, -m[7] * y.y)));\n"
            "  b.y = F(m[4], x.y, F(m[5], x.x, F(m[6], y.y, m[7] * y.x)));\n"
            "  x = a; y = b;\n}\n");
        o.f("__device__ __forceinline__ void u_real(T2 &x, T2 &y, const R *m) {\n"
            "  const u64 *q = (const u64 *)m; const u64 X = pk(x.x, x.y), Y = pk(y.x, y.y);\n"
            "  const u64 a = fma2(q[0], X, mul2(q[1], Y));\n"
            "  const u64 b = fma2(q[2], X, mul2(q[3], Y));\n"
            "  x = upk(a); y = upk(b);\n}\n");
    }
    // rotations [a -b; b a] and reflections [a b; b -a] with the larger entry divided out (its
    // product over the pass is applied by a later gate, real_forms): q = b / a or a / b
    if (dbl) {
        o.f("__device__ __forceinline__ void u_rot_a(T2 &x, T2 &y, const R *m) { const R q = m[0]; T2 a; a.x = F(-q, y.x, x.x); "
            "a.y = F(-q, y.y, x.y); y.x = F(q, x.x, y.x); y.y = F(q, x.y, y.y); x = a; }\n");
        o.f("__device__ __forceinline__ void u_ref_b(T2 &x, T2 &y, const R *m) { const R q = m[0]; T2 a; a.x = F(q, x.x, y.x); "
            "a.y = F(q, x.y, y.y); y.x = F(-q, y.x, x.x); y.y = F(-q, y.y, x.y); x = a; }\n");
    } else {  // m = {q, q, -q, -q}
        o.f("__device__ __forceinline__ void u_rot_a(T2 &x, T2 &y, const R *m) { const u64 *q = (const u64 *)m; "
            "const u64 X = pk(x.x, x.y), Y = pk(y.x, y.y); x = upk(fma2(q[1], Y, X)); y = upk(fma2(q[0], X, Y)); }\n");
        o.f("__device__ __forceinline__ void u_ref_b(T2 &x, T2 &y, const R *m) { const u64 *q = (const u64 *)m; "
            "const u64 X = pk(x.x, x.y), Y = pk(y.x, y.y); x = upk(fma2(q[0], X, Y)); y = upk(fma2(q[1], Y, X)); }\n");
    }
    o.f("__device__ __forceinline__ void u_rot_b(T2 &x, T2 &y, const R *m) { const R q = m[0]; T2 a; a.x = F(q, x.x, -y.x); "
        "a.y = F(q, x.y, -y.y); y.x = F(q, y.x, x.x); y.y = F(q, y.y, x.y); x = a; }\n");
    o.f("__device__ __forceinline__ void u_ref_a(T2 &x, T2 &y, const R *m) { const R q = m[0]; T2 a; a.x = F(q, y.x, x.x); "
        "a.y = F(q, y.y, x.y); y.x = F(q, x.x, -y.x); y.y = F(q, x.y, -y.y); x = a; }\n");
    o.f("__device__ __forceinline__ void u_mul(T2 &x, R ar, R ai) {\n"
        "  T2 a; a.x = F(ar, x.x, -ai * x.y); a.y = F(ar, x.y, ai * x.x); x = a;\n}\n");
    o.f("__device__ __forceinline__ void u_diag(T2 &x, T2 &y, const R *m) { u_mul(x, m[0], m[1]); u_mul(y, m[6], m[7]); }\n");
    o.f("__device__ __forceinline__ void u_swap(T2 &x, T2 &y) { T2 t = x; x = y; y = t; }\n");
    // Sums over the warp of M values per lane at once: each step trades half of the values with the
    // partner lane, so M sums take M - 1 + log2(32 / M) shuffles instead of 5 M; value i ends in the
    // lanes with lane / (32 / M) == i.
    o.f("template <int M> __device__ __forceinline__ R warp_sums(R (&q)[M], int lane) {\n"
        "  int of = 16;\n"
        "#pragma unroll\n"
        "  for (int m = M; m > 1; m >>= 1, of >>= 1) {\n"
        "    const bool up = lane & of;\n"
        "#pragma unroll\n"
        "    for (int i = 0; i < M / 2; ++i) if (i < m / 2) {\n"
        "      const R keep = up ? q[i + m / 2] : q[i], send = up ? q[i] : q[i + m / 2];\n"
        "      q[i] = keep + __shfl_xor_sync(0xffffffffu, send, of);\n"
        "    }\n"
        "  }\n"
        "  R s = q[0];\n"
        "#pragma unroll\n"
        "  for (int o_ = 16 / M; o_ > 0; o_ >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o_);\n"
        "  return s;\n}\n");
    o.f("__device__ __forceinline__ void kahan(R *s, R *c, R v) { const R y = v - *c; const R t = *s + y; *c = (t - *s) - y; "
        "*s = t; }\n");
    o.f("__device__ __forceinline__ void cp16(void *s, const void *g) {\n"
        "  asm volatile(\"cp.async.cg.shared.global [%%0], [%%1], 16;\\n\" :: \"r\"((u32)__cvta_generic_to_shared(s)), "
        "\"l\"(g) : \"memory\");\n}\n");
    o.f("__device__ __forceinline__ void cpcommit() { asm volatile(\"cp.async.commit_group;\\n\" ::: \"memory\"); }\n");
    o.f("__device__ __forceinline__ void cpwait0() { asm volatile(\"cp.async.wait_group 0;\\n\" ::: \"memory\"); }\n");
}

// Expression of the tile swizzle of `a` (the same bijection as tile_swizzle, k_tile.cuh).
std::string swz_expr(const char *a, int sw) {
    std::string x = std::string("(") + a + " >> " + std::to_string(sw) + ")";
    std::string f = x;
    for (int i = 3; i < kTileMaxBits; i += 3) f += " ^ (" + x + " >> " + std::to_string(i) + ")";
    return std::string("(") + a + " ^ (((" + f + ") & 7u) << " + std::to_string(sw - 3) + "))";
}

// Tile predicate of a set of gates: "" if some gate has no non-local control (every tile
// is selected), else the condition that one of them selects the tile at `bv` (a variable).
std::string any_selects(const RegGate *g, int count, const char *bv = "base") {
    std::vector<std::pair<uint64_t, uint64_t>> seen;
    std::string c;
    for (int i = 0; i < count; ++i) {
        if (g[i].hmask == 0) return "";
        bool dup = false;
        for (auto &s : seen) dup |= s.first == g[i].hmask && s.second == g[i].hvals;
        if (dup) continue;
        seen.push_back({g[i].hmask, g[i].hvals});
        char b[96];
        std::snprintf(b, sizeof(b), "%s((%s & 0x%llxull) == 0x%llxull)", c.empty() ? "" : " || ", bv,
                      (unsigned long long)g[i].hmask, (unsigned long long)g[i].hvals);
        c += b;
    }
    return c;
}

// Expressions of the gates' matrices (m), their update forms (real_forms) and gradient
// accumulator indices (consecutive in the order of the pass's gates).
struct Refs {
    std::vector<std::string> m;
    std::vector<int> form;
    std::vector<int> acc;
};

// How a pass applies its real gates. An uncontrolled rotation or reflection acts on every pair, so
// its larger entry can be divided out of the whole vector: 2 multiply-adds per output pair instead
// of a product and a multiply-add each (half the arithmetic; the divided entry is at least 1/sqrt(2)
// of the row, so nothing grows by more than sqrt(2) per gate). The last such gate of a pass, and
// every kRealRun-th, is applied in full with the product of the divided entries. Form 0: in full; 1:
// rotation, 2: reflection, divided. Inner products of psi and lambda taken in between are scaled
// back by the square of the product when they are summed. (Batch: only the rotations that each
// state's angles drive; their matrices, with the products, are formed per state beforehand.)
constexpr int kRealRun = 24;
bool divisible(const RegGate &g, bool batched) {
    return g.op == OP_REAL && g.rot && g.cqm == 0 && g.crm == 0 && g.hmask == 0 && (!batched || g.pkind == QS_GATE_RY);
}
std::vector<int> real_forms(const RegGate *g, int count, bool batched) {
    std::vector<int> form(count, 0), at;
    for (int i = 0; i < count; ++i)
        if (divisible(g[i], batched)) at.push_back(i);
    for (size_t j = 0; j + 1 < at.size(); ++j)
        if ((j + 1) % kRealRun != 0) form[at[j]] = g[at[j]].rot;
    return form;
}

// The derivative products of one rotation over its selected pairs, added up in `dot`: for float32 as
// packed multiply-adds (real and imaginary parts in the two lanes).
void emit_dots(Out &o, const RegGate &G, int E, char pauli, const char *v, const char *w, bool dbl) {
    const int p = G.p;
    bool first = true;
    for (int e = 0; e < E; ++e) {
        if (((e >> p) & 1) || (e & G.cqm) != G.cqv) continue;
        const int e2 = e | (1 << p);
        if (pauli == 'Y' && !dbl) {  // Im <l|Y p> = (l1 . p0) - (l0 . p1), real dot products
            o.f(first ? "u64 dp = mul2(pk(%s[%d].x, %s[%d].y), pk(%s[%d].x, %s[%d].y));\n"
                      : "dp = fma2(pk(%s[%d].x, %s[%d].y), pk(%s[%d].x, %s[%d].y), dp);\n",
                w, e2, w, e2, v, e, v, e);
            o.f(first ? "u64 dm = mul2(pk(%s[%d].x, %s[%d].y), pk(%s[%d].x, %s[%d].y));\n"
                      : "dm = fma2(pk(%s[%d].x, %s[%d].y), pk(%s[%d].x, %s[%d].y), dm);\n",
                w, e, w, e, v, e2, v, e2);
        } else if (pauli == 'Y') {
            o.f("dot += (%s[%d].x * %s[%d].x + %s[%d].y * %s[%d].y) - (%s[%d].x * %s[%d].x + %s[%d].y * %s[%d].y);\n", w, e2, v,
                e, w, e2, v, e, w, e, v, e2, w, e, v, e2);
        } else if (pauli == 'Z') {  // Im <l|Z p> = Im(conj(l0) p0) - Im(conj(l1) p1)
            o.f("dot += (%s[%d].x * %s[%d].y - %s[%d].y * %s[%d].x) - (%s[%d].x * %s[%d].y - %s[%d].y * %s[%d].x);\n", w, e, v,
                e, w, e, v, e, w, e2, v, e2, w, e2, v, e2);
        } else if (pauli == 'S') {
            const int es = G.side ? e2 : e;
            o.f("dot %s= (R)2 * (%s[%d].x * %s[%d].y - %s[%d].y * %s[%d].x);\n", G.side ? "-" : "+", w, es, v, es, w, es, v,
                es);
        }
        first = false;
    }
    if (pauli == 'Y' && !dbl) o.f("{ const T2 sp = upk(dp), sm = upk(dm); dot += (sp.x + sp.y) - (sm.x + sm.y); }\n");
}

// The pair updates of one gate on row registers v (and, adjoint, w with the derivative dot
// when the gate has a parameter). A rotation U = exp(-i theta P / 2) about the Pauli P = Y or Z
// (pauli 'Y' / 'Z') has dU/dtheta = (-i/2) P U, so with psi' = U^dagger psi (the amplitudes
// after the un-apply) Re <lambda| dU psi'> = Re <lambda| (-i/2) P psi> = Im <lambda| P psi> / 2:
// it is taken from the pair before the un-apply, 4 products per pair, no derivative matrix
// (the caller halves the sum). pauli 'S': a Z rotation on one side, whose other side follows from
// Im <lambda|psi> = 0 (plan_adjoint_gates).
void emit_gate_pairs(Out &o, const RegGate &G, int gi, int E, bool adjoint, bool param, char pauli, const char *v,
                     const char *w, const Refs &refs, bool dbl) {
    const char *M = refs.m[gi].c_str();
    const int p = G.p;
    if (refs.form[gi]) {  // divided: which entry was larger is a (uniform) parameter
        if (adjoint && param) emit_dots(o, G, E, pauli, v, w, dbl);
        const char *fn = refs.form[gi] == 1 ? "u_rot" : "u_ref";
        for (int b = 0; b < 2; ++b) {
            o.f(b ? "} else {\n" : "if (%s[4] == 0) {\n", M);
            for (int e = 0; e < E; ++e) {
                if ((e >> p) & 1) continue;
                o.f("%s_%c(%s[%d], %s[%d], %s);\n", fn, "ab"[b], v, e, v, e | (1 << p), M);
                if (adjoint) o.f("%s_%c(%s[%d], %s[%d], %s);\n", fn, "ab"[b], w, e, w, e | (1 << p), M);
            }
        }
        o.f("}\n");
        return;
    }
    if (adjoint && param) emit_dots(o, G, E, pauli, v, w, dbl);
    for (int e = 0; e < E; ++e) {
        if ((e >> p) & 1) continue;
        if ((e & G.cqm) != G.cqv) continue;
        const int e2 = e | (1 << p);
        auto op = [&](const char *a) {
            switch (G.op) {
            case OP_GEN: o.f("u_gen(%s[%d], %s[%d], %s);\n", a, e, a, e2, M); break;
            case OP_REAL: o.f("u_real(%s[%d], %s[%d], %s);\n", a, e, a, e2, M); break;
            case OP_DIAG: o.f("u_diag(%s[%d], %s[%d], %s);\n", a, e, a, e2, M); break;
            case OP_SWAP: o.f("u_swap(%s[%d], %s[%d]);\n", a, e, a, e2); break;
            case OP_SIDE: o.f("u_mul(%s[%d], %s[0], %s[1]);\n", a, G.side ? e2 : e, M, M); break;
            default: break;
            }
        };
        op(v);
        if (adjoint) op(w);
    }
}

// A run of consecutive diagonal gates (diag(a, d) or one side only) in a register group: they
// commute, so their product is applied at once. The gates are sorted into classes by the
// element bits their factor depends on (target place, in-row controls); per row, each class
// multiplies its gates' factors (a for target bit 0, d for bit 1) where the gate's tile and row
// predicates hold, and each element is then multiplied by the factors of the classes that
// select it: one complex product per gate and row plus one per selected element and class,
// instead of one per selected element and gate.
void emit_diag_run(Out &o, const RegGate *gs, int gi0, int count, int E, bool adjoint, const Refs &refs) {
    struct Cls {
        int p, cqm, cqv;
        bool has_a = false, has_d = false;
    };
    std::vector<Cls> cls;
    std::vector<int> cls_of(count);
    for (int i = 0; i < count; ++i) {
        const RegGate &R = gs[i];
        int c = -1;
        for (size_t j = 0; j < cls.size(); ++j)
            if (cls[j].p == R.p && cls[j].cqm == R.cqm && cls[j].cqv == R.cqv) c = (int)j;
        if (c < 0) {
            cls.push_back(Cls{R.p, R.cqm, R.cqv});
            c = (int)cls.size() - 1;
        }
        cls_of[i] = c;
        const bool a = R.op == OP_DIAG || (R.op == OP_SIDE && R.side == 0);
        const bool d = R.op == OP_DIAG || (R.op == OP_SIDE && R.side == 1);
        cls[c].has_a |= a;
        cls[c].has_d |= d;
    }
    o.f("      { // %d diagonal gates in %zu classes\n", count, cls.size());
    for (size_t c = 0; c < cls.size(); ++c) {
        if (cls[c].has_a) o.f("        T2 fa%zu; fa%zu.x = 1; fa%zu.y = 0;\n", c, c, c);
        if (cls[c].has_d) o.f("        T2 fd%zu; fd%zu.x = 1; fd%zu.y = 0;\n", c, c, c);
    }
    for (int i = 0; i < count; ++i) {
        const RegGate &R = gs[i];
        const int gi = gi0 + i, c = cls_of[i];
        std::string cond;
        char t[128];
        if (R.hmask) {
            std::snprintf(t, sizeof(t), "((base & 0x%llxull) == 0x%llxull)", (unsigned long long)R.hmask,
                          (unsigned long long)R.hvals);
            cond = t;
        }
        if (R.crm) {
            std::snprintf(t, sizeof(t), "%s((ra & 0x%xu) == 0x%xu)", cond.empty() ? "" : " && ", R.crm, R.crv);
            cond += t;
        }
        o.f("        if (%s) {", cond.empty() ? "true" : cond.c_str());
        const char *M = refs.m[gi].c_str();
        if (R.op == OP_DIAG)
            o.f(" u_mul(fa%d, %s[0], %s[1]); u_mul(fd%d, %s[6], %s[7]);", c, M, M, c, M, M);
        else
            o.f(" u_mul(f%c%d, %s[0], %s[1]);", R.side ? 'd' : 'a', c, M, M);
        o.f(" }\n");
    }
    for (int e = 0; e < E; ++e) {
        for (size_t c = 0; c < cls.size(); ++c) {
            if ((e & cls[c].cqm) != cls[c].cqv) continue;
            const bool hi = (e >> cls[c].p) & 1;
            if (hi ? !cls[c].has_d : !cls[c].has_a) continue;
            const char f = hi ? 'd' : 'a';
            o.f("        u_mul(v[%d], f%c%zu.x, f%c%zu.y);\n", e, f, c, f, c);
            if (adjoint) o.f("        u_mul(w[%d], f%c%zu.x, f%c%zu.y);\n", e, f, c, f, c);
        }
    }
    o.f("      }\n");
}

// The Pauli of a parameterised gate of the sweep: its rotation kind (batch), or the structure
// the planner forces on rotations (RY: real, RZ: diagonal); 0 when neither.
char pauli_of(const RegGate &R, bool batched) {
    if (batched) return R.pkind == QS_GATE_RY ? 'Y' : R.pkind == QS_GATE_RZ ? 'Z' : 0;
    return R.op == OP_REAL ? 'Y' : R.op == OP_DIAG ? 'Z' : R.op == OP_SIDE ? 'S' : 0;
}

}  // namespace

namespace {

// Whether the rows of a group, one per thread, cover runs of at least 32 bytes of the state per
// access: complex64 without qubits 1 and 2 in registers (qubit 0 may be, its pairs move as vectors),
// complex128 without 0 and 1.
bool direct_rows(const TileGroup &Gr, int r, bool dbl) {
    uint32_t Q = 0;
    for (int q = 0; q < r; ++q) Q |= 1u << Gr.q[q];
    return (Q & (dbl ? 3u : 6u)) == 0;
}

// The local qubits that the bits of a group's row number stand for: first those whose bits spread a
// warp's rows over all shared-memory banks (tile_swizzle: complex64's qubit 0 in place, qubit b above on
// bank bit (b - low) mod 3: the lowest free one of each class), then the others, ascending. In plain
// ascending order 38 % of the shared-memory wavefronts of a random circuit's passes were conflicts.
std::vector<int> row_bits(const TileGroup &Gr, int k, int r, bool dbl) {
    uint32_t left = (1u << k) - 1u;
    for (int q = 0; q < r; ++q) left &= ~(1u << Gr.q[q]);
    const int low = dbl ? 0 : 1;
    std::vector<int> pos;
    auto take = [&](int b) {
        pos.push_back(b);
        left &= ~(1u << b);
    };
    if (low && (left & 1u)) take(0);
    for (int c = 0; c < 3; ++c)
        for (int b = low + c; b < k; b += 3)
            if ((left >> b) & 1u) {
                take(b);
                break;
            }
    for (int b = 0; b < k; ++b)
        if ((left >> b) & 1u) take(b);
    return pos;
}

// " | (...)" terms that put bit i of rho at bit to[i], by runs that move by the same distance.
std::string scatter_terms(const std::vector<int> &to, const char *type) {
    std::string a;
    for (size_t i = 0; i < to.size();) {
        size_t j = i + 1;
        while (j < to.size() && to[j] - (int)j == to[i] - (int)i) ++j;
        const uint32_t mask = ((1u << j) - 1u) & ~((1u << i) - 1u);
        const int d = to[i] - (int)i;
        char b[96];
        std::snprintf(b, sizeof(b), " | ((%s)(rho & 0x%xu) %s %d)", type, mask, d < 0 ? ">>" : "<<", d < 0 ? -d : d);
        a += b;
        i = j;
    }
    return a;
}

}  // namespace

// A block alternates between copies, row moves and arithmetic with block barriers in between, so an
// SM needs other blocks to fill its pipes, and the next tile's copy must run meanwhile: two tile
// buffers wherever two blocks still fit, and three blocks where their buffers fit and the rows are
// complex64 (80 registers a thread: 1000-gate circuit at n = 28 57.8 -> 56.1 ms, QFT29 7.88 -> 7.68,
// n = 24 gradient 7.99 -> 7.61; complex128 rows alone take 64). One buffer costs 15-20 %; blocks of 128
// threads, 5-qubit groups and tiles of 2^11 or 2^13 amplitudes were within 3 % or slower, rows of
// 64 or 32 contiguous bytes (one or two more qubits per pass) 15 and 40 % slower.
JitShape jit_shape(int dtype, bool adjoint, int k) {
    const size_t tile = (size_t(1) << k) * (dtype == QS_C64 ? 8 : 16) * (adjoint ? 2 : 1);
    if (dtype == QS_C64 && 6 * tile <= 200 * 1024) return {3, true};
    return {adjoint && dtype == QS_C128 ? 1 : 2, 2 * tile <= 100 * 1024};
}

std::string jit_pass_source(int dtype, bool adjoint, const TilePass &P, const TileGroup *groups,
                            const RegGate *gates, const char *kname, bool batched) {
    const bool dbl = dtype == QS_C128;
    const int SW = dbl ? 3 : 4;
    const int VEC = dbl ? 1 : 2;
    const int T = kTileThreads;
    const int k = P.k;
    const uint32_t nvec = (1u << k) / VEC;
    const uint32_t steps = (nvec + T - 1) / T;
    const int G = P.gate_count;
    const RegGate *pg = gates + P.gate_begin;
    // Matrix of each gate as an expression: parameters of the kernel (single state), or, in a
    // batch, shared-memory rows for the parameterised gates (pm_; J = index among them), copied in
    // with each tile from the matrices of the tile's state.
    std::vector<int> pj(G, -1);
    int NPG = 0;
    if (batched)
        for (int i = 0; i < G; ++i)
            if (pg[i].pkind != 0) pj[i] = NPG++;
    const int NP = adjoint ? (batched ? NPG : P.nparam) : 0;  // gradient accumulators
    Refs refs;
    refs.m.resize(G);
    refs.form = real_forms(pg, G, batched);
    int nacc = 0;
    for (int i = 0; i < G; ++i) {
        char b[48];
        if (pj[i] >= 0) std::snprintf(b, sizeof(b), "(pm_ + %d)", 8 * pj[i]);
        else std::snprintf(b, sizeof(b), "a.m[%d]", i);
        refs.m[i] = b;
        refs.acc.push_back(adjoint && pg[i].slot >= 0 ? nacc++ : -1);
    }
    // debug build: every global access checked against the state's size (2^n), writes counted
    const bool dbg = kDebugBuild && !batched;
    Out o;
    preamble(o, dbl);
    if (dbg) {
        o.f("struct DebugState { unsigned status, pad; u64 n_amps; unsigned *counts; u64 count_n; u64 first_bad; };\n");
        o.f("__device__ __forceinline__ bool dok(DebugState *d, u64 i, int span) {\n"
            "  if (d->n_amps == 0 || i + span <= d->n_amps) return true;\n"
            "  d->first_bad = i; atomicOr(&d->status, 1u); return false;\n}\n");
        o.f("__device__ __forceinline__ void dcount(DebugState *d, u64 i, int span) {\n"
            "  if (!d->counts) return;\n"
            "  for (int j = 0; j < span; ++j) if (i + j < d->count_n) atomicAdd(d->counts + i + j, 1u);\n}\n");
    }
    // parameter block: the fixed matrices of the pass's gates (U, or U^dagger in the adjoint
    // sweep); single-state sweep: the scales and global gradient slots of its parameterised gates
    o.f("struct alignas(16) A {\n  R m[%d][8];\n", G > 0 ? G : 1);
    if (adjoint && !batched) o.f("  double f[%d];\n  int gs[%d];\n", NP > 0 ? NP : 1, NP > 0 ? NP : 1);
    o.f("};\n");
    o.f("__device__ __forceinline__ u32 swz(u32 a) { return %s; }\n", swz_expr("a", SW).c_str());
    const int minb = jit_shape(dtype, adjoint, k).blocks;
    if (batched)
        o.f("extern \"C\" __global__ void __launch_bounds__(%d, %d) %s(T2 *__restrict__ psi, T2 *__restrict__ lam, "
            "double *__restrict__ part, u64 stride, u64 nstates, const R *__restrict__ mats, "
            "const __grid_constant__ A a) {\n",
            T, minb, kname);
    else if (adjoint)
        o.f("extern \"C\" __global__ void __launch_bounds__(%d, %d) %s(T2 *__restrict__ psi, T2 *__restrict__ lam, "
            "double *__restrict__ part, u64 part_stride, const __grid_constant__ A a%s) {\n",
            T, minb, kname, dbg ? ", DebugState *dbg" : "");
    else
        o.f("extern \"C\" __global__ void __launch_bounds__(%d, %d) %s(T2 *__restrict__ psi, const __grid_constant__ A a%s) {\n",
            T, minb, kname, dbg ? ", DebugState *dbg" : "");
    const bool db = jit_shape(dtype, adjoint, k).db;
    const uint32_t TILE = 1u << k;
    const uint32_t BUF = (adjoint ? 2 : 1) * TILE;  // one buffer: psi tile (and lambda tile)
    o.f("  extern __shared__ __align__(16) unsigned char sm_[];\n");
    o.f("  T2 *const sm0 = reinterpret_cast<T2 *>(sm_);\n");
    o.f("  R *const sr_ = reinterpret_cast<R *>(sm0 + %u);\n", (db ? 2 : 1) * BUF);
    const int pm_state = batched ? jit_batch_words(NPG, adjoint) : 0;  // reals per state
    const int pm_words = (db ? 2 : 1) * pm_state;
    if (adjoint) {
        o.f("  R *acc_s = sr_ + %d;\n", pm_words);
        o.f("  R *acc_c = acc_s + %d;\n", (NP > 0 ? NP : 1) * (T / 32));
        o.f("  for (int i = threadIdx.x; i < %d; i += %d) { acc_s[i] = 0; acc_c[i] = 0; }\n", (NP > 0 ? NP : 1) * (T / 32), T);
        o.f("  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;\n");
    }
    o.f("  const u32 tid = threadIdx.x;\n");
    // this thread's part of the copy addresses (XOR-linear in the element index)
    o.f("  const u32 o_t = tid * %d;\n", VEC);
    {
        std::string g = "0ull";
        for (int r = 0; r < P.nruns; ++r) {
            char b[160];
            std::snprintf(b, sizeof(b), " | ((u64)((o_t >> %d) & %uu) << %d)", P.run_src[r], (1u << P.run_len[r]) - 1u,
                          P.run_dst[r]);
            g += b;
        }
        o.f("  const u64 g_t = %s;\n", g.c_str());
    }
    o.f("  const u32 s_t = swz(o_t);\n");
    const bool cp_guard = nvec < (uint32_t)T;
    int logt = 0;
    while ((1ull << logt) < P.ntiles) ++logt;
    if (batched)
        o.f("  const u64 ntiles = nstates << %d;  // %llu tiles per state\n", logt, (unsigned long long)P.ntiles);
    else
        o.f("  const u64 ntiles = %lluull;\n", (unsigned long long)P.ntiles);
    {
        std::string b = "0ull";
        for (int s = 0; s < P.tnseg; ++s) {
            char t[96];
            std::snprintf(t, sizeof(t), " | ((t_ << %d) & 0x%llxull)", P.tshift[s], (unsigned long long)P.tmask[s]);
            b += t;
        }
        if (batched)  // the tile index within its state: the low bits of the batch-wide index
            o.f("  auto tile_base = [](u64 t_) -> u64 { t_ &= %lluull; return %s; };\n",
                (unsigned long long)(P.ntiles - 1), b.c_str());
        else
            o.f("  auto tile_base = [](u64 t_) -> u64 { return %s; };\n", b.c_str());
    }
    if (batched) {
        o.f("  auto gvec = [&](T2 *v_, u64 t_) -> T2 * { return v_ + (t_ >> %d) * stride; };\n", logt);
    } else {
        o.f("  auto gvec = [](T2 *v_, u64) -> T2 * { return v_; };\n");
    }
    std::string sel;
    if (P.hctrl) sel = any_selects(pg, G, "b_");
    if (!sel.empty()) o.f("  auto selected = [](u64 b_) -> bool { return %s; };\n", sel.c_str());
    // tile copies (asynchronous loads into swizzled shared-memory positions; stores from registers)
    auto copies = [&](bool load, const char *gname, const char *tname, const char *bname) {
        if (cp_guard) o.f("    if (tid < %uu) {\n", nvec);
        for (uint32_t j = 0; j < steps; ++j) {
            const uint32_t oj = j * T * VEC;
            const unsigned long long gj = (unsigned long long)scatter_host(P, oj);
            const uint32_t sj = tile_swizzle(oj, SW);
            if (dbg) {
                o.f("    if (dok(dbg, %s | g_t | 0x%llxull, %d)) ", bname, gj, VEC);
                if (!load) o.f("{ dcount(dbg, %s | g_t | 0x%llxull, %d); ", bname, gj, VEC);
            }
            if (load)  // 16 bytes: a complex128 amplitude or a pair of complex64 (tile_swizzle)
                o.f("    cp16(%s + (s_t ^ %uu), %s + (%s | g_t | 0x%llxull));\n", tname, sj, gname, bname, gj);
            else if (!dbl)
                o.f("    *reinterpret_cast<T4 *>(%s + (%s | g_t | 0x%llxull)) = *reinterpret_cast<const T4 *>(%s + (s_t ^ "
                    "%uu));\n",
                    gname, bname, gj, tname, sj);
            else
                o.f("    %s[%s | g_t | 0x%llxull] = %s[s_t ^ %uu];\n", gname, bname, gj, tname, sj);
            if (dbg && !load) o.f("    }\n");
        }
        if (cp_guard) o.f("    }\n");
    };
    auto loads = [&](const char *tname, const char *bname, const char *tau_name, const char *pm_index) {
        o.f("    {\n    T2 *tq = %s;\n    const T2 *gp_ = gvec(psi, %s);\n", tname, tau_name);
        copies(true, "gp_", "tq", bname);
        if (adjoint) {
            o.f("    T2 *tr = tq + %u;\n    const T2 *gl_ = gvec(lam, %s);\n", TILE, tau_name);
            copies(true, "gl_", "tr", bname);
        }
        if (pm_state > 0) {  // the matrices of the tile's state
            const int per = dbl ? 2 : 4, chunks = pm_state / per;
            o.f("    const R *gm_ = mats + (%s >> %d) * %dull;\n    R *sm_m = sr_ + (%s) * %d;\n", tau_name, logt, pm_state,
                db ? pm_index : "0", pm_state);
            o.f("    for (u32 c_ = tid; c_ < %du; c_ += %d) cp16(sm_m + c_ * %d, gm_ + c_ * %d);\n", chunks, T, per, per);
        }
        o.f("    }\n    cpcommit();\n");
    };
    const char *skip_next = sel.empty() ? "" : "    while (nxt < ntiles && !selected(tile_base(nxt))) nxt += gridDim.x;\n";
    o.f("  u64 tau = blockIdx.x;\n");
    if (!sel.empty()) o.f("  while (tau < ntiles && !selected(tile_base(tau))) tau += gridDim.x;\n");
    if (db) o.f("  int cur = 0;\n");
    if (db) {
        o.f("  if (tau < ntiles) {\n    const u64 b0 = tile_base(tau);\n");
        loads("sm0", "b0", "tau", "0");
        o.f("  }\n");
    }
    o.f("  while (tau < ntiles) {\n");
    o.f("    const u64 base = tile_base(tau);\n");
    o.f("    u64 nxt = tau + gridDim.x;\n%s", skip_next);
    if (db)
        o.f("    T2 *tp = sm0 + cur * %u;\n", BUF);
    else
        o.f("    T2 *tp = sm0;  // one buffer\n");
    if (adjoint) o.f("    T2 *tl = tp + %u;\n", TILE);
    if (pm_state > 0) o.f("    const R *const pm_ = sr_ + %s * %d;\n", db ? "cur" : "0", pm_state);
    if (db) {
        // one barrier: this tile has arrived, and every thread is done with the one before, whose
        // buffer the next tile's copy takes
        o.f("    cpwait0();\n    __syncthreads();\n");
        o.f("    if (nxt < ntiles) {\n      const u64 nb = tile_base(nxt);\n      T2 *tn = sm0 + (cur ^ 1) * %u;\n", BUF);
        loads("tn", "nb", "nxt", "cur ^ 1");
        o.f("    }\n");
    } else {
        loads("tp", "base", "tau", "0");
        o.f("    cpwait0();\n    __syncthreads();\n");
    }
    const bool end_sync = !db || (adjoint && batched && NP > 0);  // a barrier after the tile's last access

    bool stored = false;
    for (int gi_ = 0; gi_ < P.group_count; ++gi_) {
        const TileGroup &Gr = groups[P.group_begin + gi_];
        const int r = Gr.r;
        const int E = 1 << r;
        const uint32_t rows = 1u << (k - r);
        const uint32_t rblocks = (rows + T - 1) / T;
        const int gb = Gr.gate_begin - P.gate_begin;  // pass-relative
        o.f("    // register group %d: qubits", gi_);
        for (int q = 0; q < r; ++q) o.f(" %d", Gr.q[q]);
        o.f(", %d gates\n", Gr.gate_count);
        std::string gcond;
        if (Gr.hctrl && !Gr.has_g && !Gr.has_s) gcond = any_selects(pg + gb, Gr.gate_count);
        o.f("    if (%s) {\n", gcond.empty() ? "true" : gcond.c_str());
        // element offsets of the gather and the scatter
        std::vector<uint32_t> og(E), os(E);
        for (int e = 0; e < E; ++e) {
            uint32_t off = 0;
            for (int q = 0; q < r; ++q)
                if ((e >> q) & 1) off ^= Gr.qsw[q];
            og[e] = Gr.has_g ? Gr.gperm[e] : off;
            os[e] = Gr.has_s ? Gr.sperm[e] : off;
        }
        // The last group writes its rows straight to the state where every tile runs it and its
        // qubits leave the low ones to the lanes (runs of at least 32 bytes per store): the tile's
        // last trip through shared memory and a block barrier less.
        const bool direct = gi_ + 1 == P.group_count && gcond.empty() && direct_rows(Gr, r, dbl);
        std::vector<unsigned long long> ge(E);
        for (int e = 0; e < E; ++e) ge[e] = scatter_host(P, tile_swizzle(os[e], SW));
        if (direct) {
            o.f("    T2 *gp_ = gvec(psi, tau);\n");
            if (adjoint) o.f("    T2 *gl_ = gvec(lam, tau);\n");
        }
        stored = direct;
        const std::vector<int> rowpos = row_bits(Gr, k, r, dbl);
        for (uint32_t rb = 0; rb < rblocks; ++rb) {
            o.f("    {\n      const u32 rho = %uu + tid;\n", rb * T);
            const bool guard = rows < (rb + 1) * (uint32_t)T;
            const std::string ra = "0u" + scatter_terms(rowpos, "u32");
            o.f("      const u32 ra = %s;\n      const u32 rs = swz(ra);\n", ra.c_str());
            o.f("      const bool act = %s;\n", guard ? (std::string("rho < ") + std::to_string(rows) + "u").c_str() : "true");
            o.f("      T2 v[%d];\n", E);
            if (adjoint) o.f("      T2 w[%d];\n", E);
            o.f("      if (act) {\n");
            // float32 amplitudes that differ in local qubit 0 are one 16-byte vector
            auto row_move = [&](bool load, const char *reg, const char *tile, const std::vector<uint32_t> &off) {
                for (int e = 0; e < E; ++e) {
                    if (!dbl && !(e & 1) && E > 1 && (off[e] ^ off[e | 1]) == 1u) {
                        const int e0 = (off[e] & 1u) ? e | 1 : e, e1 = e0 ^ 1;
                        if (load)
                            o.f("        { const T4 q = *reinterpret_cast<const T4 *>(%s + (rs ^ %uu)); %s[%d].x = q.x; "
                                "%s[%d].y = q.y; %s[%d].x = q.z; %s[%d].y = q.w; }\n",
                                tile, off[e0], reg, e0, reg, e0, reg, e1, reg, e1);
                        else
                            o.f("        { T4 q; q.x = %s[%d].x; q.y = %s[%d].y; q.z = %s[%d].x; q.w = %s[%d].y; "
                                "*reinterpret_cast<T4 *>(%s + (rs ^ %uu)) = q; }\n",
                                reg, e0, reg, e0, reg, e1, reg, e1, tile, off[e0]);
                        ++e;
                    } else if (load) {
                        o.f("        %s[%d] = %s[rs ^ %uu];\n", reg, e, tile, off[e]);
                    } else {
                        o.f("        %s[rs ^ %uu] = %s[%d];\n", tile, off[e], reg, e);
                    }
                }
            };
            row_move(true, "v", "tp", og);
            if (adjoint) row_move(true, "w", "tl", og);
            o.f("      } else {\n");
            for (int e = 0; e < E; ++e) {
                o.f("        v[%d].x = 0; v[%d].y = 0;\n", e, e);
                if (adjoint) o.f("        w[%d].x = 0; w[%d].y = 0;\n", e, e);
            }
            o.f("      }\n");
            auto mergeable = [&](int g) {
                const RegGate &R = pg[gb + g];
                return (R.op == OP_DIAG || R.op == OP_SIDE) && !(adjoint && R.slot >= 0);
            };
            // derivative products wait in registers and are summed over the warp kDotRun at a time
            constexpr int kDotRun = 8;
            int npend = 0, pend0 = 0;
            auto flush_dots = [&]() {
                if (npend == 0) return;
                int M = 1;
                while (M < npend) M *= 2;
                o.f("      { R q_[%d] = {", M);
                for (int i = 0; i < M; ++i) {
                    if (i < npend) o.f("%sdt%d", i ? ", " : "", pend0 + i);
                    else o.f(", 0");
                }
                o.f("};\n        const R s_ = warp_sums<%d>(q_, lane);\n", M);
                o.f("        if ((lane & %d) == 0%s) { const int i_ = %d + (lane / %d), j_ = i_ * %d + warp; kahan(acc_s + j_, acc_c "
                    "+ j_, s_%s); } }\n",
                    32 / M - 1, M > npend ? (" && lane / " + std::to_string(32 / M) + " < " + std::to_string(npend)).c_str() : "",
                    pend0, 32 / M, T / 32, batched ? (" * pm_[" + std::to_string(8 * NPG) + " + i_]").c_str() : "");
                npend = 0;
            };
            for (int g = 0; g < Gr.gate_count; ++g) {
                if (g + 1 < Gr.gate_count && mergeable(g) && mergeable(g + 1)) {
                    int h = g;
                    while (h < Gr.gate_count && mergeable(h)) ++h;
                    emit_diag_run(o, pg + gb + g, gb + g, h - g, E, adjoint, refs);
                    g = h - 1;
                    continue;
                }
                const RegGate &R = pg[gb + g];
                const int gi = gb + g;  // pass-relative gate index
                const int slot = adjoint && R.slot >= 0 ? refs.acc[gi] : -1;
                o.f("      // gate %d: op %d, place %d, cq %x/%x, rows %x/%x\n", gi, R.op, R.p, R.cqm, R.cqv, R.crm, R.crv);
                const bool tile_guard = R.hmask != 0;
                if (slot >= 0) {
                    if (npend == 0) pend0 = slot;
                    o.f("      R dt%d = 0;\n", slot);
                    ++npend;
                }
                if (tile_guard)
                    o.f("      if ((base & 0x%llxull) == 0x%llxull) {\n", (unsigned long long)R.hmask,
                        (unsigned long long)R.hvals);
                else
                    o.f("      {\n");
                if (slot >= 0) o.f("        R dot = 0;\n");
                std::string rc = "act";
                if (R.crm) {
                    char t[80];
                    std::snprintf(t, sizeof(t), "act && ((ra & 0x%xu) == 0x%xu)", R.crm, R.crv);
                    rc = t;
                }
                const bool need_rc = guard || R.crm;
                if (need_rc) o.f("        if (%s) {\n", rc.c_str());
                const char pauli = slot >= 0 ? pauli_of(R, batched) : 0;
                emit_gate_pairs(o, R, gi, E, adjoint, slot >= 0, pauli, "v", "w", refs, dbl);
                if (need_rc) o.f("        }\n");
                if (slot >= 0) o.f("        dt%d = (R)0.5 * dot;\n", slot);
                o.f("      }\n");
                if (npend == kDotRun) flush_dots();
            }
            flush_dots();
            o.f("      if (act) {\n");
            if (direct) {
                std::vector<int> to;
                for (int b : rowpos) to.push_back(__builtin_ctzll(scatter_host(P, 1u << b)));
                o.f("        const u64 ga = base%s;\n", scatter_terms(to, "u64").c_str());
                for (int vec = 0; vec < (adjoint ? 2 : 1); ++vec) {
                    const char *reg = vec ? "w" : "v", *gv = vec ? "gl_" : "gp_";
                    for (int e = 0; e < E; ++e) {
                        const bool pair = !dbl && !(e & 1) && E > 1 && (ge[e] ^ ge[e | 1]) == 1u;
                        const int e0 = pair && (ge[e] & 1u) ? e | 1 : e;
                        if (dbg) o.f("        if (dok(dbg, ga | 0x%llxull, %d)) { dcount(dbg, ga | 0x%llxull, %d);", ge[e0], pair ? 2 : 1, ge[e0], pair ? 2 : 1);
                        if (pair)
                            o.f("        { T4 q; q.x = %s[%d].x; q.y = %s[%d].y; q.z = %s[%d].x; q.w = %s[%d].y; "
                                "*reinterpret_cast<T4 *>(%s + (ga | 0x%llxull)) = q; }\n",
                                reg, e0, reg, e0, reg, e0 ^ 1, reg, e0 ^ 1, gv, ge[e0]);
                        else
                            o.f("        %s[ga | 0x%llxull] = %s[%d];\n", gv, ge[e0], reg, e);
                        if (dbg) o.f("        }\n");
                        e += pair;
                    }
                }
            } else {
                row_move(false, "v", "tp", os);
                if (adjoint) row_move(false, "w", "tl", os);
            }
            o.f("      }\n    }\n");
        }
        o.f("    }\n%s", stored && !end_sync ? "" : "    __syncthreads();\n");
    }
    if (!stored) {
        o.f("    {\n    T2 *gp_ = gvec(psi, tau);\n");
        copies(false, "gp_", "tp", "base");
        if (adjoint) {
            o.f("    T2 *gl_ = gvec(lam, tau);\n");
            copies(false, "gl_", "tl", "base");
        }
        o.f("    }\n%s", end_sync ? "    __syncthreads();\n" : "");
    }
    if (adjoint && batched && NP > 0) {
        // this tile's gradient partials (sum over the block's warps), then fresh accumulators;
        // the loop's next block barrier orders them before the next tile adds to them
        o.f("    for (int p = threadIdx.x; p < %d; p += %d) {\n", NP, T);
        o.f("      double s = 0.0;\n");
        o.f("      for (int w_ = 0; w_ < %d; ++w_) { s += (double)acc_s[p * %d + w_] - (double)acc_c[p * %d + w_]; "
            "acc_s[p * %d + w_] = 0; acc_c[p * %d + w_] = 0; }\n",
            T / 32, T / 32, T / 32, T / 32, T / 32);
        o.f("      part[((u64)p * nstates + (tau >> %d)) * %lluull + (tau & %lluull)] = s;\n    }\n", logt,
            (unsigned long long)P.ntiles, (unsigned long long)(P.ntiles - 1));
    }
    o.f("    tau = nxt;\n%s  }\n", db ? "    cur ^= 1;\n" : "");
    if (adjoint && !batched && NP > 0) {
        o.f("  __syncthreads();\n");
        o.f("  for (int p = threadIdx.x; p < %d; p += %d) {\n", NP, T);
        o.f("    double s = 0.0;\n");
        o.f("    for (int w_ = 0; w_ < %d; ++w_) s += (double)acc_s[p * %d + w_] - (double)acc_c[p * %d + w_];\n", T / 32,
            T / 32, T / 32);
        o.f("    part[(u64)a.gs[p] * part_stride + blockIdx.x] = s * a.f[p];\n  }\n");
    }
    o.f("}\n");
    return o.s;
}

namespace {

// ---------------------------------------------------------------------------------------------
// Compile cache
// ---------------------------------------------------------------------------------------------

struct Module {
    std::string source;       // all kernels of the module
    std::vector<char> cubin;
    std::vector<std::string> names;
    cudaLibrary_t lib = nullptr;  // loaded on first launch
    std::vector<cudaKernel_t> kernels;
    std::vector<size_t> smem_set[64];  // per device: dynamic shared memory configured per kernel
    std::vector<int> occ[64];          // per device: resident blocks per SM per kernel (0 = unknown)
};

std::mutex g_mu;
std::vector<std::unique_ptr<Module>> g_modules;
std::unordered_map<std::string, std::pair<int, int>> g_by_source;  // kernel source -> (module, kernel)
std::unordered_map<std::string, std::pair<int, int>> g_by_shape;   // shape key -> (module, kernel)

// Everything a pass's generated source depends on, as bytes (the matrices excluded): looking
// this up costs far less than generating the source, so a repeated circuit finds its kernels
// without writing them again.
std::string shape_key(int dtype, bool adjoint, bool batched, const TilePass &P, const TileGroup *groups,
                      const RegGate *gates) {
    std::string k;
    auto put = [&k](const void *p, size_t n) { k.append(static_cast<const char *>(p), n); };
    const int hdr[5] = {dtype, adjoint ? 1 : 0, batched ? 1 : 0, P.gate_count, P.group_count};
    put(hdr, sizeof(hdr));
    put(&P.n, sizeof(P.n));
    put(&P.k, sizeof(P.k));
    put(&P.nruns, sizeof(P.nruns));
    put(P.run_src, sizeof(P.run_src));
    put(P.run_len, sizeof(P.run_len));
    put(P.run_dst, sizeof(P.run_dst));
    put(P.tmask, sizeof(P.tmask));
    put(P.tshift, sizeof(P.tshift));
    put(&P.tnseg, sizeof(P.tnseg));
    put(&P.ntiles, sizeof(P.ntiles));
    put(&P.hctrl, sizeof(P.hctrl));
    put(&P.nparam, sizeof(P.nparam));
    for (int i = 0; i < P.group_count; ++i) {
        TileGroup g = groups[P.group_begin + i];
        g.gate_begin -= P.gate_begin;
        put(&g, sizeof(g));
    }
    for (int i = 0; i < P.gate_count; ++i) {
        const RegGate &g = gates[P.gate_begin + i];
        put(&g.p, 4);  // p, cqm, cqv, pad0
        put(&g.crm, sizeof(g.crm));
        put(&g.crv, sizeof(g.crv));
        put(&g.op, sizeof(g.op));
        put(&g.side, sizeof(g.side));
        put(&g.slot, sizeof(g.slot));
        put(&g.rot, sizeof(g.rot));
        put(&g.hmask, sizeof(g.hmask));
        put(&g.hvals, sizeof(g.hvals));
        if (batched) put(&g.pkind, sizeof(g.pkind));  // the rotations whose matrices are each state's own
    }
    return k;
}

bool compile_cubin(const std::string &src, std::vector<char> *cubin, std::string *err) {
    nvrtcProgram prog;
    nvrtcResult r = nvrtcCreateProgram(&prog, src.c_str(), "qs_jit_pass.cu", 0, nullptr, nullptr);
    if (r != NVRTC_SUCCESS) {
        *err = std::string("nvrtcCreateProgram: ") + nvrtcGetErrorString(r);
        return false;
    }
    const char *opts[] = {"--gpu-architecture=sm_103a", "-std=c++17", "--fmad=true", "-DQS_JIT=1"};
    r = nvrtcCompileProgram(prog, (int)(sizeof(opts) / sizeof(opts[0])), opts);
    if (r != NVRTC_SUCCESS) {
        size_t ls = 0;
        nvrtcGetProgramLogSize(prog, &ls);
        std::string log(ls, '\0');
        if (ls) nvrtcGetProgramLog(prog, &log[0]);
        *err = std::string("NVRTC compile failed: ") + nvrtcGetErrorString(r) + "\n" + log.substr(0, 4000);
        nvrtcDestroyProgram(&prog);
        return false;
    }
    size_t n = 0;
    r = nvrtcGetCUBINSize(prog, &n);
    if (r == NVRTC_SUCCESS) {
        cubin->resize(n);
        r = nvrtcGetCUBIN(prog, cubin->data());
    }
    nvrtcDestroyProgram(&prog);
    if (r != NVRTC_SUCCESS) {
        *err = std::string("nvrtcGetCUBIN: ") + nvrtcGetErrorString(r);
        return false;
    }
    return true;
}

// ---------------------------------------------------------------------------------------------
// On-disk kernel cache (QS_JIT_CACHE_DIR)
// ---------------------------------------------------------------------------------------------
// With QS_JIT_CACHE_DIR=<directory> every compiled kernel is also written there, one file per
// kernel source, and a later process loads it instead of compiling. A file holds a header, the
// kernel's full source and its cubin; it is used only when the stored source equals the
// wanted one byte for byte (so neither a name collision nor a stale file can give another
// kernel), and written under a temporary name then renamed (readers never see a partial one).
constexpr char kDiskMagic[8] = {'Q', 'S', 'J', 'I', 'T', 'C', '1', '\n'};

std::string disk_cache_dir() {
    const char *d = std::getenv("QS_JIT_CACHE_DIR");
    return (d && *d) ? std::string(d) : std::string();
}

// File of a kernel source: FNV-1a of the source, the compile options and the NVRTC version.
std::string disk_path(const std::string &dir, const std::string &src) {
    int major = 0, minor = 0;
    nvrtcVersion(&major, &minor);
    uint64_t h = 1469598103934665603ull;
    auto mix = [&h](const char *p, size_t n) {
        for (size_t i = 0; i < n; ++i) {
            h ^= (unsigned char)p[i];
            h *= 1099511628211ull;
        }
    };
    char v[64];
    const int m = std::snprintf(v, sizeof(v), "sm_103a;c++17;fmad;nvrtc %d.%d;", major, minor);
    mix(v, (size_t)m);
    mix(src.data(), src.size());
    char name[64];
    std::snprintf(name, sizeof(name), "/qs_jit_%016llx.bin", (unsigned long long)h);
    return dir + name;
}

bool disk_load(const std::string &path, const std::string &src, std::vector<char> *cubin) {
    FILE *f = std::fopen(path.c_str(), "rb");
    if (!f) return false;
    std::vector<char> all;
    char buf[1 << 16];
    size_t got;
    while ((got = std::fread(buf, 1, sizeof(buf), f)) > 0) all.insert(all.end(), buf, buf + got);
    std::fclose(f);
    const size_t hdr = sizeof(kDiskMagic) + sizeof(uint64_t);
    if (all.size() < hdr || std::memcmp(all.data(), kDiskMagic, sizeof(kDiskMagic)) != 0) return false;
    uint64_t len = 0;
    std::memcpy(&len, all.data() + sizeof(kDiskMagic), sizeof(len));
    if (len != src.size() || all.size() <= hdr + len || std::memcmp(all.data() + hdr, src.data(), len) != 0) return false;
    cubin->assign(all.begin() + (ptrdiff_t)(hdr + len), all.end());
    return true;
}

void disk_store(const std::string &path, const std::string &src, const std::vector<char> &cubin) {
    const std::string tmp = path + ".tmp" + std::to_string((unsigned long long)std::hash<std::thread::id>()(
                                                std::this_thread::get_id()));
    FILE *f = std::fopen(tmp.c_str(), "wb");
    if (!f) return;  // not writable: the cache is an optimisation only
    const uint64_t len = src.size();
    bool ok = std::fwrite(kDiskMagic, 1, sizeof(kDiskMagic), f) == sizeof(kDiskMagic) &&
              std::fwrite(&len, 1, sizeof(len), f) == sizeof(len) && std::fwrite(src.data(), 1, src.size(), f) == src.size() &&
              std::fwrite(cubin.data(), 1, cubin.size(), f) == cubin.size();
    ok = (std::fclose(f) == 0) && ok;
    if (!ok || std::rename(tmp.c_str(), path.c_str()) != 0) std::remove(tmp.c_str());
}

}  // namespace

bool jit_prepare_programs(int dtype, const std::vector<JitRequest> &reqs, std::string *err, double *compile_seconds,
                          int *compiled_modules) {
    if (compile_seconds) *compile_seconds = 0.0;
    if (compiled_modules) *compiled_modules = 0;
    const size_t es = dtype == QS_C64 ? 8 : 16, rs = dtype == QS_C64 ? 4 : 8;
    // every pass of every request, in order
    struct Item {
        const FusedProgram *prog;
        int pass;
        bool adjoint, batched;
        size_t req;
    };
    std::vector<Item> items;
    for (size_t ri = 0; ri < reqs.size(); ++ri) {
        const JitRequest &r = reqs[ri];
        r.out->assign(r.prog->passes.size(), JitPass{});
        for (size_t p = 0; p < r.prog->passes.size(); ++p) items.push_back({r.prog, (int)p, r.adjoint, r.batched, ri});
    }
    // one source per pass (kernel name fixed: the source text alone keys the cache); a pass
    // whose shape was seen before needs no source
    std::vector<std::string> srcs(items.size()), keys(items.size());
    std::vector<char> known(items.size(), 0);
    std::lock_guard<std::mutex> lock(g_mu);
    for (size_t i = 0; i < items.size(); ++i) {
        const Item &it = items[i];
        const FusedProgram &prog = *it.prog;
        keys[i] = shape_key(dtype, it.adjoint, it.batched, prog.passes[it.pass], prog.groups.data(), prog.gates.data());
        if (g_by_shape.count(keys[i])) {
            known[i] = 1;
            continue;
        }
        srcs[i] = jit_pass_source(dtype, it.adjoint, prog.passes[it.pass], prog.groups.data(), prog.gates.data(),
                                  "qs_pass", it.batched);
    }
    // passes whose source is not cached yet go into new modules (renamed kernels)
    std::vector<int> missing;
    std::unordered_map<std::string, int> first_of;
    for (size_t p = 0; p < srcs.size(); ++p) {
        if (known[p] || g_by_source.count(srcs[p])) continue;
        if (first_of.count(srcs[p])) continue;
        first_of[srcs[p]] = (int)p;
        missing.push_back((int)p);
    }
    const std::string dir = disk_cache_dir();
    if (!missing.empty() && !dir.empty()) {
        ::mkdir(dir.c_str(), 0755);  // if missing (one level; an error leaves the cache unused)
        // one module per kernel: loaded from the directory where present, else compiled
        // (concurrently) and written there
        auto t0 = std::chrono::steady_clock::now();
        std::vector<std::unique_ptr<Module>> mods(missing.size());
        std::vector<size_t> todo;
        for (size_t i = 0; i < missing.size(); ++i) {
            mods[i] = std::make_unique<Module>();
            mods[i]->source = srcs[missing[i]];
            mods[i]->names.push_back("qs_pass");
            if (!disk_load(disk_path(dir, mods[i]->source), mods[i]->source, &mods[i]->cubin)) todo.push_back(i);
        }
        std::vector<std::string> errs(mods.size());
        std::vector<char> ok(mods.size(), 1);
        unsigned hw = std::thread::hardware_concurrency();
        if (hw == 0) hw = 4;
        std::atomic<size_t> next{0};
        {
            std::vector<std::thread> th;
            for (unsigned w = 0; w < std::min<size_t>(hw, todo.size()); ++w)
                th.emplace_back([&] {
                    for (size_t q; (q = next.fetch_add(1)) < todo.size();) {
                        Module &m = *mods[todo[q]];
                        ok[todo[q]] = compile_cubin(m.source, &m.cubin, &errs[todo[q]]) ? 1 : 0;
                        if (ok[todo[q]]) disk_store(disk_path(dir, m.source), m.source, m.cubin);
                    }
                });
            for (auto &t : th) t.join();
        }
        for (size_t i = 0; i < mods.size(); ++i)
            if (!ok[i]) {
                *err = errs[i];
                return false;
            }
        for (size_t i = 0; i < mods.size(); ++i) {
            g_by_source[srcs[missing[i]]] = {(int)g_modules.size(), 0};
            g_modules.push_back(std::move(mods[i]));
        }
        if (compile_seconds)
            *compile_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        if (compiled_modules) *compiled_modules = (int)todo.size();
        missing.clear();
    }
    if (!missing.empty()) {
        auto t0 = std::chrono::steady_clock::now();
        // split the new kernels into modules compiled concurrently (NVRTC is thread-safe):
        // contiguous chunks of about equal source size, one per hardware thread at most
        size_t total = 0;
        for (int p : missing) total += srcs[p].size();
        unsigned hw = std::thread::hardware_concurrency();
        if (hw == 0) hw = 4;
        const size_t nmod = std::max<size_t>(1, std::min<size_t>({(size_t)hw, missing.size(), 32}));
        std::vector<std::unique_ptr<Module>> mods;
        std::vector<std::vector<int>> members;
        {
            size_t acc = 0, cur = 0;
            mods.push_back(std::make_unique<Module>());
            members.emplace_back();
            for (size_t i = 0; i < missing.size(); ++i) {
                const std::string &src = srcs[missing[i]];
                if (acc >= (cur + 1) * total / nmod && !members.back().empty() && cur + 1 < nmod) {
                    ++cur;
                    mods.push_back(std::make_unique<Module>());
                    members.emplace_back();
                }
                Module &m = *mods.back();
                const size_t idx = m.names.size();
                const std::string nm = "qs_pass_" + std::to_string(idx);
                std::string s2 = src;
                const size_t at = s2.find(" qs_pass(");
                s2.replace(at, 9, " " + nm + "(");
                m.source += "namespace m" + std::to_string(idx) + " {\n" + s2 + "}\n";
                m.names.push_back(nm);
                members.back().push_back(missing[i]);
                acc += src.size();
            }
        }
        // QS_JIT_DUMP=<directory>: write each compiled module's source there (diagnostics)
        if (const char *dir = std::getenv("QS_JIT_DUMP")) {
            if (*dir) {
                for (size_t i = 0; i < mods.size(); ++i) {
                    const std::string path =
                        std::string(dir) + "/qs_jit_module_" + std::to_string(g_modules.size() + i) + ".cu";
                    if (FILE *f = std::fopen(path.c_str(), "w")) {
                        std::fwrite(mods[i]->source.data(), 1, mods[i]->source.size(), f);
                        std::fclose(f);
                    }
                }
            }
        }
        std::vector<std::string> errs(mods.size());
        std::vector<char> ok(mods.size(), 0);
        {
            std::vector<std::thread> th;
            for (size_t i = 0; i < mods.size(); ++i)
                th.emplace_back([&, i] { ok[i] = compile_cubin(mods[i]->source, &mods[i]->cubin, &errs[i]) ? 1 : 0; });
            for (auto &t : th) t.join();
        }
        for (size_t i = 0; i < mods.size(); ++i)
            if (!ok[i]) {
                *err = errs[i];
                return false;
            }
        for (size_t i = 0; i < mods.size(); ++i) {
            const int mi = (int)g_modules.size();
            for (size_t j = 0; j < members[i].size(); ++j) g_by_source[srcs[members[i][j]]] = {mi, (int)j};
            g_modules.push_back(std::move(mods[i]));
        }
        if (compile_seconds)
            *compile_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        if (compiled_modules) *compiled_modules = (int)mods.size();
    }
    for (size_t i = 0; i < items.size(); ++i) {
        if (!known[i]) g_by_shape[keys[i]] = g_by_source.at(srcs[i]);
        const auto &mk = g_by_shape.at(keys[i]);
        const Item &it = items[i];
        const FusedProgram &prog = *it.prog;
        JitPass &j = (*reqs[it.req].out)[it.pass];
        j.entry = mk.first;
        j.kernel = mk.second;
        const TilePass &P = prog.passes[it.pass];
        const size_t T = size_t(1) << P.k;
        int npg = 0;  // batch: parameterised gates of the pass
        if (it.batched)
            for (int g = P.gate_begin; g < P.gate_begin + P.gate_count; ++g) npg += prog.gates[g].pkind != 0;
        const size_t NP = it.adjoint ? (size_t)std::max(1, it.batched ? npg : P.nparam) : 0;
        const bool db = jit_shape(dtype, it.adjoint, P.k).db;
        const size_t pm = it.batched ? (size_t)jit_batch_words(npg, it.adjoint) * (db ? 2 : 1) : 0;
        j.smem = (db ? 2 : 1) * (it.adjoint ? 2 : 1) * T * es +
                 (pm + 2 * NP * (kTileThreads / 32)) * rs;
        j.nparam_gates = npg;
        const size_t G = P.gate_count > 0 ? P.gate_count : 1;
        size_t bytes = G * 8 * rs;
        if (it.adjoint && !it.batched) bytes = ((bytes + 7) & ~size_t(7)) + NP * (sizeof(double) + sizeof(int));
        j.arg_bytes = (bytes + 15) & ~size_t(15);
        j.batched = it.batched;
    }
    return true;
}

bool jit_prepare_program(int dtype, bool adjoint, const FusedProgram &prog, std::vector<JitPass> *out,
                         std::string *err, double *compile_seconds, int *compiled_modules) {
    return jit_prepare_programs(dtype, {JitRequest{&prog, adjoint, false, out}}, err, compile_seconds, compiled_modules);
}

namespace {

// The kernel of a compiled pass on the current device: loaded on first use, its dynamic shared
// memory allowed, its resident blocks per SM looked up once.
cudaError_t jit_kernel(const JitPass &jp, cudaKernel_t *kern, int *occ) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    std::lock_guard<std::mutex> lock(g_mu);
    if (jp.entry < 0 || jp.entry >= (int)g_modules.size()) return cudaErrorInvalidValue;
    Module *m = g_modules[jp.entry].get();
    if (!m->lib) {
        cudaError_t e = cudaLibraryLoadData(&m->lib, m->cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0);
        if (e != cudaSuccess) return e;
        m->kernels.resize(m->names.size());
        for (size_t i = 0; i < m->names.size(); ++i) {
            e = cudaLibraryGetKernel(&m->kernels[i], m->lib, m->names[i].c_str());
            if (e != cudaSuccess) return e;
        }
    }
    *kern = m->kernels[jp.kernel];
    auto &ss = m->smem_set[dev];
    auto &oc = m->occ[dev];
    if (ss.size() < m->kernels.size()) {
        ss.resize(m->kernels.size(), 0);
        oc.resize(m->kernels.size(), 0);
    }
    if (jp.smem > 48 * 1024 && ss[jp.kernel] < jp.smem) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(*kern),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)jp.smem);
        if (e != cudaSuccess) return e;
        ss[jp.kernel] = jp.smem;
        oc[jp.kernel] = 0;
    }
    if (oc[jp.kernel] == 0) {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, reinterpret_cast<const void *>(*kern), kTileThreads,
                                                          jp.smem) != cudaSuccess ||
            v < 1) {
            cudaGetLastError();
            v = 1;
        }
        oc[jp.kernel] = v;
    }
    *occ = oc[jp.kernel];
    return cudaSuccess;
}

// The matrices of a pass's gates (state precision), 8 reals each: row-major complex; float32 real
// gates as {a, a, b, b, c, c, d, d} for the packed update; divided gates (real_forms) as
// {q, q, -q, -q, which, ...}. scale (may be null): per gate, the product divided out before it.
template <typename Real>
void put_matrices(const FusedProgram &prog, const TilePass &P, const std::vector<int> &form, unsigned char *dst,
                  std::vector<double> *scale) {
    const RegGate *g = prog.gates.data() + P.gate_begin;
    Real *out = reinterpret_cast<Real *>(dst);
    double pending = 1.0;
    for (int i = 0; i < P.gate_count; ++i, out += 8) {
        if (scale) (*scale)[i] = pending;
        const double *U = g[i].U;
        if (form[i]) {
            const double a = U[0], b = U[4];
            // (a Hadamard's entries are equal: dividing by b leaves two packed multiply-adds)
            const bool wide = std::fabs(b) > std::fabs(a) || (form[i] == 2 && std::fabs(b) == std::fabs(a));
            const double d = wide ? b : a, q = d != 0.0 ? (wide ? a : b) / d : 0.0;
            out[0] = out[1] = (Real)q;
            out[2] = out[3] = (Real)-q;
            out[4] = wide ? (Real)1 : (Real)0;
            out[5] = out[6] = out[7] = 0;
            pending *= d;
            continue;
        }
        const bool full = pending != 1.0 && divisible(g[i], false);
        for (int k = 0; k < 8; ++k) out[k] = (Real)(full ? U[k] * pending : U[k]);
        if (full) pending = 1.0;
        if (sizeof(Real) == 4 && g[i].op == OP_REAL)
            for (int k = 0; k < 8; k += 2) out[k + 1] = out[k];
    }
}

void put_matrices(int dtype, const FusedProgram &prog, const TilePass &P, const std::vector<int> &form, unsigned char *dst,
                  std::vector<double> *scale = nullptr) {
    if (dtype == QS_C64) put_matrices<float>(prog, P, form, dst, scale);
    else put_matrices<double>(prog, P, form, dst, scale);
}

}  // namespace

cudaError_t jit_load(const std::vector<JitPass> &passes) {
    for (const JitPass &jp : passes) {
        cudaKernel_t kern;
        int occ = 0;
        cudaError_t e = jit_kernel(jp, &kern, &occ);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_jit_pass(int dtype, const JitPass &jp, const FusedProgram &prog, int p, void *psi, void *lam,
                            double *part, size_t part_stride, cudaStream_t st) {
    cudaKernel_t kern;
    int occ = 1;
    cudaError_t e = jit_kernel(jp, &kern, &occ);
    if (e != cudaSuccess) return e;
    const TilePass &P = prog.passes[p];
    const bool adjoint = lam != nullptr;
    // parameter block: matrices (state precision), gradient slots
    std::vector<unsigned char> blk(jp.arg_bytes, 0);
    const int G = P.gate_count;
    const RegGate *g = prog.gates.data() + P.gate_begin;
    const size_t rs = dtype == QS_C64 ? 4 : 8;
    const size_t G1 = G > 0 ? G : 1;
    std::vector<double> scale(G);
    put_matrices(dtype, prog, P, real_forms(g, G, false), blk.data(), &scale);
    if (adjoint) {
        const size_t NP1 = P.nparam > 0 ? P.nparam : 1;
        double *f = reinterpret_cast<double *>(&blk[(G1 * 8 * rs + 7) & ~size_t(7)]);
        int *gs = reinterpret_cast<int *>(f + NP1);
        int j = 0;
        for (int i = 0; i < G; ++i)
            if (g[i].slot >= 0) {
                f[j] = scale[i] * scale[i];
                gs[j++] = P.param_gslot[g[i].slot];
            }
    }
    uint64_t cap = (uint64_t)device_sm_count() * occ;
    if (adjoint) cap = std::min<uint64_t>(cap, part_stride);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(P.ntiles, cap));
    unsigned long long stride = part_stride;
    void *dbg = debug_state_address();  // debug build only: the generated kernels take it last
    void *args_fwd[] = {&psi, blk.data(), &dbg};
    void *args_adj[] = {&psi, &lam, &part, &stride, blk.data(), &dbg};
    return cudaLaunchKernel(reinterpret_cast<const void *>(kern), dim3(grid), dim3(kTileThreads),
                            adjoint ? args_adj : args_fwd, jp.smem, st);
}

int jit_batch_words(int nparam_gates, bool adjoint) {
    return 8 * nparam_gates + (adjoint ? (nparam_gates + 3) & ~3 : 0);
}

void jit_batch_gates(const FusedProgram &prog, int p, bool adjoint, std::vector<BatchMatGate> *out) {
    const TilePass &P = prog.passes[p];
    const RegGate *g = prog.gates.data() + P.gate_begin;
    const std::vector<int> form = real_forms(g, P.gate_count, true);
    for (int i = 0; i < P.gate_count; ++i) {
        if (g[i].pkind == 0) continue;
        BatchMatGate d;
        d.pidx = g[i].pidx;
        d.kind = g[i].op == OP_REAL ? (form[i] ? BM_RY_DIVIDED : divisible(g[i], true) ? BM_RY_FULL : BM_RY_CONTROLLED)
                                    : (g[i].op == OP_SIDE ? BM_RZ_SIDE : BM_RZ);
        d.adjoint = adjoint;
        out->push_back(d);
    }
}

cudaError_t launch_jit_pass_batched(int dtype, const JitPass &jp, const FusedProgram &prog, int p, void *psi,
                                    void *lam, double *part, uint64_t stride, uint64_t nstates, const void *mats,
                                    cudaStream_t st) {
    if (!jp.batched) return cudaErrorInvalidValue;
    cudaKernel_t kern;
    int occ = 1;
    cudaError_t e = jit_kernel(jp, &kern, &occ);
    if (e != cudaSuccess) return e;
    const TilePass &P = prog.passes[p];
    std::vector<unsigned char> blk(jp.arg_bytes, 0);
    put_matrices(dtype, prog, P, std::vector<int>(P.gate_count, 0), blk.data());
    const uint64_t total = nstates * P.ntiles;
    const uint64_t cap = (uint64_t)device_sm_count() * occ;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(total, cap));
    unsigned long long stride_ = stride, nst = nstates;
    void *args[] = {&psi, &lam, &part, &stride_, &nst, const_cast<void **>(&mats), blk.data()};
    return cudaLaunchKernel(reinterpret_cast<const void *>(kern), dim3(grid), dim3(kTileThreads), args, jp.smem, st);
}

}  // namespace qs
