// Host check that no integer sum of the FP64 zone formulas leaves its 64 bits (fixed.cuh).
//
// Each formula is instantiated three times over a probe team, whose fluxes are given numbers instead of functions of the
// node states (which lets them take any signs):
//   Sym          a scalar that follows every integer as a linear functional of the values entered into a frame; each one
//                that meets a fraction, leaves or changes its frame is an operand, and its L1 norm must fit the frame;
//   double       the kernels' own integers, driven with the sign pattern of each operand and the largest mantissas;
//   long double  the same formulas in 80-bit arithmetic.
// Prints "name value bound" lines: the largest L1 norm over the frame's room, and the largest difference of the two
// arithmetics over the bound for a sum that has not wrapped.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>

struct Sym {
    int id;                            // an input's number, 0 for what has been computed
    Sym() : id(0) {}
    Sym(double) : id(0) {}
};
inline Sym operator+(Sym, Sym) { return {}; }
inline Sym operator-(Sym, Sym) { return {}; }
inline Sym operator*(Sym, Sym) { return {}; }
inline Sym operator/(Sym, Sym) { return {}; }
inline Sym operator-(Sym) { return {}; }
inline Sym& operator+=(Sym& a, Sym) { a.id = 0; return a; }
inline bool operator>(Sym, Sym) { return false; }
inline bool operator<(Sym, Sym) { return false; }
inline Sym sqrt(Sym) { return {}; }
inline Sym fmin(Sym, Sym) { return {}; }
inline Sym fmax(Sym, Sym) { return {}; }
inline Sym fabs(Sym) { return {}; }

#include "../paper_1006_2146_gb300/csrc/weno.cuh"
#include "../paper_1006_2146_gb300/csrc/step_inst.cuh"
using namespace ader;
typedef long double LD;

typedef std::map<int, double> Functional;
struct Operand {
    Functional c;
    double norm, room;
};
static std::vector<Operand> operands;
static int fresh = 0;
static void operand(const Functional& c, double room) {
    Operand o{c, 0.0, room};
    for (auto& x : c) o.norm += std::fabs(x.second);
    if (o.norm > 0) operands.push_back(o);
}

template <int LSH>
struct SymFix {
    Functional c;
};
template <int LSH>
SymFix<LSH> combine(const SymFix<LSH>& a, double k, const SymFix<LSH>& b, double l) {
    SymFix<LSH> r;
    for (auto& x : a.c) r.c[x.first] += k * x.second;
    for (auto& x : b.c) r.c[x.first] += l * x.second;
    return r;
}
template <int LSH> SymFix<LSH> operator+(const SymFix<LSH>& a, const SymFix<LSH>& b) { return combine(a, 1, b, 1); }
template <int LSH> SymFix<LSH> operator-(const SymFix<LSH>& a, const SymFix<LSH>& b) { return combine(a, 1, b, -1); }
template <int LSH> SymFix<LSH> operator-(const SymFix<LSH>& a) { return combine(a, -1, a, 0); }

namespace ader {
template <int NV, int LSH>
Vec<NV, SymFix<LSH>> operator*(double s, const Vec<NV, SymFix<LSH>>& a) {
    Vec<NV, SymFix<LSH>> r;
    for (int i = 0; i < NV; ++i) {
        if (std::fabs(s) != (double)(long long)std::fabs(s)) operand(a[i].c, std::ldexp(1.0, 10 - LSH));
        r[i] = combine(a[i], s, a[i], 0);
    }
    return r;
}
template <int NV, int LSH>
struct SymFrame {
    using S = SymFix<LSH>;
    void include(const Vec<NV, Sym>&) {}
    void close() {}
    Vec<NV, S> enter(const Vec<NV, Sym>& m) const {
        Vec<NV, S> r;
        for (int i = 0; i < NV; ++i) r[i].c[m[i].id ? m[i].id : --fresh] = 1.0;
        return r;
    }
    SymFrame extended(const Vec<NV, Sym>*, int) const { return {}; }
    void join(const SymFrame&) {}
    Vec<NV, S> from(const SymFrame&, const Vec<NV, S>& u) const {
        for (int i = 0; i < NV; ++i) operand(u[i].c, std::ldexp(1.0, 10 - LSH));
        return u;
    }
    Vec<NV, Sym> leave(const Vec<NV, S>& u) const {
        from(*this, u);
        return {};
    }
};
template <int LSH, int NV> struct FrameAt<LSH, NV, Sym> { using T = SymFrame<NV, LSH>; };
}  // namespace ader

// input n: a mode (n below 1000) or the j-th flux of the k-th exchange (1000 k + j)
static std::map<int, double> drive;
template <class R> R input(int n) {
    auto it = drive.find(n);
    return it == drive.end() ? R(0) : R(it->second);
}
template <> Sym input<Sym>(int n) {
    Sym s;
    s.id = n;
    return s;
}

template <int NV_, class R_>
struct ProbeTeam {
    static constexpr int NV = NV_, NL = 1;
    using R = R_;
    using V = Vec<1, R>;
    R gm1 = R(0.4), cx, cy, cz;
    int v = 0;
    mutable int calls = 0;
    ProbeTeam() : cx(0.99999), cy(0.99998), cz(0.99997) {}
    int var(int) const { return v; }
    bool lead() const { return false; }
    R zone_max(R x) const { return x; }
    bool any(bool x) const { return x; }
    static bool waits(bool) { return false; }
    void give(V* x, int n, int& at, R c, bool scaled) const {
        for (int k = 0; k < n; ++k) {
            x[k][0] = input<R>(++at);
            if (scaled) x[k][0] = c * x[k][0];
        }
    }
    template <int N, int A, bool SC> void fluxes(const V*, V* f, V* g, V* h) const {
        int at = 1000 * ++calls;
        give(f, N + A, at, cx, SC);
        give(g, N + A, at, cy, SC);
        give(h, N + A, at, cz, SC);
    }
    V axis_differences(const V*, R) const {
        int at = 1000 * ++calls;
        V r;
        give(&r, 1, at, R(1), false);
        return r;
    }
    template <int D, int N, int M> void face_fluxes(const V*, const V*, V* f, bool* ok) const {
        int at = 1000 * ++calls;
        give(f, N, at, R(1), false);
        for (int s = 0; s < M; ++s) ok[s] = true;
    }
    template <int N> void sources(const V*, const Src<R>&, V*) const {}
};

template <int ORDER, int FORM, class R>
static std::vector<R> predicted() {
    ProbeTeam<5, R> t;
    constexpr int L = ModeCount<ORDER>::L;
    Vec<1, R> m[L + 1];
    for (int k = 1; k <= L; ++k) m[k][0] = k <= ModeCount<ORDER>::LS ? input<R>(k) : R(0);
    PredCtl ctl{ORDER - 1, 0.0, 0, 0, false};
    if (FORM == FORM_MODAL) ZoneOps<ORDER>::template predict_modal<false>(t, m, ctl, nullptr, nullptr);
    else ZoneOps<ORDER>::template predict_nodal<false>(t, m, ctl, nullptr, nullptr);
    std::vector<R> out;
    for (int k = 1; k <= L; ++k) out.push_back(m[k][0]);
    return out;
}

template <int ORDER, int NV, class R>
static std::vector<R> faces() {
    ProbeTeam<NV, R> t;
    constexpr int L = ModeCount<ORDER>::L;
    std::vector<R> S3(6 * side_values(NV) + 6 * EDGE_STATE_VALUES, R(0)), out;
    StepArgs a{};
    a.grid = Grid{1, 1, 1, 1};
    a.solver = NV == 8 ? SOLVER_LINEARIZED : SOLVER_HLL;
    a.S3 = S3.data();
    Vec<1, R> m[L + 1];
    for (int k = 1; k <= L; ++k) m[k][0] = input<R>(k);
    for (t.v = NV == 8 ? 5 : 0; t.v < (NV == 8 ? 8 : 1); ++t.v) {
        t.calls = 0;
        FrameOf<ORDER, 1, R> fr;
        Vec<1, typename FrameOf<ORDER, 1, R>::S> s[L + 1];
        enter_frame<ORDER>(m, fr, s);
        store_faces_team<ORDER, 0>(t, a, 0, true, m[1], fr, s);
        store_faces_team<ORDER, 1>(t, a, 0, true, m[1], fr, s);
        store_faces_team<ORDER, 2>(t, a, 0, true, m[1], fr, s);
        out.insert(out.end(), S3.begin(), S3.end());
    }
    return out;
}

template <class F, class G, class H>
static void check(const char* name, F sym, G fix, H real) {
    operands.clear();
    sym();
    const std::vector<Operand> ops = operands;
    double worst = 0, diff = 0;
    for (const Operand& o : ops) {
        worst = std::fmax(worst, o.norm / o.room);
        // the operand's signs on the inputs it has; what it takes from earlier results has no number of its own
        drive.clear();
        for (auto& x : o.c)
            if (x.first > 0) drive[x.first] = x.second < 0 ? -(2.0 - std::ldexp(1.0, -52)) : 2.0 - std::ldexp(1.0, -52);
        if (drive.empty()) continue;
        const std::vector<double> a = fix();
        const std::vector<LD> b = real();
        for (size_t i = 0; i < a.size(); ++i) diff = std::fmax(diff, (double)std::fabs(a[i] - b[i]));
    }
    std::printf("%s_norm %.17g %.17g\n", name, worst, 1.0 - std::ldexp(1.0, -40));
    // a value of 2 enters with a unit of 2^-51 - LSH or less, a formula carries at most 2^9 of them and as many cut
    // products, and the iterations multiply by up to 2^5; a wrapped sum is off by 2^7 or more times a coefficient of
    // 2^-8 or more
    std::printf("%s_driven %.17g %.17g\n", name, diff, std::ldexp(1.0, -36));
}

template <int ORDER, int FORM>
static void predictor(const char* name) {
    check(name, [] { predicted<ORDER, FORM, Sym>(); }, [] { return predicted<ORDER, FORM, double>(); },
          [] { return predicted<ORDER, FORM, LD>(); });
}
template <int ORDER, int NV>
static void face(const char* name) {
    check(name, [] { faces<ORDER, NV, Sym>(); }, [] { return faces<ORDER, NV, double>(); },
          [] { return faces<ORDER, NV, LD>(); });
}

// the fourth-order WENO on every sign pattern of its six differences
static void weno() {
    double diff = 0;
    for (int s = 0; s < 64; ++s) {
        double a[7] = {0}, b, c, d;
        for (int k = 0; k < 6; ++k) a[k + 1] = a[k] + (s >> k & 1 ? -1.0 : 1.0) * (2.0 - std::ldexp(1.0, -49));
        LD al[7], bl, cl, dl;
        for (int k = 0; k < 7; ++k) al[k] = a[k];
        weno4(a, b, c, d);
        weno4(al, bl, cl, dl);
        diff = std::fmax(diff, (double)std::fmax(std::fabs(b - bl), std::fmax(std::fabs(c - cl), std::fabs(d - dl))));
    }
    std::printf("weno4_driven %.17g %.17g\n", diff, std::ldexp(1.0, -47));      // 2^5 roundings of values up to 2
}

int main() {
    predictor<3, FORM_MODAL>("modal3");
    predictor<3, FORM_NODAL>("nodal3");
    predictor<4, FORM_MODAL>("modal4");
    predictor<4, FORM_NODAL>("nodal4");
    face<2, 5>("faces2");
    face<3, 5>("faces3");
    face<4, 5>("faces4");
    face<2, 8>("mhd2");
    face<3, 8>("mhd3");
    face<4, 8>("mhd4");
    weno();
    return 0;
}
