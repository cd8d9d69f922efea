// whg_wide.cuh -- the step for small ensembles: four lanes per planet.
//
// An FP64 or integer warp instruction takes its pipe the same time whatever
// the number of active lanes, and where an ensemble leaves most
// sub-partitions idle or with one warp, a step's time is the number of
// instructions on one warp's path.  Here every planet has four lanes ("roles"),
// so a warp holds a quarter of the systems, and what is one instruction per
// coordinate, scalar product or pair distance in step_body becomes one
// instruction altogether: role c < 3 keeps coordinate c, roles 0..2 form one
// scalar product each, role k - 1 evaluates the pairs at lane distance k.
// (The solver of Kepler's equation is one chain; all roles run it alike.)
// 14 FP64 instructions per warp and step instead of 41, one pair round
// instead of L/2.  Every sum keeps step_body's order: the same bits.
//
// Measured, us per step, step_body's / this kernel: one 8-planet system 3.84 /
// 2.18, 608 4.08 / 2.21, ten 2-planet systems 2.70 / 1.85, 100 test particles
// 2.08 / 1.55; whg_kernels_common.cu has where it stops paying.  168 registers:
// three warps per sub-partition (with 174, two; 1500 systems 3.58 against 5.60).
//
// Lanes: Group<L>'s blocks of L lanes in fours; block 4 j + r is role r of the
// warp's system j.  State is read from and written to the usual layout.
#pragma once

#include "whg_device.cuh"

namespace whg {

template <int L>
struct WideGroup : Group<L> {
    static constexpr int SYSTEMS = Group<L>::SPW / 4;     // systems per warp
    int r, c;                                             // role; coordinate kept (role 3 doubles z)
    bool in_system;
    __device__ __forceinline__ WideGroup()
    {
        r = this->slot & 3;
        c = r < 2 ? r : 2;
        in_system = this->in_group && (this->slot >> 2) < SYSTEMS;
    }
    // lane of planet (p + k) mod L in role j
    __device__ __forceinline__ int lane_of(int j, int k) const
    {
        int q = this->p + k;
        q = q >= L ? q - L : (q < 0 ? q + L : q);
        return in_system ? this->base + (j - r) * L + q : this->lane;
    }
    // all lanes of the system
    __device__ __forceinline__ unsigned system_mask() const
    {
        constexpr unsigned ones = 4 * L >= 32 ? WHG_FULL_MASK : (1u << (4 * L & 31)) - 1u;
        return in_system ? ones << ((this->slot >> 2) * 4 * L & 31) : 1u << this->lane;
    }
    template <typename T>
    __device__ __forceinline__ T mine(T x, T y, T z) const { return c == 0 ? x : (c == 1 ? y : z); }
    // the vector whose coordinates the roles keep
    template <typename T>
    __device__ __forceinline__ void whole(T v, T& x, T& y, T& z) const
    {
        x = __shfl_sync(WHG_FULL_MASK, v, lane_of(0, 0));
        y = __shfl_sync(WHG_FULL_MASK, v, lane_of(1, 0));
        z = __shfl_sync(WHG_FULL_MASK, v, lane_of(2, 0));
    }
};

// mass_sum's component of this lane's coordinate: the same products and sums.
template <int L>
__device__ __forceinline__ double wide_mass_sum(const WideGroup<L>& g, double m, double x)
{
    if (L == 4 || L == 8) {
        constexpr int H = L / 2;
        const double xq = __shfl_xor_sync(WHG_FULL_MASK, x, H), mq = __shfl_xor_sync(WHG_FULL_MASK, m, H);
        const bool own = ((g.p & H) == 0) == (g.c < 2);   // the lane whose product mass_sum keeps in the FMA
        double k = fma(own ? m : mq, own ? x : xq, (own ? mq : m) * (own ? xq : x));
        k += __shfl_xor_sync(WHG_FULL_MASK, k, H / 2);
        if (L == 8) k += __shfl_xor_sync(WHG_FULL_MASK, k, 1);
        return k;
    }
    return group_sum<L>(g, __dmul_rn(m, x));
}

// sum_floats of this lane's coordinate.
template <int L>
__device__ __forceinline__ float wide_sum_float(const WideGroup<L>& g, float x)
{
    if (L == 1) return x;
    if (L == 4 || L == 8) {
#pragma unroll
        for (int o = L / 2; o; o >>= 1) x = pairs::add(x, __shfl_xor_sync(WHG_FULL_MASK, x, o));
        return x;
    }
    float s = 0.0f;
#pragma unroll
    for (int j = 0; j < L; ++j) s = pairs::add(s, __shfl_sync(WHG_FULL_MASK, x, g.in_group ? g.base + j : g.lane));
    return s;
}

// sum_pairs of this lane's coordinate.
template <int L>
__device__ __forceinline__ pairs::Pair wide_sum_pair(const WideGroup<L>& g, pairs::Pair x)
{
    if (L == 1) return x;
    if (L == 4 || L == 8) {
#pragma unroll
        for (int o = L / 2; o; o >>= 1) x = add_xor<L>(x, x, o);
        return x;
    }
    pairs::Pair s = {0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < L; ++j) s = pairs::sum(s, shfl_pair<L>(x, g.in_group ? g.base + j : g.lane));
    return s;
}

// interact_pairs on kept coordinates (q, v).  hmk: hm of the partner at the
// role's distance.
template <int L, int GRM>
__device__ __forceinline__ bool wide_interact(const WideGroup<L>& g, const Masses<L>& c, const pairs::Pair& hmk,
                                              double& q, double& v, const double* thr2, bool hill, bool& close)
{
    const double P = wide_mass_sum<L>(g, c.m, v);
    q = fma(c.merged ? 2.0 * c.jc : c.jc, P, q);
    bool ok = true;
    if (L > 1 || GRM != 0) {
        const fixed::u64 bq = fixed::bits_of(q);
        const int e = fixed::exponent_of(bq);
        unsigned ex, ey, ez;
        g.whole(((unsigned)e << 16) | (unsigned)fixed::exponent_of(fixed::bits_of(v)), ex, ey, ez);
        const unsigned top = __vmaxu2(ex, __vmaxu2(ey, ez));
        const int ev = (int)(top & 0xffffu);
        const int eq = group_max<L>(g, c.real ? (int)(top >> 16) : 0);
        const int K2 = 2 * (1040 - eq);
        const int el = ev - 1023 - K2;
        ok = (unsigned)(eq - 1007) <= 56u && (unsigned)(el + 60) <= 120u;
        const float vl = fixed::bits_to_f32((unsigned)(127 + el) << 23);
        const pairs::Coord C = pairs::chunks(c.real ? fixed::to_fixed(bq, 5 + eq - e)
                                                    : (g.c == 0 ? (long long)(32 + g.p) << 54 : 0ll));
        pairs::Coord X, Y, Z;
        g.whole(C.c2, X.c2, Y.c2, Z.c2);
        g.whole(C.c1, X.c1, Y.c1, Z.c1);
        g.whole(C.c0, X.c0, Y.c0, Z.c0);
        pairs::Pair a = {0.0f, 0.0f};
        auto accept = [](const pairs::Separation& s, float w, float scale) {
            return fmaxf(pairs::mul(w, pairs::mul(s.r2, s.y1)), pairs::mul(w, 256.0f)) <= pairs::mul(scale, 1.0f / 1024.0f);
        };
        auto gr_kick = [&]() {                           // its terms before those of the pairs, as interact_pairs has them
            if (GRM == 0) return;
            const pairs::Pair ox = pairs::own(X), oy = pairs::own(Y), oz = pairs::own(Z);
            const pairs::Separation s = pairs::separation(ox, oy, oz);
            const float sc = fixed::bits_to_f32((unsigned)(127 + 1040 - eq) << 23);
            pairs::Pair k;
            k.h = pairs::mul(c.kgp.h, sc);
            k.l = pairs::mul(c.kgp.l, sc);
            const pairs::Pair w = pairs::product(k, pairs::inverse_fourth(s));
            const float vg = gr_scale(vl, (int)(top >> 16), c.jm, K2);
            ok = ok & accept(s, -w.h, GRM == 1 ? vg : vl);
            pairs::Pair o;
            o.h = g.mine(ox.h, oy.h, oz.h);
            o.l = g.mine(ox.l, oy.l, oz.l);
            pairs::Pair f = pairs::product(w, o);
            if (GRM == 2) {
                const pairs::Pair b = wide_sum_pair<L>(g, pairs::product(c.mrp, f));
                pairs::accumulate(f, -b.h, -b.l);
                ok = ok & (fabsf(f.h) <= pairs::mul(vg, 1.0f / 1024.0f));
            }
            pairs::accumulate(a, f.h, f.l);
            const float p = wide_sum_float<L>(g, pairs::mul(c.mf, f.h));
            q = fma(c.jc, P + pairs::widen(p, K2), q);
        };
        if (L == 1) gr_kick();
        if (L > 1) {
            const int k = 2 * (g.r + 1) <= L ? g.r + 1 : 1;      // this role's distance (roles beyond L/2 idle along)
            auto at = [&](const pairs::Coord& x, int j) {
                const int to = g.lane_of(j, k);
                pairs::Coord y;
                y.c2 = __shfl_sync(WHG_FULL_MASK, x.c2, to);
                y.c1 = __shfl_sync(WHG_FULL_MASK, x.c1, to);
                y.c0 = __shfl_sync(WHG_FULL_MASK, x.c0, to);
                return y;
            };
            const pairs::Coord JX = at(C, 0), JY = at(C, 1), JZ = at(C, 2);
            const pairs::Separation s = pairs::separation(pairs::difference(JX, X), pairs::difference(JY, Y),
                                                          pairs::difference(JZ, Z));
            const pairs::Pair r3 = pairs::inverse_cube(s);
            const pairs::Pair wj = pairs::product(hmk, r3), wi = pairs::product(c.hmp, r3);
            const float vj = __shfl_sync(WHG_FULL_MASK, vl, g.lane_of(g.r, k));
            const bool fit = accept(s, wj.h, vl) & ((2 * k == L) | accept(s, wi.h, vj));
            const pairs::Pair fx = pairs::product(wj, s.x), fy = pairs::product(wj, s.y), fz = pairs::product(wj, s.z);
            const pairs::Pair gx = pairs::product(wi, s.x), gy = pairs::product(wi, s.y), gz = pairs::product(wi, s.z);
            const bool on = (g.r == k - 1) & ((c.pairs_on >> k) & 1u);
            ok = ok & (fit | !on);
            if (hill) {
                const double r2 = pairs::widen(s.r2, -K2);       // by the leading part, where that decides
                const double t2 = k == 1 ? thr2[0] : (k == 2 ? thr2[1] : (k == 3 ? thr2[2] : thr2[3]));
                const long long t = __double_as_longlong(t2), b = __double_as_longlong(r2);
                if (on && b - (1LL << 32) < t) close |= __double_as_longlong(r2 + pairs::widen(s.r2l, -K2)) < t;
            }
            auto from = [&](float x, float y, float z, int lane) {
                const float sx = __shfl_sync(WHG_FULL_MASK, x, lane), sy = __shfl_sync(WHG_FULL_MASK, y, lane),
                            sz = __shfl_sync(WHG_FULL_MASK, z, lane);
                return g.mine(sx, sy, sz);
            };
            gr_kick();
#pragma unroll
            for (int d = 1; 2 * d <= L; ++d) {                   // in step_body's order
                const int own = g.lane_of(d - 1, 0);
                const float h = from(fx.h, fy.h, fz.h, own), l = from(fx.l, fy.l, fz.l, own);
                pairs::accumulate(a, h, l);
                if (2 * d < L) {
                    const int back = g.lane_of(d - 1, -d);
                    const float bh = from(gx.h, gy.h, gz.h, back), bl = from(gx.l, gy.l, gz.l, back);
                    pairs::accumulate(a, -bh, -bl);
                }
            }
        }
        v += pairs::widen(a.h, K2) + pairs::widen(a.l, K2);
    }
    if (GRM == 0 && !c.merged) q = fma(c.jc, P, q);
    return ok;
}

// step_body for the systems of wide warp w of bucket b (first: its first wide
// warp).
template <int L, int NT, int GRM>
__device__ __forceinline__ void wide_body(const WhgState& st, const WhgBuckets& bk, int b, int w, int first,
                                          long long nsteps)
{
    const WideGroup<L> g;
    const int local = (w - first) * WideGroup<L>::SYSTEMS + (g.slot >> 2);
    const bool has = g.in_system && local < bk.sys0[b + 1] - bk.sys0[b];
    const int s = has ? bk.sys0[b] + local : 0;
    const size_t lane = has ? (size_t)(bk.warp0[b] + local / Group<L>::SPW) * 32 + (size_t)(local % Group<L>::SPW) * L + g.p : 0;
    WHG_CHECK(st, (long long)lane < st.nl, WHG_BOUND_LANE);
    WHG_CHECK(st, !has || (s >= 0 && s < st.S), WHG_BOUND_SYSTEM);
    const double m = has ? st.m[lane] : 0.0;
    double qx = has ? st.qx[lane] : parked_x(g.p), qy = has ? st.qy[lane] : 0.0, qz = has ? st.qz[lane] : 0.0;
    double vx = has ? st.vx[lane] : 0.0, vy = has ? st.vy[lane] : 0.0, vz = has ? st.vz[lane] : 0.0;
    const double mu = has ? st.m0[s] : 1.0;
    const double dt = has ? st.dt[s] : 1.0e-3;
    const int npl = has ? st.nplan[s] : 0;
    int status = has ? st.status[s] : 0;
    const long long nstep0 = has ? st.nstep[s] : 0;
    const double rej2 = has ? st.rej2[s] : 0.0;
    const bool real = has && g.p < npl;
    bool alive = has && status == 0;
    const Masses<L> mc = masses_of<L, GRM>(g, real, m, mu, dt, st.c_light, GRM == 0 && st.merge, false);
    pairs::Pair hmk = mc.hmj[0];
#pragma unroll
    for (int d = 2; 2 * d <= L; ++d)
        if (g.r == d - 1) hmk = mc.hmj[d - 1];
    const bool hill = st.hill > 0.0;
    double thr2[4] = {0.0, 0.0, 0.0, 0.0};
    if (hill) {
        const double a = has ? st.a0[lane] : 0.0;
#pragma unroll
        for (int k = 1; 2 * k <= L; ++k) {
            const int to = g.at(k);
            const double mj = __shfl_sync(WHG_FULL_MASK, m, to);
            const double aj = __shfl_sync(WHG_FULL_MASK, a, to);
            const double rh = st.hill * cbrt((m + mj) / (3.0 * mu)) * 0.5 * (a + aj);
            thr2[k - 1] = rh * rh;
        }
    }
    const unsigned gmask = g.system_mask();
    long long done = 0;
    for (long long k = 0; k < nsteps; ++k) {
        if (!__any_sync(WHG_FULL_MASK, alive)) break;        // whole warp frozen
        double q = g.mine(qx, qy, qz), v = g.mine(vx, vy, vz);
        const double sq = q, sv = v;
        const double hK = (nstep0 + done == 0) ? 0.5 * dt : dt;
        // r0^2, Q.v and v^2, one per role
        const bool av = g.r == 2, bv = g.r == 1 || g.r == 2;
        const double s1 = fma(av ? vx : qx, bv ? vx : qx, fma(av ? vy : qy, bv ? vy : qy, (av ? vz : qz) * (bv ? vz : qz)));
        double r0sq, eta0, v2;
        g.whole(s1, r0sq, eta0, v2);
        const bool far = __double_as_longlong(r0sq) > __double_as_longlong(rej2);
        fixed::Solution o;
        bool bound = fixed::solve<NT, false>(mu, hK, r0sq, eta0, v2, o);
        if (bound) {
            const double nq = fma(-o.fm1n, q, fma(o.g, v, q));
            v = fma(-o.fdn, q, fma(-o.gdm1n, v, v));
            q = nq;
        } else if (alive) {
            const GeneralDrift<false> r = kepler_general_call<NT, false>(mu, hK, r0sq, eta0, v2, qx, qy, qz, vx, vy, vz);
            q = g.mine(r.qx, r.qy, r.qz);
            v = g.mine(r.vx, r.vy, r.vz);
            bound = r.bound;
        }
        bool close = false;
        const double dq = q, dv = v;
        const bool ok = wide_interact<L, GRM>(g, mc, hmk, q, v, thr2, hill, close);
        const unsigned redo = __ballot_sync(WHG_FULL_MASK, real && alive && !ok);
        if (redo) {                                          // every role redoes the whole system
            double x, y, z, ux, uy, uz;
            g.whole(dq, x, y, z);
            g.whole(dv, ux, uy, uz);
            SubStep t{mc.m, mc.hm, mc.mrat, mc.jc, mc.kgr, x, y, z, ux, uy, uz, {0.0, 0.0, 0.0},
                      {thr2[0], thr2[1], thr2[2], thr2[3]}, false, mc.merged, false};
            interact_general<L, GRM>(&t);
            if (redo & gmask) {
                q = g.mine(t.qx, t.qy, t.qz);
                v = g.mine(t.vx, t.vy, t.vz);
                close = t.close;
            }
        }
        const bool fin = is_finite(q) & is_finite(v);
        const unsigned bad_h = __ballot_sync(WHG_FULL_MASK, real && !bound) & gmask;
        const unsigned bad_n = __ballot_sync(WHG_FULL_MASK, real && !fin) & gmask;
        const unsigned bad_c = __ballot_sync(WHG_FULL_MASK, real && close) & gmask;
        const unsigned bad_e = __ballot_sync(WHG_FULL_MASK, real && far) & gmask;
        const bool good = (bad_h | bad_n | bad_c | bad_e) == 0u;
        if (!(alive && real && good)) {                      // roll back: no planet, frozen, failed
            q = sq;
            v = sv;
        }
        if (alive && !good) {
            status |= (bad_n ? WHG_STATUS_NONFINITE : 0) | (bad_h ? WHG_STATUS_HYPERBOLIC : 0) |
                      (bad_c ? WHG_STATUS_CLOSE_ENCOUNTER : 0) | (bad_e ? WHG_STATUS_EJECTED : 0);
            alive = false;
        }
        done += alive ? 1 : 0;
        g.whole(q, qx, qy, qz);
        g.whole(v, vx, vy, vz);
    }
    if (real && g.r == 0) {
        st.qx[lane] = qx; st.qy[lane] = qy; st.qz[lane] = qz;
        st.vx[lane] = vx; st.vy[lane] = vy; st.vz[lane] = vz;
    }
    if (has && g.p == 0 && g.r == 0) {
        st.status[s] = status;
        st.nstep[s] = nstep0 + done;
    }
}

template <int NT, int GRM>
__global__ void __maxnreg__(168) k_step_wide(WhgState st, WhgBuckets bk, long long n)
{
    const int w = warp_index();
    int first = 0, b = 0;
    for (; b < bk.nb; ++b) {                                 // the wide warps of the buckets, one after another
        const int here = whg_wide_warps_of(bk, b);
        if (w < first + here) break;
        first += here;
    }
    if (b >= bk.nb) return;                                  // whole warps beyond the last bucket
    WHG_DISPATCH_L(bk.L[b], (wide_body<L_, NT, GRM>(st, bk, b, w, first, n)))
}

}  // namespace whg
