// Step 3 over the classified cell records: A_i by Eq. (sainexclu) and the gradient entry of
// atom i, one warp per atom.
//
// Bound: instruction issue in the mixed form (atan2f, square roots and divisions on partly
// filled warps), the FP64 unit in the FP64 form, where one warp instruction occupies a
// sub-partition for 64 cycles however many of its lanes are active.  So each kind of work is
// first compacted into a list and then spread over the lanes, one term per lane:
//   * dihedral angles (and their gradient) of the tetrahedra of C, one lane per (tetrahedron,
//     open edge) pair - about 19 a globule atom; one lane per face walked them before, 5 to 8
//     one after another on about 7 lanes.  They pass through shared memory to the face's lane,
//     which adds them in the face's order (the mixed form's sums keep their rounding);
//   * exterior triangles, several lanes each.
// The lengths |q| of the plane vectors are taken once per plane, not once per term.
// Mixed form: 20k globule 137 -> 98 us, 5k 42 -> 33.5, 1M shell 5.5 -> 4.1 ms; its loop over the rounds
// and 18 blocks also fix how its float terms round (without the loop, at 14 - 16 blocks: 84 - 87 us at 20k,
// areas other by 2e-7).  FP64 form: 5k 717 -> 181 us.
#pragma once
#include "dsasa_kernels.cuh"
#include "dsasa_math.cuh"

namespace dsasa {

namespace {

// resident blocks (of 2 warps) per SM that the register budget is sized for
template <class R> struct TermBlocks { static constexpr int value = 18; };
template <> struct TermBlocks<double> { static constexpr int value = 10; };

template <class R, bool GRAD> struct alignas(16) TermSmem {
    R pq[64][4];                      // plane vector q and its length
    R dih[3 * 64][GRAD ? 4 : 1];      // by 3 t + k: (the gradient and) the angle, last
    R inv[sizeof(R) == 8 ? 64 : 1];   // 1 / |q| (FP64 form)
    int pg[64];
    uchar4 tv[64], ta[64];            // cell vertices (planes; w: kf), their neighbours (w: tf)
    uint8_t start[64], eflag[64], face[64];
    uint8_t item[3 * 64], tri[3 * 64 / 2 + 2];   // (t << 2) | k
};

// dihedral angle of (O, a, b, c) along (O, a), la = |a|
template <class R> __device__ __forceinline__ R dihedral_o(P3<R> a, R la, P3<R> b, P3<R> c) {
    const P3<R> mc = cross3(a, b), md = cross3(a, c);
    const R v6 = dot3(a, cross3(b, c));
    return ds_atan2(la * (v6 < (R)0 ? -v6 : v6), dot3(mc, md));
}

// One lane of an exterior triangle (i, a, b) in the FP64 form.  With u = p_a - p_i, w = p_b - p_i,
// the triple point x on the side of u x w satisfies x.x = R_i^2, x.u = b_u, x.w = b_w (b the bisector
// offsets); s is its height over the plane of the centres.  The angle along (i, a) of the tetrahedron
// (i, a, b, x) is also the half arc of circle (i, a) on both spheres (lens_grad), so the three owners'
// lens gradients with respect to p_i need the angles along (i, a) and (i, b) only:
//   d/dp_i = 2 s / |u x w| ((w_a R_a - w_i R_i) (w - (u.w)/(u.u) u) + (w_b R_b - w_i R_i) (u - (u.w)/(w.w) w))
//          + 2 theta_ia / |u| (w_i R_i (1 - b_u/(u.u)) + w_a R_a b_u/(u.u)) u + (the same for b),
// and S_iab^(i) = 2 pi R_i^2 - 2 R_i (b_u theta_ia / |u| + b_w theta_ib / |w|) - 2 R_i^2 theta_ix.
// The lens gradients one owner at a time and Eq. (trianglev) took 9 atan2 and about 40 divisions
// and square roots a triangle; this takes 3 and 2, one atan2 on each of 3 lanes (the lengths come from the table of planes).
// The three angles are taken from one computed x, by its cross products: the area is stationary in
// x (on a sphere, moving the corner where two arcs meet changes the area to second order), so the
// rounding of x cancels between them.  By Gram entries, with x.u, x.w and x.x at their exact
// values beside the rounded s, it did not: largest area error on two 13,007-atom RNAs 1.1e-12 A^2
// against long double, now 1.3e-13, as with a separate evaluation of each (1.2e-13); rms 3.2e-14 /
// 1.8e-14 / 1.9e-14.  It costs 260 -> 268 us a call of 5,000 atoms.
struct TriGram {
    P3<double> u, w, n;          // n = u x w
    double uu, ww, uw, bu, bw;   // Gram entries, bisector offsets
    double nn;                   // |n|^2
    double iu, iw, in;           // 1 / |u|, 1 / |w|, 1 / |n|
    double h;                    // s
    P3<double> x;                // the triple point
};
__device__ __forceinline__ TriGram tri_gram(P3<double> u, P3<double> w, double iu, double iw, double Ri, double Ra, double Rb) {
    TriGram g;
    g.u = u;
    g.w = w;
    g.n = cross3(u, w);
    g.uu = dot3(u, u);
    g.ww = dot3(w, w);
    g.uw = dot3(u, w);
    g.bu = 0.5 * (g.uu + (Ri - Ra) * (Ri + Ra));
    g.bw = 0.5 * (g.ww + (Ri - Rb) * (Ri + Rb));
    g.iu = iu;
    g.iw = iw;
    g.nn = dot3(g.n, g.n);
    g.in = rsqrt(g.nn);
    double in2 = g.in * g.in;
    in2 = fma(in2, fma(-g.nn, in2, 1.0), in2);   // 1 / |n|^2 to its last bit
    const P3<double> z = (cross3(w, g.n) * g.bu + cross3(g.n, u) * g.bw) * in2;   // the foot of x
    const double s2 = Ri * Ri - dot3(z, z);
    g.h = s2 > 0.0 ? sqrt(s2) : 0.0;
    g.x = z + g.n * (g.h * g.in);
    return g;
}

template <class R, bool GRAD>
__global__ void __launch_bounds__(WARPS_TERMS * 32, TermBlocks<R>::value) k_terms(AtomArgs A) {
    constexpr bool FFM = sizeof(R) == 4;
    __shared__ TermSmem<R, GRAD> smem_all[WARPS_TERMS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    TermSmem<R, GRAD>* S = &smem_all[wib];
    const bool EXPORT = !GRAD && A.rec != nullptr;   // (an export asks for no gradient)
    const unsigned lt = lanemask_lt();
    const R zero = (R)0;
    const double TWO_PI = 6.283185307179586476925;
    grid_dep_trigger();
    grid_dep_wait();
    for (int s = blockIdx.x * WARPS_TERMS + wib; s < A.n; s += gridDim.x * WARPS_TERMS) {
    const CellRecF* rec = (const CellRecF*)A.cells + s;

    // ---------------- the record: the header and the first half of every table in one memory
    // round trip (an atom has about 32 planes and 24 vertex slots), the second half if it is used
    const int i = DS_IDX(A.sidx[s], A.n, A.status);
    const int flag = rec->flag;
    const int4 hd = *reinterpret_cast<const int4*>(&rec->iK);   // iK, icl, nc, hw
    float4 rq[2];
    int rg[2];
    uint8_t rs[2], re[2], rkf[2], rtf[2];
    uchar4 rv[2], ra[2];
    auto load = [&](int h) {
        const int e = lane + 32 * h;
        if constexpr (FFM) rq[h] = *(const float4*)rec->pq[e];
        rg[h] = rec->pg[e];
        rs[h] = rec->start[e];
        re[h] = rec->eflag[e];
        rv[h] = rec->tv[e];
        ra[h] = rec->ta[e];
        rkf[h] = rec->kf[e];
        rtf[h] = rec->tf[e];
    };
    load(0);
    if (flag != CELL_OK) continue;   // the outputs of this atom are written
    const bool iK = hd.x != 0, icl = hd.y != 0;
    const int np = NG + hd.z, hw = hd.w;
    const bool two = np > 32 || hw > 32;
    if (two) load(1);
    const double Ri = A.R[i];
    const R Rr = (R)Ri;
    const float2 ri2 = A.Rhl[i];
    const double wi_w = A.w ? A.w[i] : 1.0;
    const R wif = (R)wi_w;
    int nf = 0;   // open exterior faces
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !two) break;
        const int e = lane + 32 * h;
        if (e >= np) re[h] = 0;
        if (e >= hw) {
            rv[h] = make_uchar4(NONE, NONE, NONE, 0);
            rkf[h] = rtf[h] = 0;
        }
        P3<R> q;
        if constexpr (FFM) q = {rq[h].x, rq[h].y, rq[h].z};
        else {
            const int g = DS_IDX(e < np ? max(rg[h], 0) : 0, A.n, A.status);
            const AtomD pk = load_atom(A.ad + g), pi = load_atom(A.ad + i);
            q = {pk.x - pi.x, pk.y - pi.y, pk.z - pi.z};
        }
        S->pq[e][0] = q.x;
        S->pq[e][1] = q.y;
        S->pq[e][2] = q.z;
        if constexpr (FFM) S->pq[e][3] = norm3(q);
        else {
            const R qq = dot3(q, q), iq = rsqrt(qq);
            R l = qq * iq;   // the length and its reciprocal, each corrected to its last bit
            l = fma((R)0.5 * iq, fma(-l, l, qq), l);
            S->pq[e][3] = l;
            S->inv[e] = fma(iq, fma(-l, iq, (R)1), iq);
        }
        S->pg[e] = rg[h];
        S->start[e] = rs[h];
        S->eflag[e] = re[h];
        S->tv[e] = make_uchar4(rv[h].x, rv[h].y, rv[h].z, rkf[h]);
        S->ta[e] = make_uchar4(ra[h].x, ra[h].y, ra[h].z, rtf[h]);
        const bool open = e >= NG && (re[h] & 3) == 1;
        const unsigned b = __ballot_sync(FULL, open);
        if (open) S->face[nf + __popc(b & lt)] = (uint8_t)e;
        nf += __popc(b);
    }
    __syncwarp();
    auto pos = [&](int e) -> P3<R> { return {S->pq[e & 63][0], S->pq[e & 63][1], S->pq[e & 63][2]}; };
    auto plen = [&](int e) -> R { return S->pq[e & 63][3]; };

    // ---------------- the lists of dihedral angles and of exterior triangles
    int nd = 0, nt = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !two) break;
        const int t = lane + 32 * h;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const bool want = rkf[h] == 1 && (S->eflag[tv_get(rv[h], k) & 63] & 3) == 1;
            const unsigned b = __ballot_sync(FULL, want);
            if (want) S->item[nd + __popc(b & lt)] = (uint8_t)((t << 2) | k);
            nd += __popc(b);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            bool want = (rtf[h] >> (4 + k)) & 1;   // processed by its canonical owner only
            if (want) want = !(rkf[h] == 1 && S->tv[tv_get(ra[h], k) & 63].w == 1);   // interior: coefficient 0
            const unsigned b = __ballot_sync(FULL, want);
            if (want) S->tri[nt + __popc(b & lt)] = (uint8_t)((t << 2) | k);
            nt += __popc(b);
        }
    }
    __syncwarp();

    // ---------------- dihedral angles of the tetrahedra of C along open edges (i, a), and d/dp_i
    for (int j = lane; j < nd; j += 32) {
        const int t = S->item[j] >> 2, k = S->item[j] & 3;
        const uchar4 v = S->tv[t];
        const int a = tv_get(v, k);
        const P3<R> pa = pos(a), pb = pos(tv_get(v, (k + 1) % 3)), pc = pos(tv_get(v, (k + 2) % 3));
        const R la = plen(a);
        R* d = S->dih[3 * t + k];
        if constexpr (!FFM) {
            // the angle and its gradient d/dp_i (dihedral_grad_s for a positive orientation) with one
            // division and the length from the table
            const P3<R> mc = cross3(pa, pb), md = cross3(pa, pc);
            const R v6 = dot3(mc, pc);
            d[GRAD ? 3 : 0] = atan2(la * fabs(v6), dot3(mc, md));
            if constexpr (GRAD) {
                const R mc2 = dot3(mc, mc), md2 = dot3(md, md), f = la / (mc2 * md2), i2 = S->inv[a] * S->inv[a];
                const R cb = f * md2 * ((R)1 - dot3(pb, pa) * i2), cd = f * mc2 * (dot3(pc, pa) * i2 - (R)1);
                d[0] = mc.x * cb + md.x * cd;
                d[1] = mc.y * cb + md.y * cd;
                d[2] = mc.z * cb + md.z * cd;
            }
            continue;
        }
        const R th = dihedral_o(pa, la, pb, pc);
        if constexpr (GRAD) {
            // (i, a, b, c) is positively oriented: (a, b, c) is counter-clockwise
            const P3<R> O = {zero, zero, zero};
            const P3<R> g = dihedral_grad_u_in(O, pa, pb, pc, (R)1);
            d[0] = g.x;
            d[1] = g.y;
            d[2] = g.z;
            d[3] = th;
        } else {
            d[0] = th;
        }
    }
    __syncwarp();

    // Vectors, angles and the gradient are evaluated in R (float in the mixed mode).  The area
    // terms are combined in a form where pi multiplies only quantities of the radii and
    // distances (pi, R_i and R_i^2 rounded to float would bias every term the same way, and the
    // terms cancel about 30-fold in A_i).  Mixed mode: the radius quantities (R, R^2, R_i -+ R_j,
    // 2 pi) enter as float pairs and the lane's terms are summed in float-float (no FP64
    // instruction per term); the per-atom constants 4 pi R_i^2 and c 2 pi R_i^2 are added once in
    // FP64 at the end.
    double area_acc = 0.0;
    GAcc<R> gacc;
    const FF Ri_ff = {ri2.x, ri2.y}, Ri2_ff = ff_mul(Ri_ff, Ri_ff);
    FF acc_ff = {0.f, 0.f};
    float cf_sum = 0.f;
    float vtx_const = 0.f;   // 2 when the vertex term is present: its 4 pi R_i^2 = 2 (2 pi R_i^2)
    const float TWO_PI_H = 6.28318548202514648f, TWO_PI_L = -1.74845553e-07f;   // 2 pi = H + L

    // ---------------- edges (i, a) of C that are not closed
    for (int j = lane; j < nf; j += 32) {
        const int a = S->face[j];
        R phi_sum = zero;
        P3<R> gsum = {zero, zero, zero};
        const int st = S->start[a] & 63;
        int t = st;
        for (int step = 0; step < 64; ++step) {
            const uchar4 v = S->tv[t];
            const int k = v.x == a ? 0 : (v.y == a ? 1 : 2);
            if (v.w == 1) {
                const R* d = S->dih[3 * t + k];
                if constexpr (GRAD) {
                    const Row4<R> x = load_row(d);
                    phi_sum += x.v[3];
                    gsum = gsum + P3<R>{x.v[0], x.v[1], x.v[2]};
                } else {
                    phi_sum += d[0];
                }
            }
            t = tv_get(S->ta[t], k) & 63;
            if (t == st) break;
        }
        // edge term of A_i (Eqs. phiedge, edge): - Phi_ia S_ia^(i) with
        // S_ia^(i) = 2 pi R_i h_i and Phi_ia = 1 - sum(theta) / 2 pi, i.e.
        // R_i h_i (sum(theta) - 2 pi); h_i = (R_i + R_a - d)(R_a - R_i + d) / 2d
        const P3<R> pa = pos(a);
        const int ga = DS_IDX(S->pg[a], A.n, A.status);
        const R dr = plen(a), inv2d = FFM ? (R)0.5 / dr : (R)0.5 * S->inv[FFM ? 0 : a];
        R Raf, dR2;
        if constexpr (FFM) {
            const float2 ra2 = A.Rhl[ga];
            const FF Ra = {ra2.x, ra2.y}, Sp = ff_add(Ri_ff, Ra), Dm = ff_sub(Ra, Ri_ff);
            const float hi = ((Sp.h - dr) + Sp.l) * ((Dm.h + dr) + Dm.l) * inv2d;
            acc_ff = ff_add(acc_ff, ff_mul_f(Ri_ff, hi * ((phi_sum - TWO_PI_H) - TWO_PI_L)));
            Raf = Ra.h;
            dR2 = ff_mul(ff_sub(Ri_ff, Ra), Sp).h;
        } else {
            const double Ra = A.R[ga];
            const double hi = ((Ri + Ra) - dr) * ((Ra - Ri) + dr) * inv2d;
            area_acc += Ri * hi * (phi_sum - TWO_PI);
            Raf = Ra;
            dR2 = (Ri - Ra) * (Ri + Ra);
        }
        if constexpr (GRAD) {
            const R waf = A.w ? (R)A.w[ga] : (R)1;
            const R ti = (dr * dr + dR2) * inv2d, ta = (dr * dr - dR2) * inv2d;
            const R phi = (R)1 - phi_sum * (R)(1.0 / TWO_PI);
            // vertex + edge parts of the dihedral derivatives around ia (Eq. inexclu)
            const R kap = -(wif * Rr * ti + waf * Raf * ta);
            // cap derivatives (Eq. edge): -Phi (2 pi / d)(w_i R_i t_a + w_a R_a t_i) u
            R cf;
            if constexpr (FFM) cf = -phi * (R)TWO_PI / (dr * dr) * (wif * Rr * ta + waf * Raf * ti);
            else cf = -phi * (R)TWO_PI * (S->inv[a] * S->inv[a]) * (wif * Rr * ta + waf * Raf * ti);
            gacc.add(kap * gsum.x + cf * pa.x, kap * gsum.y + cf * pa.y, kap * gsum.z + cf * pa.z);
        }
    }

    // ---------------- vertex term Omega_i 4 pi R_i^2 (Eq. vertex), Omega_i = 1 - sum of solid
    // angles / 4 pi (with the half solid angles h_T of its tetrahedra:
    // Omega_i 4 pi R_i^2 = 4 pi R_i^2 - 2 R_i^2 sum h_T)
    if (iK && !icl) {
        R om = zero;
#pragma unroll 1
        for (int h = 0; h < (two ? 2 : 1); ++h) {
            const uchar4 v = S->tv[lane + 32 * h];
            if (v.w == 1) {
                const P3<R> a = pos(v.x), b = pos(v.y), c = pos(v.z);
                const R la = plen(v.x), lb = plen(v.y), lc = plen(v.z);
                R num = dot3(a, cross3(b, c));
                num = num < (R)0 ? -num : num;
                const R den = la * lb * lc + dot3(a, b) * lc + dot3(a, c) * lb + dot3(b, c) * la;
                om += ds_atan2(num, den);
            }
        }
        if constexpr (FFM) {
            // - 2 R_i^2 (half solid angles) in float-float; the 4 pi R_i^2 is added once below
            acc_ff = ff_add(acc_ff, ff_mul_f(Ri2_ff, -2.f * om));
            vtx_const = 2.f;
        } else {
            // (lane 0 adds the 4 pi R_i^2; by itself it would round alike for every atom of a radius)
            area_acc += 2.0 * Ri * Ri * ((lane == 0 ? TWO_PI : 0.0) - om);
        }
    }

    // ---------------- exterior triangles: c_iab S_iab^(i) (Eq. trianglev) and the gradient of the
    // triangle terms of i, a and b (Eq. triangle) and of the dihedral (wing) terms that do not
    // cancel.  Mixed form: one lane per triangle for the area term, then three for the gradient
    // (lanes 30 and 31 idle), the lens gradients of the owners i, a and b; part 0 adds the wing
    // dihedral term when one tetrahedron of C holds the triangle
    if constexpr (FFM) {
        for (int j = lane; j < nt; j += 32) {
            const int t = S->tri[j] >> 2, k = S->tri[j] & 3;
            const uchar4 v = S->tv[t];
            const int a = tv_get(v, k), b = tv_get(v, (k + 1) % 3);
            const int nk = (v.w == 1) + (S->tv[tv_get(S->ta[t], k) & 63].w == 1);
            const float cff = 1.f - 0.5f * (float)nk;
            const int ga = DS_IDX(S->pg[a & 63], A.n, A.status), gb = DS_IDX(S->pg[b & 63], A.n, A.status);
            const float2 ra2 = A.Rhl[ga], rb2 = A.Rhl[gb];
            const FF Ra = {ra2.x, ra2.y}, Rb = {rb2.x, rb2.y};
            const FF x = tri_term_ff(pos(a), pos(b), Ri_ff, Ra, Rb, Ri2_ff, -1.f);
            acc_ff = ff_add(acc_ff, FF{cff * x.h, cff * x.l});
            cf_sum += cff;
        }
        if constexpr (GRAD)
        for (int j = lane < 30 ? lane : 3 * nt; j < 3 * nt; j += 30) {
            const int e = j / 3, part = j - 3 * e;
            const int t = S->tri[e] >> 2, k = S->tri[e] & 3;
            const uchar4 v = S->tv[t];
            const uint8_t a = tv_get(v, k), b = tv_get(v, (k + 1) % 3), cc = tv_get(v, (k + 2) % 3);
            const int t2 = tv_get(S->ta[t], k) & 63;
            const bool on_t = v.w == 1;
            const int nk = (int)on_t + (S->tv[t2].w == 1);
            const R cff = (R)1 - (R)0.5 * (R)nk;
            const P3<R> pa = pos(a), pb = pos(b);
            const int ga = DS_IDX(S->pg[a & 63], A.n, A.status), gb = DS_IDX(S->pg[b & 63], A.n, A.status);
            const float2 ra2 = A.Rhl[ga], rb2 = A.Rhl[gb];
            const FF Ra = {ra2.x, ra2.y}, Rb = {rb2.x, rb2.y};
            const R Raf = Ra.h, Rbf = Rb.h, dRab = ff_mul(ff_sub(Ra, Rb), ff_add(Ra, Rb)).h;
            if (GRAD && part < 3) {
                const P3<R> O = {zero, zero, zero};
                const R waf = A.w ? (R)A.w[ga] : (R)1, wbf = A.w ? (R)A.w[gb] : (R)1;
                // owner i: d/dp_i = -(g2 + g3); owner a: p_i is the second centre; owner b
                const P3<R> u = part == 0 ? pa : (part == 1 ? O - pa : O - pb);
                const P3<R> w = part == 0 ? pb : (part == 1 ? pb - pa : pa - pb);
                const R r0 = part == 0 ? Rr : (part == 1 ? Raf : Rbf);
                const R r1 = part == 0 ? Raf : Rr;
                const R r2 = part == 2 ? Raf : Rbf;
                P3x2f<R> lg = lens_grad_in(u, w, r0, r1, r2, (R)-1);
                if (lg.refine) {
                    // The lens gradient is linear in the height s_t of the triple points over
                    // the plane of the centres, whose float value (R^2 - |z|^2) errs by about
                    // 2^-24 R^2 / s_t: for the few lens gradients (about 0.4 %) whose s_t^2 is
                    // below 0.01 R^2 it is taken from the float64 coordinates (the same for the
                    // three owners: it depends on the three spheres only) and the gradient
                    // redone.  Each FP64 instruction occupies a GB300 sub-partition for 64
                    // cycles, so the FP64 work is kept that rare and short (Gram form).
                    const double px = A.xyz[3 * i], py = A.xyz[3 * i + 1], pz = A.xyz[3 * i + 2];
                    const P3<double> qa = {A.xyz[3 * ga] - px, A.xyz[3 * ga + 1] - py, A.xyz[3 * ga + 2] - pz};
                    const P3<double> qb = {A.xyz[3 * gb] - px, A.xyz[3 * gb + 1] - py, A.xyz[3 * gb + 2] - pz};
                    const float s2 = triple_height2_gram(qa, qb, Ri, A.R[ga], A.R[gb]);
                    lg = lens_grad_in(u, w, r0, r1, r2, (R)(s2 > 0.f ? sqrtf(s2) : 0.f));
                }
                const R f = cff * (part == 0 ? -wif : (part == 1 ? waf : wbf));
                R sx = f * (part == 0 ? lg.a.x + lg.b.x : lg.a.x);
                R sy = f * (part == 0 ? lg.a.y + lg.b.y : lg.a.y);
                R sz = f * (part == 0 ? lg.a.z + lg.b.z : lg.a.z);
                if (part == 0 && nk == 1) {
                    // the single tetrahedron of C on this triangle: (i, a, b, x); its
                    // orientation is + when it is the cell vertex t, - when it is t2
                    const uchar4 w2 = S->tv[t2];
                    const uint8_t xo = (w2.x != a && w2.x != b) ? w2.x : ((w2.y != a && w2.y != b) ? w2.y : w2.z);
                    const uint8_t x = on_t ? cc : xo;
                    const R dab = norm3(pb - pa), inv2 = (R)0.5 / dab;
                    const R tab = (dab * dab + dRab) * inv2, tba = (dab * dab - dRab) * inv2;
                    const R kap = -(waf * Raf * tab + wbf * Rbf * tba);
                    const P3<R> gc = dihedral_grad_c_in(pa, pb, O, pos(x), on_t ? (R)1 : (R)-1);
                    sx += kap * gc.x;
                    sy += kap * gc.y;
                    sz += kap * gc.z;
                }
                gacc.add(sx, sy, sz);
            }
        }
    } else {
        // FP64 form: three lanes per triangle, one angle each (lanes 30 and 31 idle)
        const int part = lane % 3;
        const double iRi = 1.0 / Ri;
        for (int j0 = 0; j0 < nt; j0 += 10) {
            const int j = j0 + lane / 3;
            const bool on = lane < 30 && j < nt;
            const int e = S->tri[on ? j : 0];
            const int t = e >> 2, k = e & 3;
            const uchar4 v = S->tv[t];
            const int a = tv_get(v, k), b = tv_get(v, (k + 1) % 3);
            const int t2 = tv_get(S->ta[t], k) & 63;
            const bool on_t = v.w == 1;
            const int nk = (int)on_t + (S->tv[t2].w == 1);
            const R cff = (R)1 - (R)0.5 * (R)nk;
            const P3<R> pa = pos(a), pb = pos(b);
            const int ga = DS_IDX(S->pg[a & 63], A.n, A.status), gb = DS_IDX(S->pg[b & 63], A.n, A.status);
            const double Ra = A.R[ga], Rb = A.R[gb];
            const double la = plen(a), lb = plen(b);
            const TriGram g = tri_gram(pa, pb, S->inv[a & 63], S->inv[b & 63], Ri, Ra, Rb);
            // this lane's angle: along (i, a), (i, b), (i, x) (|x| = R_i but for rounding: to second order)
            const P3<double> ax = part == 0 ? g.u : (part == 1 ? g.w : g.x);
            const P3<double> mc = cross3(ax, part == 0 ? g.w : g.u), md = cross3(ax, part == 2 ? g.w : g.x);
            const double le = part == 0 ? la : (part == 1 ? lb : 0.5 * (Ri + dot3(ax, ax) * iRi));
            const double num = le * fabs(dot3(mc, part == 2 ? g.w : g.x)), den = dot3(mc, md);
            const double th = atan2(num, den);
            if (on) {
                area_acc += cff * (part == 0 ? -2.0 * Ri * (g.bu * g.iu) * th
                                             : (part == 1 ? -2.0 * Ri * (g.bw * g.iw) * th
                                                          : Ri * Ri * (TWO_PI - 2.0 * th)));
                if constexpr (GRAD) {
                    const double waf = A.w ? A.w[ga] : 1.0, wbf = A.w ? A.w[gb] : 1.0;
                    const double wRi = wif * Ri, wRa = waf * Ra, wRb = wbf * Rb;
                    const double iuu = g.iu * g.iu, iww = g.iw * g.iw;
                    // lane 0: theta_ia, lane 1: theta_ib, lane 2: the height s and the wing
                    double cu = 0.0, cw = 0.0, cn = 0.0;
                    if (part == 0) {
                        const double f = g.bu * iuu;
                        cu = cff * 2.0 * th * g.iu * (wRi * (1.0 - f) + wRa * f);
                    } else if (part == 1) {
                        const double f = g.bw * iww;
                        cw = cff * 2.0 * th * g.iw * (wRi * (1.0 - f) + wRb * f);
                    } else {
                        const double f = cff * 2.0 * g.h * g.in, fa = f * (wRa - wRi), fb = f * (wRb - wRi);
                        cu = fb - fa * g.uw * iuu;
                        cw = fa - fb * g.uw * iww;
                        if (nk == 1) {
                            // the single tetrahedron of C on this triangle, positively oriented
                            // when it is the cell vertex t: the gradient of its dihedral angle
                            // along (a, b) is -+ |p_b - p_a| n / |n|^2, its factor
                            // -(w_a R_a t_ab + w_b R_b t_ba)
                            const double dab2 = dot3(pb - pa, pb - pa), dRab = (Ra - Rb) * (Ra + Rb);
                            cn = (on_t ? 0.5 : -0.5) * (wRa * (dab2 + dRab) + wRb * (dab2 - dRab)) * (g.in * g.in);
                        }
                    }
                    gacc.add(cu * g.u.x + cw * g.w.x + cn * g.n.x, cu * g.u.y + cw * g.w.y + cn * g.n.y,
                             cu * g.u.z + cw * g.w.z + cn * g.n.z);
                }
            }
        }
    }

    double gx = 0.0, gy = 0.0, gz = 0.0;
    if constexpr (FFM) {
        // one float-float warp sum of every lane's terms (the same order on every run; lane 0's
        // value is used), then the per-atom constants (2 + c) 2 pi R_i^2 in FP64
        FF tot = acc_ff;
        for (int o = 16; o > 0; o >>= 1)
            tot = ff_add(tot, FF{__shfl_xor_sync(FULL, tot.h, o), __shfl_xor_sync(FULL, tot.l, o)});
        for (int o = 16; o > 0; o >>= 1) cf_sum += __shfl_xor_sync(FULL, cf_sum, o);
        area_acc = ff_to_double(tot) + ((double)cf_sum + (double)vtx_const) * TWO_PI * Ri * Ri;
    } else {
        // the four sums together: lanes 8 k .. 8 k + 7 end with sum k (6 FP64 additions instead of 20)
        const bool up = lane & 16, odd = lane & 8;
        double s0 = up ? gacc.y : area_acc, s1 = up ? gacc.z : gacc.x;
        const double o0 = up ? area_acc : gacc.y, o1 = up ? gacc.x : gacc.z;
        s0 += __shfl_xor_sync(FULL, o0, 16);
        s1 += __shfl_xor_sync(FULL, o1, 16);
        double t0 = odd ? s1 : s0;
        const double t1 = odd ? s0 : s1;
        t0 += __shfl_xor_sync(FULL, t1, 8);
        for (int o = 4; o > 0; o >>= 1) t0 += __shfl_xor_sync(FULL, t0, o);
        area_acc = t0;   // (lane 0)
        gx = __shfl_sync(FULL, t0, 8);
        gy = __shfl_sync(FULL, t0, 16);
        gz = __shfl_sync(FULL, t0, 24);
    }
    if constexpr (GRAD && FFM) gacc.reduce(gx, gy, gz);
    if (lane == 0) {
        A.areas[i] = iK ? area_acc : 0.0;
        if (GRAD && A.grad) {
            A.grad[3 * i] = iK ? gx : 0.0;
            A.grad[3 * i + 1] = iK ? gy : 0.0;
            A.grad[3 * i + 2] = iK ? gz : 0.0;
        }
        if (A.mol_done) molecule_count(A, i);
    }

    // ---------------- optional export of the simplices of C containing i
    if (EXPORT) {
        if (lane == 0 && iK) export_simplex(A, i, i, -1, -1, -1);
        for (int a = NG + lane; a < np; a += 32)
            if (S->eflag[a] & 1) export_simplex(A, i, i, S->pg[a], -1, -1);
        for (int h = 0; h < (two ? 2 : 1); ++h) {
            const int t = lane + 32 * h;
            const uchar4 v = S->tv[t];
            if (v.x == NONE) continue;
            if (v.w == 1) export_simplex(A, i, i, S->pg[v.x], S->pg[v.y], S->pg[v.z]);
            for (int k = 0; k < 3; ++k)
                if ((S->ta[t].w >> (4 + k)) & 1)
                    export_simplex(A, i, i, S->pg[tv_get(v, k)], S->pg[tv_get(v, (k + 1) % 3)], -1);
        }
    }
    __syncwarp();
    }
}

}  // namespace

}  // namespace dsasa
