// Step 2: which simplices of a cell that contain atom i are in the dual complex C.
//
// Bound: instruction issue and the instruction cache (the predicates are long straight code).
// The tests are spread over the lanes, each predicate in one copy of its code:
//   * tetrahedra: one lane per cell vertex;
//   * triangles: the cell edges without a tetrahedron of C (about a third of 36) are compacted
//     into a list, one lane each, where one lane per vertex tried its three edges one after
//     another before;
//   * edges: no face is walked.  The vertices mark their faces (present, not closed, a triangle
//     of C on it), and "the orthocentre of face a lies inside its polygon" is one test per
//     directed cell edge (a, b), again compacted.
// A test that its filter leaves open is collected and resolved out of line with exact predicates.
// 20,003-atom globule 90 -> 53 us, 1,000,000-atom shell 3.80 -> 1.76 ms.
#pragma once
#include "dsasa_kernels.cuh"
#include "dsasa_math.cuh"

namespace dsasa {

namespace {

// resident blocks (of WARPS_CLASS warps) per SM (20,003-atom globule: 53 us, at 12 61, at 20 56, at 24 59)
constexpr int MINB_CLASS = 16;

// working arrays of one cell's classification (64 planes, 64 vertex slots)
struct alignas(16) ClassTmp {
    unsigned v[64];          // planes of the vertex, its state in the top byte: 0 not in C, 1 tetrahedron
                             // of C, 2 on a ghost plane (dead slot: DEADV)
    unsigned adj[64];        // its neighbours across edges (v0 v1), (v1 v2), (v2 v0)
    uint8_t ek[64][4];       // edge k of vertex t: 1 its triangle is in C, 3 and processed here
    uint8_t act[64], ncl[64], tri[64], out[64], opn[64];   // per face: present, not closed, holds a triangle of C,
                                                           // orthocentre outside, a test left open
    uint8_t item[192], left[96];                           // (t << 2) | k: edges to test, edges left open
};

__device__ __forceinline__ Ctx make_ctx(const AtomArgs& A, int i) {
    Ctx c;
    c.xyz = A.xyz;
    c.R = A.R;
    for (int k = 0; k < 3; ++k) c.pi[k] = A.xyz[3 * i + k];
    c.Ri = A.R[i];
    c.h = ghost_h(c.Ri);
    c.i = i;
    c.n = A.n;
    c.status = A.status;
    return c;
}

// the cold paths: FP32 magnitudes, FP64, exact expansions
template <class SM> __device__ __noinline__ bool tet_exact(const SM* S, const AtomArgs& A, int i, unsigned tv) {
    const Ctx c = make_ctx(A, i);
    const float R = (float)c.Ri;
    return psign<PK_TET>(S, c, FA<float>{R * R, R * R}, tv & 255u, (tv >> 8) & 255u, (tv >> 16) & 255u) <= 0;
}
template <class SM> __device__ __noinline__ bool tri_exact(const SM* S, const AtomArgs& A, int i, int a, int b, int cc, int d) {
    const Ctx c = make_ctx(A, i);
    const float R = (float)c.Ri;
    const FA<float> wi = {R * R, R * R};
    return psign<PK_TRI>(S, c, wi, a, b) <= 0 && (cc < NG || psign<PK_TRIB>(S, c, wi, a, b, cc) <= 0) &&
           (d < NG || psign<PK_TRIB>(S, c, wi, a, b, d) <= 0);
}
template <class SM> __device__ __noinline__ bool edge_exact(const SM* S, const ClassTmp* T, const AtomArgs& A, int i, int a, int hw) {
    const Ctx c = make_ctx(A, i);
    const float R = (float)c.Ri;
    const FA<float> wi = {R * R, R * R};
    if (psign<PK_EDGE>(S, c, wi, a, 0) > 0) return false;
    for (int t = 0; t < hw; ++t) {
        const unsigned v = T->v[t];
        for (int k = 0; k < 3; ++k) {
            const int x = (v >> (8 * k)) & 255u, b = (v >> (8 * ((k + 1) % 3))) & 255u;
            if ((v & DEADV) != DEADV && x == a && b >= NG && psign<PK_EDGEB>(S, c, wi, a, b) > 0) return false;
        }
    }
    return true;
}
template <class SM> __device__ __noinline__ int vert_exact(const SM* S, const AtomArgs& A, int i, int a) {
    return resolve_exact(make_ctx(A, i), PK_VERT, S->pg[a], 0, 0, 0, true);
}

// signs of the tests of cell edge (a, b) whose end vertices lie on planes cc and d: -1 in C, 0 left
// open, 1 not in C.  The orthocentre of the triangle (i, a, b) serves the three tests.
template <class SM> __device__ __forceinline__ int tri_filter(const SM* S, float w, int a, int b, int cc, int d) {
    const PlaneN<FA<float>> Pa = fplane(S, a), Pb = fplane(S, b);
    V3<FA<float>> Z;
    FA<float> W;
    tri_hom(Pa, Pb, Z, W);
    const FA<float> wi = {w, w};
    const int s1 = fa_sign(vdot(Z, Z) - wi * W * W, G32, TINY32);
    if (s1 >= 0) return s1;
    int s = -1;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const int l = k == 0 ? cc : d;
        if (l < NG) continue;
        const PlaneN<FA<float>> L = fplane(S, l);
        const int s2 = fa_sign(vdot(L.q, Z) - L.b * W, G32, TINY32);
        if (s2 > 0) return 1;
        if (s2 == 0) s = 0;
    }
    return s;
}

// Classifies the cell of atom i: slot t = 32 r + lane has planes TV (dead: DEADV), neighbours TA and
// the filter value P of its tetrahedron test (|z|^2 - w_i in homogeneous form).  Writes the
// classification into the record, or the outputs of an atom that no simplex of C holds.
template <class SM>
__device__ __forceinline__ void classify_cell(const SM* S, ClassTmp* T, const AtomArgs& A, int i, CellRecF* rec,
                                              int nc, int hw, const unsigned (&TV)[2], const unsigned (&TA)[2],
                                              const FA<float> (&P)[2], float w) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const int nr = hw > 32 ? 2 : 1, np = NG + nc;
    for (int x = lane; x < 80; x += 32) ((unsigned*)T->act)[x] = 0;
    // ---------------- tetrahedra of C (cell vertices inside B_i)
    unsigned kf[2] = {0, 0};
    bool open = false;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (r >= nr || TV[r] == DEADV) continue;
        const unsigned v = TV[r];
        if ((v & 255u) < NG || ((v >> 8) & 255u) < NG || (v >> 16) < NG) kf[r] = 2;
        else {
            const int sg = fa_sign(P[r], G32, TINY32);
            kf[r] = sg < 0 ? 1 : 0;
            if (sg == 0) {
                kf[r] = 4;
                open = true;
            }
        }
    }
    if (__any_sync(FULL, open)) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (kf[r] == 4) kf[r] = tet_exact(S, A, i, TV[r]) ? 1 : 0;
    }
    __syncwarp();
    bool all_in = true;   // every vertex of the cell inside B_i
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (r >= nr) continue;
        const int t = r * 32 + lane;
        T->v[t] = TV[r] | kf[r] << 24;
        T->adj[t] = TA[r];
        *(unsigned*)T->ek[t] = 0;
        if (TV[r] == DEADV) continue;
        if (kf[r] != 1) all_in = false;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const unsigned a = (TV[r] >> (8 * k)) & 255u;
            T->act[a] = 1;
            if (kf[r] != 1) T->ncl[a] = 1;
        }
    }
    const bool icl = __all_sync(FULL, all_in);   // (the vote orders the stores above before the loads below)
    __syncwarp();
    // ---------------- triangles of C (cell edges meeting B_i): by an end vertex in C, else by the tests
    auto mark = [&](int t, int k, int t2, int a, int b) {
        const unsigned adj2 = T->adj[t2];
        const int k2 = (adj2 & 255u) == (unsigned)t ? 0 : (((adj2 >> 8) & 255u) == (unsigned)t ? 1 : 2);
        T->ek[t][k] = 3;
        T->ek[t2][k2] = 1;
        T->tri[a] = 1;
        T->tri[b] = 1;
    };
    int ni = 0;
#pragma unroll 1
    for (int h = 0; h < 3 * nr; ++h) {
        const int r = h >= 3, k = h - 3 * r, t = r * 32 + lane;
        const unsigned v = r ? TV[1] : TV[0], ta = r ? TA[1] : TA[0], kt = r ? kf[1] : kf[0];
        const int t2 = (ta >> (8 * k)) & 63u;
        const int a = (v >> (8 * k)) & 255u, b = (v >> (k == 2 ? 0 : 8 * k + 8)) & 255u;
        bool want = v != DEADV && t2 > t && a >= NG && b >= NG;   // each cell edge once
        if (want && (kt == 1 || (T->v[t2] >> 24) == 1)) {
            mark(t, k, t2, a, b);
            want = false;
        }
        const unsigned bl = __ballot_sync(FULL, want);
        if (want) T->item[ni + __popc(bl & lt)] = (uint8_t)((t << 2) | k);
        ni += __popc(bl);
    }
    __syncwarp();
    // the planes a, b of edge k of vertex t, the third plane cc of t and the third plane d across it
    auto edge_of = [&](unsigned x, int& t, int& k, int& t2, int& a, int& b, int& cc, int& d) {
        t = x >> 2;
        k = x & 3;
        const unsigned v = T->v[t];
        t2 = (T->adj[t] >> (8 * k)) & 63u;
        a = (v >> (8 * k)) & 255u;
        b = (v >> (k == 2 ? 0 : 8 * k + 8)) & 255u;
        cc = (v >> (k == 0 ? 16 : 8 * k - 8)) & 255u;
        const unsigned w2 = T->v[t2];
        const int x0 = w2 & 255u, x1 = (w2 >> 8) & 255u, x2 = (w2 >> 16) & 255u;
        d = (x0 != a && x0 != b) ? x0 : ((x1 != a && x1 != b) ? x1 : x2);
    };
    int nl = 0;
    for (int j0 = 0; j0 < ni; j0 += 32) {
        bool lft = false;
        unsigned x = 0;
        if (j0 + lane < ni) {
            x = T->item[j0 + lane];
            int t, k, t2, a, b, cc, d;
            edge_of(x, t, k, t2, a, b, cc, d);
            const int sg = tri_filter(S, w, a, b, cc, d);
            if (sg < 0) mark(t, k, t2, a, b);
            lft = sg == 0;
        }
        const unsigned bl = __ballot_sync(FULL, lft);
        if (lft) T->left[nl + __popc(bl & lt)] = (uint8_t)x;
        nl += __popc(bl);
    }
    if (nl) {
        __syncwarp();
        for (int j = lane; j < nl; j += 32) {
            int t, k, t2, a, b, cc, d;
            edge_of(T->left[j], t, k, t2, a, b, cc, d);
            if (tri_exact(S, A, i, a, b, cc, d)) mark(t, k, t2, a, b);
        }
    }
    __syncwarp();
    // ---------------- edges of C (faces meeting B_i): a triangle of C on the face, or the face's
    // orthocentre in B_i and on the inner side of every cell edge of the face
    ni = 0;
#pragma unroll 1
    for (int h = 0; h < 3 * nr; ++h) {
        const int r = h >= 3, k = h - 3 * r, t = r * 32 + lane;
        const unsigned v = r ? TV[1] : TV[0];
        const int a = (v >> (8 * k)) & 255u, b = (v >> (k == 2 ? 0 : 8 * k + 8)) & 255u;
        const bool want = v != DEADV && a >= NG && b >= NG && !T->tri[a & 63];
        const unsigned bl = __ballot_sync(FULL, want);
        if (want) T->item[ni + __popc(bl & lt)] = (uint8_t)((t << 2) | k);
        ni += __popc(bl);
    }
    __syncwarp();
    for (int j = lane; j < ni; j += 32) {
        const unsigned x = T->item[j], v = T->v[x >> 2];
        const int k = x & 3, a = (v >> (8 * k)) & 255u, b = (v >> (k == 2 ? 0 : 8 * k + 8)) & 255u;
        const int sg = fsign<PK_EDGEB>(S, FA<float>{w, w}, a, b);
        if (sg > 0) T->out[a] = 1;
        else if (sg == 0) T->opn[a] = 1;
    }
    __syncwarp();
    bool eK = false;   // some edge of C holds i
    for (int e = lane; e < np; e += 32) {
        uint8_t flag = 0;
        if (e >= NG && T->act[e]) {
            bool in = T->tri[e];
            if (!in && !T->out[e]) {
                const int se = fsign<PK_EDGE>(S, FA<float>{w, w}, e, e);
                if (se < 0 && !T->opn[e]) in = true;
                else if (se <= 0) in = edge_exact(S, T, A, i, e, hw);
            }
            if (in) {
                flag = T->ncl[e] ? 1 : 3;
                eK = true;
            }
        }
        rec->eflag[e] = flag;
    }
    // ---------------- vertex i in C: an edge of C holds it, or p_i lies in its own cell
    bool iK = __any_sync(FULL, eK);
    if (!iK) {
        bool ok = true;
        for (int a = NG + lane; a < np; a += 32) {
            if (!T->act[a]) continue;
            int sg = fa_sign(FA<float>{S->pq[a][3], S->pm[a][1]}, G32, TINY32);
            if (sg == 0) sg = vert_exact(S, A, i, a);
            if (sg < 0) ok = false;
        }
        iK = __all_sync(FULL, ok);
    }
    if (!iK && A.rec == nullptr) {
        // no simplex of C holds i: A_i = 0 (and V_i = 0) and no gradient gathers
        if (lane == 0) {
            A.areas[i] = 0.0;
            if (A.grad) { A.grad[3 * i] = A.grad[3 * i + 1] = A.grad[3 * i + 2] = 0.0; }
            if (A.vol) A.vol[i] = 0.0;
            if (A.vgrad) { A.vgrad[3 * i] = A.vgrad[3 * i + 1] = A.vgrad[3 * i + 2] = 0.0; }
            if (A.mol_done) molecule_count(A, i);
            rec->flag = CELL_DONE;
        }
        __syncwarp();
        return;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int t = r * 32 + lane;
        if (t >= hw) continue;
        const unsigned x = *(const unsigned*)T->ek[t];
        rec->kf[t] = (uint8_t)kf[r];
        rec->tf[t] = (uint8_t)((x & 1u) | (x >> 7 & 2u) | (x >> 14 & 4u) | (x << 3 & 16u) | (x >> 4 & 32u) | (x >> 11 & 64u));
    }
    if (lane == 0) {
        rec->iK = iK;
        rec->icl = icl;
    }
    __syncwarp();
}

struct alignas(16) ClassSmem {
    using Real = float;
    static constexpr int kNE = 64, kNT = 64;
    float pq[64][4];
    float pm[64][2];
    int pg[64];
    ClassTmp tmp;
};

// (a template, so that only the unit that launches it compiles it)
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32, MINB_CLASS) k_class(const __grid_constant__ AtomArgs A) {
    __shared__ ClassSmem smem_all[WARPS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    ClassSmem* S = &smem_all[wib];
    grid_dep_trigger();
    grid_dep_wait();
    const int s = blockIdx.x * WARPS + wib;
    if (s >= A.n) return;
    CellRecF* rec = (CellRecF*)A.cells + s;
    // the record: the header and the first half of every table in one memory round trip, the second
    // half if it is used
    const int i = DS_IDX(A.sidx[s], A.n, A.status);
    const int flag = rec->flag;
    const int4 hd = *reinterpret_cast<const int4*>(&rec->iK);   // iK, icl, nc, hw
    float4 q[2];
    float pb[2];
    int g[2];
    uchar4 v[2], a[2];
    auto load = [&](int h) {
        const int e = lane + 32 * h;
        q[h] = *(const float4*)rec->pq[e];
        pb[h] = rec->pB[e];
        g[h] = rec->pg[e];
        v[h] = rec->tv[e];
        a[h] = rec->ta[e];
    };
    load(0);
    if (flag != CELL_OK) return;   // the outputs of this atom are written
    const int nc = hd.z, hw = hd.w;
    const bool two = NG + nc > 32 || hw > 32;
    if (two) load(1);
    const float Ri = A.Rhl[i].x, w = Ri * Ri;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !two) break;
        const int e = lane + 32 * h;
        *(float4*)S->pq[e] = q[h];
        *(float2*)S->pm[e] = make_float2((fabsf(q[h].x) + fabsf(q[h].y) + fabsf(q[h].z)) * 1.000001f, pb[h]);
        S->pg[e] = g[h];
    }
    __syncwarp();
    unsigned TV[2], TA[2];
    FA<float> P[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        TV[h] = DEADV;
        TA[h] = 0;
        P[h] = {0.f, 0.f};
        if ((h == 1 && !two) || lane + 32 * h >= hw || v[h].x == NONE) continue;
        TV[h] = pack3(v[h].x, v[h].y, v[h].z);
        TA[h] = pack3(a[h].x, a[h].y, a[h].z);
        float V[4], Vd, Vw;
        hom_vertex(*(const float4*)S->pq[v[h].x & 63], *(const float2*)S->pm[v[h].x & 63], *(const float4*)S->pq[v[h].y & 63],
                   *(const float2*)S->pm[v[h].y & 63], *(const float4*)S->pq[v[h].z & 63], *(const float2*)S->pm[v[h].z & 63],
                   V, Vd, Vw);
        P[h].v = V[0] * V[0] + V[1] * V[1] + V[2] * V[2] - w * V[3] * V[3];
        P[h].a = (Vd * Vd + w * Vw * Vw) * 1.000001f;   // at least the sum of the squares' magnitudes
    }
    classify_cell(S, &S->tmp, A, i, rec, nc, hw, TV, TA, P, w);
}

}  // namespace

}  // namespace dsasa
