// Shrake-Rupley numerical SASA on the GPU: an on-device cross-check of the exact areas.
//
// m unit vectors s_k (supplied by the caller) are placed on every probe-inflated sphere; a
// point is exposed when it lies strictly outside every other ball that overlaps the
// sphere, and A_i = 4 pi R_i^2 (exposed points) / m (Shrake & Rupley 1973, the numerical
// method the paper's accuracy comparison uses).  The per-point decision is the one of float32
// operations without contraction (x = R_i s_k, q = float(p_j - p_i),
// d2 = (dx dx + dy dy) + dz dz, covered iff d2 <= R_j^2) so that the exposed counts can be
// compared exactly with a host evaluation of the same arithmetic; the neighbour set uses the
// exact float64 test |p_i - p_j|^2 < (R_i + R_j)^2.
//
// One warp per atom.  Bound: instruction issue.
//   * The candidates that pass the float test are packed before the float64 test, whose
//     instructions cost 64 cycles each however few lanes are active (9 rows of cells took 9 of
//     them before, 1 or 2 do now).
//   * d2 <= R_j^2 is x.q - (|q|^2 - R_j^2) / 2 >= |x|^2 / 2: three multiply-adds and a maximum
//     per pair instead of nine operations.  Only a point whose largest value comes within the
//     rounding bound of |x|^2 / 2 is decided by the operations above.
//   * The neighbours are ordered by the depth of their caps, deepest first.  Every point meets
//     the first SR_FIRST; the points still open, about a quarter, are queued and meet the
//     rest on full lanes.
// A whole call on the 5,000-atom globule with 960 points: 95 -> 51 us (5 or 12 first neighbours instead of
// 8: 50 and 51; 8 points a lane: 56); 20,000 atoms 112 us.
#include "dsasa_kernels.cuh"

namespace dsasa {

namespace {

constexpr int SR_WARPS = 4;      // atoms per block
constexpr int SR_KN = 128;       // overlapping neighbours per atom (more: capacity error)
constexpr int SR_PPL = 4;        // points per lane per pass
constexpr int SR_PASS = 32 * SR_PPL;
constexpr int SR_FIRST = 8;      // neighbours that every point meets
constexpr unsigned SR_OPEN = 0x80000000u;   // queue entry: the first neighbours left the point open

struct SRSmem {
    float4 nb[SR_KN];            // q_j = float(p_j - p_i), -(|q_j|^2 - R_j^2) / 2; then by cap depth
    float4 raw[SR_KN];           // q_j, R_j^2
    float key[SR_KN];            // distance of the cap's plane
    unsigned queue[2 * SR_PASS];
    int cand[64];
};

// the decision of one point against every neighbour by the operations that define it
__device__ __noinline__ bool sr_covered(const SRSmem* S, int nn, float px, float py, float pz) {
    bool cov = false;
    for (int j = 0; j < nn; ++j) {
        const float4 q = S->raw[j];
        const float dx = __fsub_rn(px, q.x), dy = __fsub_rn(py, q.y), dz = __fsub_rn(pz, q.z);
        const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
        cov = cov || d2 <= q.w;
    }
    return cov;
}

__global__ void __launch_bounds__(SR_WARPS * 32) k_shrake_rupley(SRArgs A) {
    __shared__ SRSmem smem_all[SR_WARPS];
    grid_dep_wait();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    SRSmem* S = &smem_all[wib];
    const int s = blockIdx.x * SR_WARPS + wib;
    if (s >= A.n) return;
    const unsigned full = 0xffffffffu;
    unsigned lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    const int i = A.sidx[s];
    const float4 fi = A.sf4[s];
    const MolGrid G = A.grids[A.molid[i]];
    const double pix = A.xyz[3 * i], piy = A.xyz[3 * i + 1], piz = A.xyz[3 * i + 2], Ri = A.R[i];

    // overlapping neighbours: float prefilter with the grid's slack, then the exact float64 test
    // of up to 32 candidates at a time
    int nn = 0, nc = 0;
    bool ovf = false;
    auto exact = [&](int count) {   // tests cand[0 .. count)
        bool ok = false;
        double qx, qy, qz, Rj;
        if (lane < count) {
            const int j = S->cand[lane];
            qx = __dsub_rn(A.xyz[3 * j], pix);
            qy = __dsub_rn(A.xyz[3 * j + 1], piy);
            qz = __dsub_rn(A.xyz[3 * j + 2], piz);
            Rj = A.R[j];
            const double dd = __dadd_rn(__dadd_rn(__dmul_rn(qx, qx), __dmul_rn(qy, qy)), __dmul_rn(qz, qz));
            const double rs = __dadd_rn(Rj, Ri);
            ok = dd < __dmul_rn(rs, rs);
        }
        const unsigned bal = __ballot_sync(full, ok);
        const int pos = nn + __popc(bal & lt);
        if (ok) {
            if (pos < SR_KN) {
                const float Rjf = (float)Rj;
                S->raw[pos] = make_float4((float)qx, (float)qy, (float)qz, __fmul_rn(Rjf, Rjf));
            } else ovf = true;
        }
        nn += __popc(bal);
    };
    NearRows near(G, A.cstart, fi, (int*)S->key);
    for (int f0 = 0; f0 < near.total; f0 += 32) {
        const int k = near.at(f0);
        bool ok = false;
        int j = -1;
        if (f0 + lane < near.total) {
            const float4 fj = A.sf4[k];
            j = A.sidx[k];
            const float dx = fj.x - fi.x, dy = fj.y - fi.y, dz = fj.z - fi.z;
            const float rr = fi.w + fj.w + G.margin;
            ok = j != i && dx * dx + dy * dy + dz * dz < rr * rr;
        }
        const unsigned bal = __ballot_sync(full, ok);
        if (ok) S->cand[nc + __popc(bal & lt)] = j;
        nc += __popc(bal);
        if (nc >= 32) {
            __syncwarp();
            exact(32);
            const int rest = lane < nc - 32 ? S->cand[32 + lane] : 0;
            __syncwarp();
            if (lane < nc - 32) S->cand[lane] = rest;
            nc -= 32;
        }
    }
    __syncwarp();
    if (nc > 0) exact(nc);
    __syncwarp();
    if (__any_sync(full, ovf) || nn > SR_KN) {
        if (lane == 0) {
            atomicOr(A.status, ST_CAND_OVF);
            A.areas[i] = __longlong_as_double(0x7ff8000000000000ll);
            if (A.exposed) A.exposed[i] = -1;
        }
        return;
    }

    // the neighbours by the depth of their caps (ties: position), and the bound of the rounding
    // of both evaluations: u = 2^-24, S = 2 |x|^2 + 2 max |q|^2 + max R_j^2 bounds (|x| + |q|)^2 +
    // R_j^2; the value below errs by at most 5 u S / 2 + u S and half of d2 by 2.5 u S; 16 u S
    // is taken
    const float Rf = (float)Ri;
    float bound = 0.f;
    for (int j = lane; j < nn; j += 32) {
        const float4 q = S->raw[j];
        const float q2 = q.x * q.x + q.y * q.y + q.z * q.z;
        S->key[j] = (q2 + Rf * Rf - q.w) * rsqrtf(q2 + 1e-30f);   // twice the distance of the cap's plane
        bound = fmaxf(bound, 2.f * q2 + q.w);
    }
    for (int o = 16; o > 0; o >>= 1) bound = fmaxf(bound, __shfl_xor_sync(full, bound, o));
    const float e0 = bound * 9.5367431640625e-07f * 1.00001f + 1e-30f;   // 2^-20 times the neighbours' part
    __syncwarp();
    int rank[SR_KN / 32];
#pragma unroll
    for (int r = 0; r < SR_KN / 32; ++r) {
        const int j = r * 32 + lane;
        rank[r] = 0;
        if (r * 32 >= nn) break;
        const float mine = j < nn ? S->key[j] : 0.f;
        for (int k = 0; k < nn; ++k) {
            const float o = S->key[k];
            rank[r] += o < mine || (o == mine && k < j);
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < SR_KN / 32; ++r) {
        const int j = r * 32 + lane;
        if (r * 32 >= nn) break;
        if (j < nn) {
            const float4 q = S->raw[j];
            S->nb[rank[r]] = make_float4(q.x, q.y, q.z, -0.5f * ((q.x * q.x + q.y * q.y + q.z * q.z) - q.w));
        }
    }
    __syncwarp();

    // points: the largest x.q - (|q|^2 - R_j^2) / 2 against |x|^2 / 2
    int cnt = 0;
    const int n1 = min(nn, SR_FIRST);
    auto scan = [&](int j0, int j1, const float (&px)[SR_PPL], const float (&py)[SR_PPL], const float (&pz)[SR_PPL],
                    float (&best)[SR_PPL]) {
#pragma unroll
        for (int p = 0; p < SR_PPL; ++p) best[p] = -INFINITY;
        for (int j = j0; j < j1; ++j) {
            const float4 q = S->nb[j];
#pragma unroll
            for (int p = 0; p < SR_PPL; ++p)
                best[p] = fmaxf(best[p], fmaf(px[p], q.x, fmaf(py[p], q.y, fmaf(pz[p], q.z, q.w))));
        }
    };
    auto place = [&](int k, float& px, float& py, float& pz, float& h, float& e) {
        px = __fmul_rn(Rf, A.pts[3 * k]);
        py = __fmul_rn(Rf, A.pts[3 * k + 1]);
        pz = __fmul_rn(Rf, A.pts[3 * k + 2]);
        h = 0.5f * (px * px + py * py + pz * pz);
        e = fmaf(h, 4.f * 9.5367431640625e-07f, e0);
    };
    int qn = 0;
    auto drain = [&](int q0, int count) {   // the queued points against the other neighbours
        float px[SR_PPL], py[SR_PPL], pz[SR_PPL], h[SR_PPL], e[SR_PPL], best[SR_PPL];
        unsigned w[SR_PPL];
#pragma unroll
        for (int p = 0; p < SR_PPL; ++p) {
            const int x = p * 32 + lane;
            w[p] = x < count ? S->queue[q0 + x] : ~0u;
            place(x < count ? (int)(w[p] & ~SR_OPEN) : 0, px[p], py[p], pz[p], h[p], e[p]);
        }
        scan(n1, nn, px, py, pz, best);
#pragma unroll
        for (int p = 0; p < SR_PPL; ++p) {
            if (p * 32 + lane >= count || best[p] > h[p] + e[p]) continue;   // covered
            const bool clear = !(w[p] & SR_OPEN) && best[p] < h[p] - e[p];
            if (clear || !sr_covered(S, nn, px[p], py[p], pz[p])) ++cnt;
        }
    };
    for (int k0 = 0; k0 < A.m; k0 += SR_PASS) {
        float px[SR_PPL], py[SR_PPL], pz[SR_PPL], h[SR_PPL], e[SR_PPL], best[SR_PPL];
#pragma unroll
        for (int p = 0; p < SR_PPL; ++p) {
            const int k = k0 + p * 32 + lane;
            place(k < A.m ? k : 0, px[p], py[p], pz[p], h[p], e[p]);
        }
        scan(0, n1, px, py, pz, best);
#pragma unroll
        for (int p = 0; p < SR_PPL; ++p) {
            const int k = k0 + p * 32 + lane;
            const bool open = k < A.m && !(best[p] > h[p] + e[p]);
            const unsigned bal = __ballot_sync(full, open);
            if (open) S->queue[qn + __popc(bal & lt)] = (unsigned)k | (best[p] < h[p] - e[p] ? 0u : SR_OPEN);
            qn += __popc(bal);
        }
        __syncwarp();
        if (qn >= SR_PASS) {
            qn -= SR_PASS;
            drain(qn, SR_PASS);
            __syncwarp();
        }
    }
    if (qn > 0) drain(0, qn);
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(full, cnt, o);
    if (lane == 0) {
        A.areas[i] = 4.0 * 3.14159265358979323846 * Ri * Ri * (double)cnt / (double)A.m;
        if (A.exposed) A.exposed[i] = cnt;
        if (A.tests) atomicAdd(A.tests, (unsigned long long)A.m * (unsigned long long)nn);
    }
}

}  // namespace

cudaError_t launch_sr(const SRArgs& a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    const cudaError_t e = launch_dependent(k_shrake_rupley, (a.n + SR_WARPS - 1) / SR_WARPS, SR_WARPS * 32, s, true, a);
    note_launches(1);
    return e;
}

}  // namespace dsasa
