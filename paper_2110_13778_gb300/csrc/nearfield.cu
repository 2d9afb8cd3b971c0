// Near field of the FMM matrix-vector product (Section 2.4, step 1 "Nearfield Calculation"):
// for every leaf c and every neighbour leaf c' in N(c), the Galerkin block of A between their
// elements is applied directly. Regular pairs use the one-point (centroid) rule
// A_i A_j K_m(c_i, c_j); identical and adjacent pairs receive their Sauter-Schwab
// correction afterwards (k_corrections). The mass terms 1/2 (1 + eps) A_i and
// 1/2 (1 + 1/eps) A_i of eq_linsysEntry are added here.
//
// Row signs follow eqbim_5/eqbim_6:
//   y1_i = 1/2 (1 + eps) A_i phi_i     - sum_j (I1_ij dphi_j + I2_ij phi_j)
//   y2_i = 1/2 (1 + 1/eps) A_i dphi_i  - sum_j (I3_ij dphi_j + I4_ij phi_j)
//
// Layout: both precisions work on pair tiles of chunks of at most 32 elements of neighbouring
// leaves (FP64: k_near64). Mixed precision: one warp per chunk of up to 32 targets, which
// evaluates each pair of distinct chunks once for both directions (k_near_tile; several
// right-hand sides: k_near32m, one direction, up to 16 densities per pair evaluation). In
// mixed precision each source leaf's partial sums are kept in FP32
// and added into FP64 accumulators per leaf (compensated leaf sums), and coordinates are
// carried as FP32 hi + lo pairs so that d = (x_hi - y_hi) + (x_lo - y_lo) keeps the
// separation of close elements to FP32 relative accuracy instead of losing digits to the
// size of the coordinates.
#include <algorithm>
#include <vector>

#include "f32x2.cuh"
#include "kernels.cuh"
#include "pb_internal.cuh"


#define NEAR_ITEM 6    // most pair tiles per warp of the mixed-precision near field
#define NEAR_ITEM_M 8  // directed tiles per warp of the several-vector near field

// ---------- FP64 near field ----------
// Pair tiles as in the mixed-precision kernel below: one warp per pair of chunks (A, B) of at most
// 32 elements of neighbouring leaves evaluates each pair once for both directions. The FP64 pipe
// (1/64 of the FP32 rate) is all that counts here: 53 FP64 operations, one reciprocal square root
// and one exponential per pair of elements, where one direction at a time took 45 and the same
// two functions per direction. The larger chunk goes to the lanes and the other is walked, so
// that only the steps of a remainder chunk with a remainder chunk leave lanes idle. At step s
// lane l meets source (l mod nb + s) mod nb; the sources' sums live in shared memory, one set
// per group of nb lanes, so that the lanes of a step write different words and the sum of a
// source has a fixed order. Every tile writes the sums of both its chunks (2 x 2 x 32 doubles),
// which k_near64_sum adds per element in tile order: no atomics, and the product does not depend
// on scheduling. 20,480 elements: near field 1.80 ms; 11.3 ms one direction at a time with a block of 128
// threads per leaf of 76.
//
// The tiles are numbered, not listed: chunk a is the first of tiles base[a] .. base[a + 1], with the
// chunks b >= a of its own leaf k, then those of the neighbour leaves after k in list order (pos[t]: the
// place of neighbour entry t there; for an entry t to a leaf before k, pos[t] is the place of k in that
// leaf's tiles). A product takes the tiles in batches of whole first chunks, of at most NEAR64_BATCH
// tiles, so that their sums take 256 MB however large the leaves are.
#define NEAR64_BATCH (1 << 18)
struct Near64Tiles {
    const long long* base;
    const int *first, *noff, *nidx, *pos;  // first: first chunk of each leaf
    int a0, a1;                            // the batch: its first chunks
};
struct Near64Src {
    double x[32], y[32], z[32], nx[32], ny[32], nz[32], phi[32], dphi[32];
    double r1[64], r2[64];  // ceil(32 / nb) groups of nb <= 32 sums: at most 63
};
__global__ void __launch_bounds__(256, 2) k_near64(int nt, const __grid_constant__ Near64Tiles q,
                                                const int* __restrict__ chunk_leaf,
                                                const int* __restrict__ chunk_first, const int* __restrict__ begin,
                                                const double4_32a* __restrict__ ep, const double4_32a* __restrict__ en,
                                                const double* __restrict__ xs, double eps, double kappa,
                                                double* __restrict__ part)
{
    __shared__ Near64Src sh[8];
    const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const long long at = q.base[q.a0] + w;
    if (at >= q.base[q.a1]) return;
    Near64Src& S = sh[threadIdx.x >> 5];
    int2 t;  // the chunks of tile `at`
    {
        int lo = q.a0, hi = q.a1;  // base[lo] <= at < base[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (q.base[mid] <= at) lo = mid;
            else hi = mid;
        }
        const int k = chunk_leaf[lo], own = q.first[k + 1] - lo;
        int j = (int)(at - q.base[lo]);
        t = make_int2(lo, lo + j);
        if (j >= own) {
            j -= own;
            t.y = lo;
            for (int e0 = q.noff[k]; e0 < q.noff[k + 1]; e0 += 32) {
                const int e = e0 + lane, c = e < q.noff[k + 1] ? q.nidx[e] : -1;
                const int b = c > k ? j - q.pos[e] : -1;
                const bool here = b >= 0 && b < q.first[c + 1] - q.first[c];
                const unsigned m = __ballot_sync(0xffffffffu, here);
                if (m) {
                    t.y = __shfl_sync(0xffffffffu, here ? q.first[c] + b : 0, __ffs(m) - 1);
                    break;
                }
            }
        }
    }
    int a0 = chunk_first[t.x], b0 = chunk_first[t.y];
    int na = min(32, begin[chunk_leaf[t.x] + 1] - a0), nb = min(32, begin[chunk_leaf[t.y] + 1] - b0);
    const bool diag = t.x == t.y;
    const int side = nb > na;  // the lanes hold the second chunk
    if (side) {
        const int a = a0, n = na;
        a0 = b0;
        na = nb;
        b0 = a;
        nb = n;
    }
    const double i4pi = 0.07957747154594767, inv_eps = 1.0 / eps;
    if (lane < nb) {
        const double4_32a p = ep[b0 + lane], n = en[b0 + lane];
        S.x[lane] = p.x;
        S.y[lane] = p.y;
        S.z[lane] = p.z;
        S.nx[lane] = n.x;
        S.ny[lane] = n.y;
        S.nz[lane] = n.z;
        S.phi[lane] = p.w * xs[b0 + lane] * i4pi;  // 1 / (4 pi) rides on the densities
        S.dphi[lane] = p.w * xs[nt + b0 + lane] * i4pi;
    }
    S.r1[lane] = S.r1[32 + lane] = 0.0;
    S.r2[lane] = S.r2[32 + lane] = 0.0;
    const bool act = lane < na;
    const int k = a0 + (act ? lane : 0);
    const double4_32a P = ep[k], Nn = en[k];
    const double phi = act ? P.w * xs[k] * i4pi : 0.0, dphi = act ? P.w * xs[nt + k] * i4pi : 0.0;
    __syncwarp();
    double s1 = 0.0, s2 = 0.0;
    const int g0 = lane / nb * nb;  // this lane's group of sums
    int m = lane - g0;
    for (int s = 0; s < nb; ++s) {
        const bool same = diag && m == lane;  // the identical pair is the correction's
        if (act && !same) {
            const double dx = P.x - S.x[m], dy = P.y - S.y[m], dz = P.z - S.z[m];
            const double ax = S.nx[m], ay = S.ny[m], az = S.nz[m];
            const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
            const double ri = rsqrt(r2);
            const double t1 = kappa * (r2 * ri);
            const double e = exp(-t1);
            const double e1 = fma(e, t1, e);                             // e^-t (1 + t)
            const double c1n = e1 - 1.0;                                 // -c1
            const double c3n = fma(e, fma(t1, t1 + 3.0, 3.0), -3.0);     // -c3
            const double ri2 = ri * ri, ri3 = ri2 * ri;
            const double nxd = fma(Nn.z, dz, fma(Nn.y, dy, Nn.x * dx));
            const double nyd = fma(az, dz, fma(ay, dy, ax * dx));
            const double nn = fma(Nn.z, az, fma(Nn.y, ay, Nn.x * ax));
            const double f2 = ri3 * fma(eps, e1, -1.0), f3 = ri3 * fma(-inv_eps, e1, 1.0);
            const double k1 = (1.0 - e) * ri;
            const double k4 = ri3 * fma(c1n, nn, -c3n * (nxd * nyd * ri2));
            const double sp = S.phi[m], sd = S.dphi[m];
            s1 = fma(k1, sd, fma(nyd * f2, sp, s1));
            s2 = fma(k4, sp, fma(-nxd * f3, sd, s2));
            if (!diag) {
                double* q1 = &S.r1[g0 + m];
                double* q2 = &S.r2[g0 + m];
                *q1 = fma(k1, dphi, fma(-nxd * f2, phi, *q1));
                *q2 = fma(k4, phi, fma(nyd * f3, dphi, *q2));
            }
        }
        __syncwarp();
        if (++m == nb) m = 0;
    }
    double* out = part + (size_t)w * 128 + side * 64;
    out[lane] = s1;
    out[32 + lane] = s2;
    if (!diag) {
        out = part + (size_t)w * 128 + (side ^ 1) * 64;
        double v1 = 0.0, v2 = 0.0;
        if (lane < nb)
            for (int g = lane; g - lane < 32; g += nb) {
                v1 += S.r1[g];
                v2 += S.r2[g];
            }
        out[lane] = v1;
        out[32 + lane] = v2;
    }
}

// One warp per chunk: y1 = 1/2 (1 + eps) A phi - A acc1, y2 = 1/2 (1 + 1/eps) A dphi - A acc2 with
// acc the tiles' sums of the chunk in tile order. ys carries acc from batch to batch (start: the first
// batch, end: the last).
__global__ void __launch_bounds__(256) k_near64_sum(int nt, int nchunks, const __grid_constant__ Near64Tiles q,
                                                    const int* __restrict__ chunk_leaf,
                                                    const int* __restrict__ chunk_first, const int* __restrict__ begin,
                                                    const double4_32a* __restrict__ ep, const double* __restrict__ part,
                                                    const double* __restrict__ xs, double eps, bool start, bool end,
                                                    double* __restrict__ ys)
{
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= nchunks) return;
    const int leaf = chunk_leaf[c], k = chunk_first[c] + lane;
    const bool act = k < begin[leaf + 1];
    const long long t0 = q.base[q.a0];
    double a1 = start || !act ? 0.0 : ys[k], a2 = start || !act ? 0.0 : ys[nt + k];
    auto add = [&](long long tile, int side) {
        const double* p = part + (size_t)(tile - t0) * 128 + side * 64;
        a1 += p[lane];
        a2 += p[32 + lane];
    };
    for (int e = q.noff[leaf]; e < q.noff[leaf + 1]; ++e) {
        const int l = q.nidx[e];
        if (l > leaf) continue;
        // as second chunk: of the chunks of a leaf before, and of the own leaf's chunks before this one
        const int own = q.first[l + 1], to = min(l == leaf ? c : own, q.a1);
        const int at = l == leaf ? c : own + q.pos[e] + c - q.first[leaf];
#pragma unroll 4
        for (int a = max(q.first[l], q.a0); a < to; ++a) add(q.base[a] + (at - a), 1);
    }
    if (c >= q.a0 && c < q.a1) {
        const long long t1 = q.base[c + 1];
#pragma unroll 4
        for (long long t = q.base[c]; t < t1; ++t) add(t, 0);
    }
    if (!act) return;
    if (end) {
        const double A = ep[k].w;
        a1 = 0.5 * (1.0 + eps) * A * xs[k] - A * a1;
        a2 = 0.5 * (1.0 + 1.0 / eps) * A * xs[nt + k] - A * a2;
    }
    ys[k] = a1;
    ys[nt + k] = a2;
}

// chunks, the numbering of the pair tiles, its batches, and the sums of one batch
static int near64_setup(pb_ctx* c)
{
    const PbLevel& lv = c->lev[c->L];
    const std::vector<int>&b = c->h_leaf_begin, &no = c->h_near_off, &ni = c->h_near_idx;
    std::vector<int>&cl = c->h_up_i[0], &cf = c->h_up_i[1], &pos = c->h_up_i[4], &first = c->h_up_i[5];
    std::vector<long long>& base = c->h_up_l64;
    cl.clear();
    cf.clear();
    first.assign(lv.ncl + 1, 0);
    for (int k = 0; k < lv.ncl; ++k) {
        for (int s = b[k]; s < b[k + 1]; s += 32) {
            cl.push_back(k);
            cf.push_back(s);
        }
        first[k + 1] = (int)cl.size();
    }
    c->nchunks = (int)cl.size();
    pos.assign(ni.size(), 0);
    base.assign(1, 0);
    for (int k = 0; k < lv.ncl; ++k) {
        int after = 0;  // chunks of the neighbour leaves after k
        for (int t = no[k]; t < no[k + 1]; ++t)
            if (ni[t] > k) {
                pos[t] = after;
                after += first[ni[t] + 1] - first[ni[t]];
            }
        for (int a = first[k]; a < first[k + 1]; ++a) base.push_back(base.back() + (first[k + 1] - a) + after);
    }
    for (int k = 0; k < lv.ncl; ++k)
        for (int t = no[k]; t < no[k + 1]; ++t)
            if (ni[t] < k)
                for (int u = no[ni[t]]; u < no[ni[t] + 1]; ++u)  // (neighbours are mutual)
                    if (ni[u] == k) pos[t] = pos[u];
    std::vector<int>& cut = c->near64_cut;
    cut.assign(1, 0);
    long long most = 0;
    for (int a = 0; a < c->nchunks; ++a) {
        if (a > cut.back() && base[a + 1] - base[cut.back()] > NEAR64_BATCH) cut.push_back(a);
        most = std::max(most, base[a + 1] - base[cut.back()]);
    }
    cut.push_back(c->nchunks);
    c->chunk_leaf = (int*)pb_alloc(c, sizeof(int) * cl.size());
    c->chunk_first = (int*)pb_alloc(c, sizeof(int) * cf.size());
    c->near64_first = (int*)pb_alloc(c, sizeof(int) * first.size());
    c->near64_pos = (int*)pb_alloc(c, sizeof(int) * pos.size());
    c->near64_base = (long long*)pb_alloc(c, sizeof(long long) * base.size());
    c->near_part = (double*)pb_alloc(c, sizeof(double) * 128 * (size_t)most);
    if (!c->chunk_leaf || !c->chunk_first || !c->near64_first || !c->near64_pos || !c->near64_base || !c->near_part)
        return pb_fail(c, PB_ERR_NOMEM, "near setup: out of memory");
    auto up = [&](void* d, const void* h, size_t n) { return cudaMemcpyAsync(d, h, n, cudaMemcpyHostToDevice, c->st); };
    PB_CUDA(c, up(c->chunk_leaf, cl.data(), sizeof(int) * cl.size()));
    PB_CUDA(c, up(c->chunk_first, cf.data(), sizeof(int) * cf.size()));
    PB_CUDA(c, up(c->near64_first, first.data(), sizeof(int) * first.size()));
    PB_CUDA(c, up(c->near64_pos, pos.data(), sizeof(int) * pos.size()));
    PB_CUDA(c, up(c->near64_base, base.data(), sizeof(long long) * base.size()));
    return PB_OK;
}

// ---------- mixed precision near field ----------
// Per matrix-vector product the sources are packed once as FP32 records
// (x_hi, y_hi, z_hi, A phi), (n_x, n_y, n_z, A dphi) beside the fixed (x_lo, y_lo, z_lo), and the
// sums are set to zero. With order (the caller's vector is in element order) the tree-ordered copy
// xs is made on the way.
__global__ void k_near_pack(int nt, const float4* __restrict__ e32p, const float4* __restrict__ e32n,
                            const int* __restrict__ order, const double* __restrict__ x, double* __restrict__ xs,
                            float4* __restrict__ sp, float4* __restrict__ sn, double* __restrict__ ys)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    float4 p = e32p[k], n = e32n[k];
    const int e = order ? order[k] : k;
    const double v1 = x[e], v2 = x[nt + e];
    if (order) {
        xs[k] = v1;
        xs[nt + k] = v2;
    }
    ys[k] = 0.0;
    ys[nt + k] = 0.0;
    double A = (double)p.w;
    sp[k] = make_float4(p.x, p.y, p.z, (float)(A * v1));
    sn[k] = make_float4(n.x, n.y, n.z, (float)(A * v2));
}


// ---------- the tile kernel (mixed precision) ----------
// Both directions of a pair at once, by tiles of one target chunk A (up to 32 targets, lane l
// holds A_l) and one source chunk B of nb <= 32 sources. K1 and K4 are symmetric in (x, y),
// and with d = x_i - x_j the double-layer kernels of the reversed pair follow from the same
// radial factors: K2(j, i) = -(n_i.d) ri3 (eps e1 - 1), K3(j, i) = (n_j.d) ri3 (1 - e1/eps).
// The tiles (A, B) -- every source chunk B of the neighbour leaves c2 >= c that follows A (B
// after A within A's own leaf) -- are cut into work items of at most NEAR_ITEM tiles of one A;
// one warp per item, so that the warps carry nearly equal work whatever the leaf order. B's
// records are staged in shared memory as packed pairs (below); at step s (s < ceil(nb / 2)) lane
// l pairs A_l with B_((l + s) mod nb) and B_((l + s + h) mod nb), h = ceil(nb / 2), and keeps
// the forward terms. The reverse terms of a full tile of another chunk (nb = 32) ride in
// registers that move one lane down after every step (shuffles), so that after 16 steps lane l
// holds the sums of sources (l + 16) mod 32 and l; in partial tiles lane j gathers those of source
// j by shuffles. Forward sums of a chunk and reverse sums of a
// tile are FP32, added into FP64 (atomics for the reverse terms and the final forward sums; ys
// starts at zero). The tile of A with itself keeps only the forward terms and drops the
// identical pair.
// Q2 > 1: the records are the points of a regular rule (Q2 per element, consecutive; Q2 divides
// 32 and every leaf starts at an element, so no chunk splits an element): the pairs of points of
// one element are dropped, which can only happen in the tile of a chunk with itself.
//
// Packed pairs: entry m of a staged tile holds source m in the low halves and source
// (m + h) mod nb in the high halves, as F0 = (x, y), F1 = (z, A phi), F2 = (n_x, n_y),
// F3 = (n_z, -A dphi) of the high coordinate parts and F4 = (x, y), F5 = (z) of the low
// parts. Every FP32 operation of the two pairs of a step is one f32x2 instruction; only the
// reciprocal square root, the exponential and the branch of the screening function run per
// half. (The packed instructions do not raise the FP32 rate; they halve the issue slots that
// bound this loop.)
//
// Bound: the FMA pipe (two cycles per packed instruction; 62 of them per step of 64 pairs, 69 %
// busy on 737,280 elements of 170 per leaf). Against shared-memory sums and the general screening
// function in every tile: 3090 -> 2567 us there, 202 -> 158 us on 81,920 elements (leaves of 71:
// 20 % of the steps are remainder tiles), 35 -> 12 us on 1280. Blocks of four warps, because items
// differ in length; seven per SM (72 registers) is the best of 5 to 8 by 1 to 4 %.
struct NearTgt2 {
    f2x px, py, pz, lx, ly, lz, nx, ny, nz, phi, dphi;
};

// s1, s2 += forward terms; q1n -= first reverse term, q2 += second reverse term (per half).
// BUMP: bump is added to r^2 of dropped pairs (so that r stays finite); scale = 1 / (4 pi) or 0.
// The Taylor series of the screening function (nine of 64 packed operations and the selections) is
// needed where kappa r < 0.125 only: FAR says that no pair of the tile is that close; other tiles ask
// the warp at every step. The bare (flushing) reciprocal square root and exponential give the bits of
// rsqrtf and __expf wherever those matter: r^2 is no subnormal number for distinct centres, and
// e^-t - 1 is -1 for a flushed e^-t as for a subnormal one.
template <bool BUMP, bool FAR>
__device__ __forceinline__ void near_pair_x2(const NearTgt2& T, const float4* __restrict__ e,
                                             const float2* __restrict__ e5, f2x bump, f2x scale, f2x eps2, f2x nieps2,
                                             f2x kappa2, f2x& s1, f2x& s2, f2x& q1n, f2x& q2)
{
    const float4 g0 = e[0], g1 = e[32], g2 = e[64], g3 = e[96], g4 = e[128];
    const float2 g5 = *e5;
    const f2x ax = x2_pack(g0.x, g0.y), ay = x2_pack(g0.z, g0.w), az = x2_pack(g1.x, g1.y);
    const f2x aphi = x2_pack(g1.z, g1.w);
    const f2x bx = x2_pack(g2.x, g2.y), by = x2_pack(g2.z, g2.w), bz = x2_pack(g3.x, g3.y);
    const f2x nadphi = x2_pack(g3.z, g3.w);
    const f2x lx = x2_pack(g4.x, g4.y), ly = x2_pack(g4.z, g4.w), lz = x2_pack(g5.x, g5.y);
    const f2x one = x2_dup(1.f), mone = x2_dup(-1.f), three = x2_dup(3.f);
    const f2x dx = x2_add(x2_sub(T.px, ax), x2_sub(T.lx, lx));
    const f2x dy = x2_add(x2_sub(T.py, ay), x2_sub(T.ly, ly));
    const f2x dz = x2_add(x2_sub(T.pz, az), x2_sub(T.lz, lz));
    f2x r2 = x2_fma(dz, dz, x2_fma(dy, dy, x2_mul(dx, dx)));
    if (BUMP) r2 = x2_add(r2, bump);
    float ra, rb;
    x2_unpack(r2, ra, rb);
    const f2x rinv = x2_pack(rsqrt_ftz(ra), rsqrt_ftz(rb));
    const f2x tt = x2_mul(kappa2, x2_mul(r2, rinv));
    float xa, xb;
    x2_unpack(x2_mul(tt, x2_dup(-1.4426950408889634f)), xa, xb);
    f2x E = x2_add(x2_pack(ex2_ftz(xa), ex2_ftz(xb)), mone);
    f2x g = x2_add(E, tt);
    if (!FAR) {
        float ta, tb;
        x2_unpack(tt, ta, tb);
        const bool sa = ta < 0.125f, sb = tb < 0.125f;
        if (__any_sync(0xffffffffu, sa || sb)) {
            // g / t^2 = 1/2 - t/6 + t^2/24 - ... (the Taylor series of e^-t - 1 + t), for small t
            f2x sg = x2_fma(x2_dup(1.f / 40320.f), tt, x2_dup(-1.f / 5040.f));
            sg = x2_fma(sg, tt, x2_dup(1.f / 720.f));
            sg = x2_fma(sg, tt, x2_dup(-1.f / 120.f));
            sg = x2_fma(sg, tt, x2_dup(1.f / 24.f));
            sg = x2_fma(sg, tt, x2_dup(-1.f / 6.f));
            sg = x2_fma(sg, tt, x2_dup(0.5f));
            const f2x gs = x2_mul(x2_mul(sg, tt), tt);
            const f2x eb = x2_sub(gs, tt);
            float gsa, gsb, gaa, gab, eba, ebb, eda, edb;
            x2_unpack(gs, gsa, gsb);
            x2_unpack(g, gaa, gab);
            x2_unpack(eb, eba, ebb);
            x2_unpack(E, eda, edb);
            g = x2_pack(sa ? gsa : gaa, sb ? gsb : gab);
            E = x2_pack(sa ? eba : eda, sb ? ebb : edb);
        }
    }
    const f2x tE = x2_mul(tt, E);
    const f2x c1n = x2_add(g, tE);                                            // -c1
    const f2x c3n = x2_fma(tE, x2_add(three, tt), x2_fma(tt, tt, x2_mul(three, g)));  // -c3
    const f2x ri = x2_mul(rinv, scale);
    const f2x ri3 = x2_mul(x2_mul(ri, rinv), rinv);
    const f2x nxd = x2_fma(T.nz, dz, x2_fma(T.ny, dy, x2_mul(T.nx, dx)));
    const f2x nyd = x2_fma(bz, dz, x2_fma(by, dy, x2_mul(bx, dx)));
    const f2x nxny = x2_fma(T.nz, bz, x2_fma(T.ny, by, x2_mul(T.nx, bx)));
    const f2x e1 = x2_add(one, c1n);
    const f2x f2 = x2_mul(ri3, x2_fma(eps2, e1, mone));   // ri3 (eps e1 - 1)
    const f2x f3 = x2_mul(ri3, x2_fma(nieps2, e1, one));  // ri3 (1 - e1 / eps)
    const f2x k1n = x2_mul(E, ri);                       // -K1
    const f2x u = x2_mul(x2_mul(nxd, nyd), x2_mul(rinv, rinv));
    const f2x k4 = x2_mul(ri3, x2_sub(x2_mul(c1n, nxny), x2_mul(c3n, u)));
    s1 = x2_fma(k1n, nadphi, x2_fma(x2_mul(nyd, f2), aphi, s1));
    s2 = x2_fma(k4, aphi, x2_fma(x2_mul(nxd, f3), nadphi, s2));
    q1n = x2_fma(k1n, T.dphi, x2_fma(x2_mul(nxd, f2), T.phi, q1n));
    q2 = x2_fma(k4, T.phi, x2_fma(x2_mul(nyd, f3), T.dphi, q2));
}

__device__ __forceinline__ f2x x2_shfl_down1(f2x v, int lane)
{
    float a, b;
    x2_unpack(v, a, b);
    a = __shfl_sync(0xffffffffu, a, (lane + 1) & 31);
    b = __shfl_sync(0xffffffffu, b, (lane + 1) & 31);
    return x2_pack(a, b);
}

// a full tile of another chunk: lane l meets sources (l + s) mod 32 and (l + s + 16) mod 32 at step
// s; the reverse sums move one lane down after every step. t1, t2: the sums of source `lane`.
template <bool FAR>
__device__ __forceinline__ void near_tile_full(const NearTgt2& T, const float4* F, const float2* F5, int lane, f2x sc,
                                               f2x eps2, f2x nieps2, f2x kappa2, f2x& s1, f2x& s2, float& t1, float& t2)
{
    f2x q1n = x2_dup(0.f), q2 = q1n;
    int m = lane;
#pragma unroll 4
    for (int s = 0; s < 16; ++s) {
        near_pair_x2<false, FAR>(T, F + m, F5 + m, q1n, sc, eps2, nieps2, kappa2, s1, s2, q1n, q2);
        q1n = x2_shfl_down1(q1n, lane);
        q2 = x2_shfl_down1(q2, lane);
        m = (m + 1) & 31;
    }
    // lane l: the low halves belong to source (l + 16) mod 32, the high halves to l
    float a1, b1, a2, b2;
    x2_unpack(q1n, a1, b1);
    x2_unpack(q2, a2, b2);
    t1 = -(b1 + __shfl_sync(0xffffffffu, a1, (lane + 16) & 31));
    t2 = b2 + __shfl_sync(0xffffffffu, a2, (lane + 16) & 31);
}

// a tile with fewer than 32 sources: lane j < nb gathers the reverse terms of source j by shuffles,
// in the order (step, low half before high half, lane), one FP32 sum per source. (Shared-memory
// atomics, four per step and lane, did this before; FP32 ones are compare-and-swap loops.)
template <bool FAR>
__device__ __forceinline__ void near_tile_part(const NearTgt2& T, const float4* F, const float2* F5, int lane, int nb,
                                               int na, bool act, f2x eps2, f2x nieps2, f2x kappa2, f2x& s1, f2x& s2,
                                               float& t1, float& t2)
{
    const float i4pi = 0.07957747154594767f;
    const int h = (nb + 1) >> 1;
    const f2x zero = x2_dup(0.f), sc = x2_dup(act ? i4pi : 0.f), scl = x2_pack(act ? i4pi : 0.f, 0.f);
    int m = lane % nb;
    // the lane that meets source `lane` in the low half at step s, and in the high half
    int p = m, ph = m - h < 0 ? m - h + nb : m - h;
    t1 = t2 = 0.f;
    for (int s = 0; s < h; ++s) {
        f2x q1n = zero, q2 = zero;
        // for odd nb the high half of the last step repeats a source: dropped
        near_pair_x2<false, FAR>(T, F + m, F5 + m, zero, (nb & 1) && s == h - 1 ? scl : sc, eps2, nieps2, kappa2, s1, s2,
                                 q1n, q2);
        float a1, b1, a2, b2;
        x2_unpack(q1n, a1, b1);
        x2_unpack(q2, a2, b2);
        for (int g = 0; g < na; g += nb) {
            const float v1 = __shfl_sync(0xffffffffu, a1, (p + g) & 31), v2 = __shfl_sync(0xffffffffu, a2, (p + g) & 31);
            if (p + g < 32) {
                t1 -= v1;
                t2 += v2;
            }
        }
        for (int g = 0; g < na; g += nb) {
            const float v1 = __shfl_sync(0xffffffffu, b1, (ph + g) & 31), v2 = __shfl_sync(0xffffffffu, b2, (ph + g) & 31);
            if (ph + g < 32) {
                t1 -= v1;
                t2 += v2;
            }
        }
        m = m + 1 == nb ? 0 : m + 1;
        p = p == 0 ? nb - 1 : p - 1;
        ph = ph == 0 ? nb - 1 : ph - 1;
    }
}

#define NEAR_FAR (1 << 30)  // flag of a tile (k_near_flag): kappa r >= 0.125 for all its pairs
#define NEAR_W 4            // warps per block
template <int Q2>
__global__ void __launch_bounds__(32 * NEAR_W, 7) k_near_tile(int nt, int nitems, const int4* __restrict__ items,
                                                    const int* __restrict__ tiles, const int* __restrict__ chunk_leaf,
                                                    const int* __restrict__ chunk_first, const int* __restrict__ begin,
                                                    const float4* __restrict__ sp, const float4* __restrict__ sn,
                                                    const float4* __restrict__ sl, double eps_d, double kappa_d,
                                                    double* __restrict__ ys)
{
    __shared__ float4 fq[NEAR_W][5 * 32];
    __shared__ float2 fq5[NEAR_W][32];
    const float i4pi = 0.07957747154594767f;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    if (w >= nitems) return;
    const int4 item = items[w];
    const int ca = item.x;
    const int c = chunk_leaf[ca], a0 = chunk_first[ca];
    const int na = min(32, begin[c + 1] - a0);
    const int k = a0 + lane;
    const bool act = lane < na;
    const int kk = act ? k : a0;
    NearTgt2 T;
    {
        const float4 tp = sp[kk], tn = sn[kk], tl = sl[kk];
        T.px = x2_dup(tp.x);
        T.py = x2_dup(tp.y);
        T.pz = x2_dup(tp.z);
        T.lx = x2_dup(tl.x);
        T.ly = x2_dup(tl.y);
        T.lz = x2_dup(tl.z);
        T.nx = x2_dup(tn.x);
        T.ny = x2_dup(tn.y);
        T.nz = x2_dup(tn.z);
        T.phi = x2_dup(act ? tp.w : 0.f);
        T.dphi = x2_dup(act ? tn.w : 0.f);
    }
    const f2x eps2 = x2_dup((float)eps_d), nieps2 = x2_dup((float)(-1.0 / eps_d)), kappa2 = x2_dup((float)kappa_d);
    const f2x zero = x2_dup(0.f);
    double acc1 = 0.0, acc2 = 0.0;
    float4* F = fq[wi];
    float2* F5 = fq5[wi];
    for (int ti = item.y; ti < item.z; ++ti) {
        const int tv = tiles[ti], cb = tv & (NEAR_FAR - 1);
        const int b0 = chunk_first[cb], se = begin[chunk_leaf[cb] + 1];
        const int nb = min(32, se - b0);
        if (nb <= 0) continue;  // no chunk is empty; the test keeps the indexing below in range
        const int h = (nb + 1) >> 1;
        // stage the tile: lane l < nb writes entry l = (source l, source (l + h) mod nb)
        {
            const int j = b0 + min(lane, nb - 1);
            const float4 p = sp[j], n = sn[j], lo = sl[j];
            int src = lane + h;
            if (src >= nb) src -= nb;
            if (lane >= nb) src = lane;
            const float Px = __shfl_sync(0xffffffffu, p.x, src), Py = __shfl_sync(0xffffffffu, p.y, src);
            const float Pz = __shfl_sync(0xffffffffu, p.z, src), Pw = __shfl_sync(0xffffffffu, p.w, src);
            const float Nx = __shfl_sync(0xffffffffu, n.x, src), Ny = __shfl_sync(0xffffffffu, n.y, src);
            const float Nz = __shfl_sync(0xffffffffu, n.z, src), Nw = __shfl_sync(0xffffffffu, n.w, src);
            const float Lx = __shfl_sync(0xffffffffu, lo.x, src), Ly = __shfl_sync(0xffffffffu, lo.y, src);
            const float Lz = __shfl_sync(0xffffffffu, lo.z, src);
            __syncwarp();
            if (lane < nb) {
                F[lane] = make_float4(p.x, Px, p.y, Py);
                F[32 + lane] = make_float4(p.z, Pz, p.w, Pw);
                F[64 + lane] = make_float4(n.x, Nx, n.y, Ny);
                F[96 + lane] = make_float4(n.z, Nz, -n.w, -Nw);
                F[128 + lane] = make_float4(lo.x, Lx, lo.y, Ly);
                F5[lane] = make_float2(lo.z, Lz);
            }
            __syncwarp();
        }
        f2x s1 = zero, s2 = zero;
        if (cb == ca) {
            // the chunk with itself: forward terms only, without the identical pair (the
            // correction's) or the pairs of one element's points
            int m = lane % nb;
            int m2 = m + h;
            if (m2 >= nb) m2 -= nb;
            const bool odd = nb & 1;
            for (int s = 0; s < h; ++s) {
                const bool okl = act && !(Q2 == 1 ? m == lane : m / Q2 == lane / Q2);
                const bool okh = act && !(odd && s == h - 1) && !(Q2 == 1 ? m2 == lane : m2 / Q2 == lane / Q2);
                f2x q1n = zero, q2 = zero;
                near_pair_x2<true, false>(T, F + m, F5 + m, x2_pack(okl ? 0.f : 1.f, okh ? 0.f : 1.f),
                                          x2_pack(okl ? i4pi : 0.f, okh ? i4pi : 0.f), eps2, nieps2, kappa2, s1, s2, q1n,
                                          q2);
                m = m + 1 == nb ? 0 : m + 1;
                m2 = m2 + 1 == nb ? 0 : m2 + 1;
            }
        } else {
            float t1, t2;
            if (nb == 32) {
                const f2x sc = x2_dup(act ? i4pi : 0.f);
                if (tv & NEAR_FAR) near_tile_full<true>(T, F, F5, lane, sc, eps2, nieps2, kappa2, s1, s2, t1, t2);
                else near_tile_full<false>(T, F, F5, lane, sc, eps2, nieps2, kappa2, s1, s2, t1, t2);
            } else {
                if (tv & NEAR_FAR) near_tile_part<true>(T, F, F5, lane, nb, na, act, eps2, nieps2, kappa2, s1, s2, t1, t2);
                else near_tile_part<false>(T, F, F5, lane, nb, na, act, eps2, nieps2, kappa2, s1, s2, t1, t2);
            }
            if (lane < nb) {
                atomicAdd(&ys[b0 + lane], (double)t1);
                atomicAdd(&ys[nt + b0 + lane], (double)t2);
            }
        }
        float a, b;
        x2_unpack(s1, a, b);
        acc1 += (double)(a + b);
        x2_unpack(s2, a, b);
        acc2 += (double)(a + b);
    }
    if (act) {
        atomicAdd(&ys[k], acc1);
        atomicAdd(&ys[nt + k], acc2);
    }
}

// Build: bounding box of every chunk's centres (or points), one warp per chunk
__global__ void k_chunk_box(int nchunks, const int* __restrict__ chunk_leaf, const int* __restrict__ chunk_first,
                            const int* __restrict__ begin, const double4_32a* __restrict__ ep, double* __restrict__ box)
{
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= nchunks) return;
    const int k = min(chunk_first[c] + lane, begin[chunk_leaf[c] + 1] - 1);
    const double4_32a p = ep[k];
    double lo[3] = {p.x, p.y, p.z}, hi[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int a = 0; a < 3; ++a)
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fmin(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmax(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    if (lane < 3) box[6 * (size_t)c + lane] = lane == 0 ? lo[0] : lane == 1 ? lo[1] : lo[2];
    else if (lane < 6) box[6 * (size_t)c + lane] = lane == 3 ? hi[0] : lane == 4 ? hi[1] : hi[2];
}

// Build: NEAR_FAR on the tiles whose chunks' boxes are at least 0.125 / kappa apart, with a margin
// of 1e-5 for the FP32 rounding of kappa r in the kernel; one thread per work item
__global__ void k_near_flag(int nitems, const int4* __restrict__ items, const double* __restrict__ box, double kappa,
                            int* __restrict__ tiles)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nitems) return;
    const int4 item = items[w];
    const double* A = box + 6 * (size_t)item.x;
    for (int t = item.y; t < item.z; ++t) {
        const int cb = tiles[t] & (NEAR_FAR - 1);
        const double* B = box + 6 * (size_t)cb;
        double d2 = 0.0;
        for (int a = 0; a < 3; ++a) {
            const double d = fmax(0.0, fmax(A[a] - B[3 + a], B[a] - A[3 + a]));
            d2 += d * d;
        }
        tiles[t] = cb | (kappa * sqrt(d2) >= 0.125 * (1.0 + 1e-5) ? NEAR_FAR : 0);
    }
}

static int near_flags(pb_ctx* c, int nchunks, const int* chunk_leaf, const int* chunk_first, const int* begin,
                      const double4_32a* ep, int nitems, const int4* items, int* tiles)
{
    double* box = (double*)pb_alloc(c, sizeof(double) * 6 * (size_t)nchunks);
    if (!box) return pb_fail(c, PB_ERR_NOMEM, "near setup: out of memory");
    k_chunk_box<<<(unsigned)(((long long)nchunks * 32 + 255) / 256), 256, 0, c->st>>>(nchunks, chunk_leaf, chunk_first,
                                                                                        begin, ep, box);
    PB_LAUNCH(c);
    k_near_flag<<<(nitems + 127) / 128, 128, 0, c->st>>>(nitems, items, box, c->prm.kappa, tiles);
    PB_LAUNCH(c);
    return PB_OK;
}

// ---------- several right-hand sides at once (mixed precision) ----------
// The pair kernels depend on the geometry only, so one evaluation serves NR densities: the
// source's geometry records are loaded once per pair and each right-hand side adds four FMAs.
// dens[r nt + j] = (A_j phi_j, A_j dphi_j) of right-hand side r.
// (and, as k_near_pack, the tree-ordered copy of an element-ordered vector and zero sums)
__global__ void k_near_dens(int nt, const float4* __restrict__ e32p, const int* __restrict__ order,
                            const double* __restrict__ x, double* __restrict__ xs, float2* __restrict__ dens,
                            double* __restrict__ ys)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    const double A = (double)e32p[k].w;
    const long long o = 2LL * nt * blockIdx.y;
    const int e = order ? order[k] : k;
    const double v1 = x[o + e], v2 = x[o + nt + e];
    if (order) {
        xs[o + k] = v1;
        xs[o + nt + k] = v2;
    }
    ys[o + k] = 0.0;
    ys[o + nt + k] = 0.0;
    dens[(size_t)nt * blockIdx.y + k] = make_float2((float)(A * v1), (float)(A * v2));
}

// Work items of at most NEAR_ITEM_M directed tiles (target chunk A, source chunk B of any
// neighbour leaf), one warp each; the item's sums are added into ys (zeroed first) with FP64
// atomics, so that items of one target chunk may run on different warps. Each tile's source
// records and its NR densities are staged in shared memory by coalesced loads (one per lane
// and record), so the pair loop reads them as shared-memory broadcasts. Two densities (r, r + 1) are
// the halves of packed FP32 pairs in the four FMAs per density. A tile's FP32 sums go into FP64
// accumulators, a conversion and an addition per value at 1/64 of the FP32 rate: float-float ones (2^-48)
// save 70 us of 2360 per product of 16 densities on 81,920 elements, but are less than FP64 and change
// last bits of products; conversions by integer operations gain nothing (2390 us).
template <int NR>
struct NearM {
    static constexpr int H = (NR + 1) / 2;  // pairs of densities
    static constexpr size_t smem = 8 * 32 * (3 * sizeof(float4) + H * sizeof(float4) + 4 * H * sizeof(f2x));
};

// the pairs of one tile: s1, s2 += per density pair
template <int NR, bool FAR>
__device__ __forceinline__ void near_m_tile(const float4 tp, const float4 tn, const float4 tl,
                                            const float4* __restrict__ s_p, const float4* __restrict__ s_n,
                                            const float4* __restrict__ s_l, const float4* __restrict__ s_d, int nb, int self,
                                            float eps, float inv_eps, float kappa, f2x* s1, f2x* s2)
{
#pragma unroll 2
    for (int q = 0; q < nb; ++q) {
        const float4 a = s_p[q], b = s_n[q], l = s_l[q];
        float K[4];
        float dx = (tp.x - a.x) + (tl.x - l.x);
        float dy = (tp.y - a.y) + (tl.y - l.y);
        float dz = (tp.z - a.z) + (tl.z - l.z);
        if (!FAR && q == self) dx = 1.0f;  // the identical pair is the correction's; keep r finite
        pb_kernels<float, FAR>(dx, dy, dz, tn.x, tn.y, tn.z, b.x, b.y, b.z, eps, inv_eps, kappa, K,
                               (!FAR && q == self) ? 0.f : 1.f);
        const f2x k0 = x2_dup(K[0]), k1 = x2_dup(K[1]), k2 = x2_dup(K[2]), k3 = x2_dup(K[3]);
#pragma unroll
        for (int h = 0; h < NearM<NR>::H; ++h) {
            const float4 d = s_d[h * 32 + q];
            const f2x x = x2_pack(d.x, d.y), y = x2_pack(d.z, d.w);
            s1[h] = x2_fma(k0, y, x2_fma(k1, x, s1[h]));
            s2[h] = x2_fma(k2, y, x2_fma(k3, x, s2[h]));
        }
    }
}

template <int NR>
__global__ void __launch_bounds__(256, 2) k_near32m(int nt, int nitems, const int4* __restrict__ items,
                                                    const int* __restrict__ tiles, const int* __restrict__ chunk_leaf,
                                                    const int* __restrict__ chunk_first,
                                                    const int* __restrict__ begin, const float4* __restrict__ sp,
                                                    const float4* __restrict__ sn, const float4* __restrict__ sl,
                                                    const float2* __restrict__ dens, double eps_d, double kappa_d,
                                                    double* __restrict__ ys, int nvalid)
{
    // dynamic shared memory: per warp the tile's source records, its densities in pairs, and the
    // item's float-float sums (kept here rather than in registers)
    constexpr int H = NearM<NR>::H;
    extern __shared__ __align__(16) unsigned char nsm[];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    float4* s_p = (float4*)nsm + wi * 32;
    float4* s_n = (float4*)nsm + 256 + wi * 32;
    float4* s_l = (float4*)nsm + 512 + wi * 32;
    float4* s_d = (float4*)nsm + 768 + wi * H * 32;                           // (x_r, x_r+1, y_r, y_r+1)
    double* s_acc = (double*)((float4*)nsm + 768 + 8 * H * 32) + wi * 4 * H * 32;  // [density][half of the row][lane]
    if (w >= nitems) return;
    const int4 item = items[w];
    const int c = chunk_leaf[item.x];
    const int k = chunk_first[item.x] + lane;
    const bool act = k < begin[c + 1];
    const int kk = act ? k : chunk_first[item.x];
    const float4 tp = sp[kk], tn = sn[kk], tl = sl[kk];
    const float eps = (float)eps_d, inv_eps = (float)(1.0 / eps_d), kappa = (float)kappa_d;
#pragma unroll
    for (int r = 0; r < 4 * H; ++r) s_acc[r * 32 + lane] = 0.0;
    for (int ti = item.y; ti < item.z; ++ti) {
        const int tv = tiles[ti], cb = tv & (NEAR_FAR - 1);
        const int sb = chunk_first[cb], se = min(sb + 32, begin[chunk_leaf[cb] + 1]);
        const int nb = se - sb;
        __syncwarp();
        if (lane < nb) {
            const int j = sb + lane;
            s_p[lane] = sp[j];
            s_n[lane] = sn[j];
            s_l[lane] = sl[j];
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const float2 d0 = dens[(size_t)nt * (2 * h) + j];
                const float2 d1 = NR > 1 ? dens[(size_t)nt * (2 * h + 1) + j] : make_float2(0.f, 0.f);
                s_d[h * 32 + lane] = make_float4(d0.x, d1.x, d0.y, d1.y);
            }
        }
        __syncwarp();
        f2x s1[H], s2[H];
#pragma unroll
        for (int h = 0; h < H; ++h) s1[h] = s2[h] = 0ull;
        if (tv & NEAR_FAR) near_m_tile<NR, true>(tp, tn, tl, s_p, s_n, s_l, s_d, nb, -1, eps, inv_eps, kappa, s1, s2);
        else near_m_tile<NR, false>(tp, tn, tl, s_p, s_n, s_l, s_d, nb, k - sb, eps, inv_eps, kappa, s1, s2);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            double* a = s_acc + 4 * h * 32 + lane;
            float v[4];
            x2_unpack(s1[h], v[0], v[2]);
            x2_unpack(s2[h], v[1], v[3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) a[32 * u] += (double)(v[u]);
        }
    }
    // densities beyond nvalid are padding of the group (finite, unused): only nvalid are added
    if (act)
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < nvalid) {
                atomicAdd(&ys[2LL * nt * r + k], s_acc[2 * r * 32 + lane]);
                atomicAdd(&ys[2LL * nt * r + nt + k], s_acc[(2 * r + 1) * 32 + lane]);
            }
}

// What ends a product. ep: ys holds the mixed near field's bare sums, which become
// y1 = 1/2 (1 + eps) A phi - A acc1, y2 = 1/2 (1 + 1/eps) A dphi - A acc2 (nullptr: ys holds rows);
// yf: the far-field part to add (or nullptr); order: the result goes to y[order[k]] in element
// order, else to y[k] in tree order.
struct MvEnd {
    int nt;
    const double4_32a* ep;
    double eps;
    const double *xs, *ys, *yf;
    const int* order;
    double* y;
};
// The roundings of a row are written out: contracted as the compiler likes, the same expressions in another
// kernel differ in the last bit, and the FP32 preconditioner, which rounds its input, carries one such bit
// on as a whole FP32 ulp of single entries of a solution (1e-7 of its maximum).
// f A x - A s
__device__ __forceinline__ double mass_row(double f, double A, double x, double s)
{
    return __fma_rn(__dmul_rn(f, A), x, -__dmul_rn(A, s));
}
__device__ __forceinline__ void mv_end(const MvEnd& m, long long o, int k, double c1, double c2)
{
    double a = m.ys[o + k], b = m.ys[o + m.nt + k];
    if (m.ep) {
        const double A = m.ep[k].w;
        a = mass_row(0.5 * (1.0 + m.eps), A, m.xs[o + k], a);
        b = mass_row(0.5 * (1.0 + 1.0 / m.eps), A, m.xs[o + m.nt + k], b);
    }
    if (m.yf) {
        c1 -= m.yf[o + k];
        c2 -= m.yf[o + m.nt + k];
    }
    const int e = m.order ? m.order[k] : k;
    m.y[o + e] = a - c1;
    m.y[o + m.nt + e] = b - c2;
}

// Sauter-Schwab corrections of identical and adjacent pairs (FP64), and the end of the product.
// One warp per 32 rows: their pairs (about 13 per row, one after the other in memory) are read as one
// coalesced stream, 512 at a time with all loads independent, the products go through shared
// memory and each lane adds its own row in order. Bound: the 36 bytes per pair from HBM (or
// L2). A thread that walked its own row took 14 us on 1280 elements, 24.5 on 81,920 and 124 on
// 737,280 (3.3 TB/s), the end of the product 4, 6 and 24 more; now 12, 24 and 142 us for
// both (the FP64 pipe is a bound too: six operations per pair, 93 us at 737,280).
#define CORR_W 4
#define CORR_B 512
__global__ void __launch_bounds__(32 * CORR_W) k_corrections(const int* __restrict__ toff, const int* __restrict__ tj,
                                                             const double* __restrict__ corr, MvEnd m)
{
    __shared__ double s1[CORR_W][CORR_B], s2[CORR_W][CORR_B];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt = m.nt;
    const int k0 = (blockIdx.x * CORR_W + w) * 32, k = k0 + lane;
    if (k0 >= nt) return;
    const int t0 = toff[min(k, nt)], t1 = toff[min(k + 1, nt)];
    const int e0 = __shfl_sync(0xffffffffu, t0, 0), e1 = __shfl_sync(0xffffffffu, t1, 31);
    const double2* c2 = reinterpret_cast<const double2*>(corr);
    double y1 = 0.0, y2 = 0.0;
    for (int base = e0; base < e1; base += CORR_B) {
        const int n = min(CORR_B, e1 - base);
#pragma unroll 4
        for (int i = lane; i < n; i += 32) {
            const int t = base + i, j = tj[t];
            const double2 a = c2[2 * (size_t)t], b = c2[2 * (size_t)t + 1];
            const double ph = m.xs[j], dph = m.xs[nt + j];
            s1[w][i] = __fma_rn(a.x, dph, __dmul_rn(a.y, ph));
            s2[w][i] = __fma_rn(b.x, dph, __dmul_rn(b.y, ph));
        }
        __syncwarp();
        for (int i = max(t0 - base, 0); i < min(t1 - base, n); ++i) {
            y1 += s1[w][i];
            y2 += s2[w][i];
        }
        __syncwarp();
    }
    if (k < nt) mv_end(m, 0, k, y1, y2);
}

// the far-field part alone, for any number of vectors
__global__ void k_mv_end(MvEnd m)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < m.nt) mv_end(m, 2LL * m.nt * blockIdx.y, k, 0.0, 0.0);
}

// Work items of the pair-tile kernel: the tiles (A, B), B a chunk of a neighbour leaf c2 >= leaf(A)
// and B >= A, cut into items of n tiles that share A. An item costs its targets' load and two
// FP64 atomics per lane, as much as a fraction of a tile; too few items leave the GPU's 152 x 24
// warps idle at the end. n = 6 where every warp gets eight items or more, fewer below (81,920
// elements: 72,000 tiles, n = 2: 178 -> 166 us; 1280: 820 tiles, n = 1: 27 -> 12 us).
static void near_pair_items(int ncl, const std::vector<int>& first_chunk, const std::vector<int>& no,
                            const std::vector<int>& ni, std::vector<int>& tl, std::vector<int4>& it)
{
    std::vector<int> start;  // first tile of each chunk
    for (int k = 0; k < ncl; ++k)
        for (int a = first_chunk[k]; a < first_chunk[k + 1]; ++a) {
            start.push_back((int)tl.size());
            for (int t = no[k]; t < no[k + 1]; ++t) {
                const int c2 = ni[t];
                if (c2 < k) continue;
                for (int bq = (c2 == k ? a : first_chunk[c2]); bq < first_chunk[c2 + 1]; ++bq) tl.push_back(bq);
            }
        }
    start.push_back((int)tl.size());
    const int n = std::max(1, std::min(NEAR_ITEM, (int)(tl.size() / (152 * 24 * 8))));
    for (size_t a = 0; a + 1 < start.size(); ++a)
        for (int t = start[a]; t < start[a + 1]; t += n)
            it.push_back(make_int4((int)a, t, std::min(t + n, start[a + 1]), 0));
}

// chunks of at most 32 targets per leaf and the packed source buffers (mixed precision)
int pb_near_setup(pb_ctx* c)
{
    // (with a regular rule of order > 1 the FP64 near field runs on its points, pb_near_q_apply)
    if (c->prm.precision != PB_MIXED) return c->q2 > 1 ? PB_OK : near64_setup(c);
    const PbLevel& lv = c->lev[c->L];
    const std::vector<int>& b = c->h_leaf_begin;  // the leaf ranges, read back by the tree build
    std::vector<int>& cl = c->h_up_i[0];
    std::vector<int>& cf = c->h_up_i[1];
    cl.clear();
    cf.clear();
    for (int k = 0; k < lv.ncl; ++k)
        for (int s = b[k]; s < b[k + 1]; s += 32) {
            cl.push_back(k);
            cf.push_back(s);
        }
    c->nchunks = (int)cl.size();
    {
        std::vector<int> first_chunk(lv.ncl + 1, 0);
        for (int k = 0; k < lv.ncl; ++k) first_chunk[k + 1] = first_chunk[k] + (b[k + 1] - b[k] + 31) / 32;
        std::vector<int>& tl = c->h_up_i[4];
        std::vector<int4>& it = c->h_up_i4;
        tl.clear();
        it.clear();
        const std::vector<int>& no = c->h_near_off;
        const std::vector<int>& ni = c->h_near_idx;
        near_pair_items(lv.ncl, first_chunk, no, ni, tl, it);
        c->near_nitems = (int)it.size();
        c->near_mitems = 0;  // the several-vector items are made on first use (pb_near_reserve)
        c->near_mitem = nullptr;
        c->near_mtiles = nullptr;
        c->near_items = (int4*)pb_alloc(c, sizeof(int4) * (it.size() + 1));
        c->near_tiles = (int*)pb_alloc(c, sizeof(int) * (tl.size() + 1));
        if (!c->near_items || !c->near_tiles) return pb_fail(c, PB_ERR_NOMEM, "near setup: out of memory");
        PB_CUDA(c, cudaMemcpyAsync(c->near_items, it.data(), sizeof(int4) * it.size(), cudaMemcpyHostToDevice, c->st));
        PB_CUDA(c, cudaMemcpyAsync(c->near_tiles, tl.data(), sizeof(int) * tl.size(), cudaMemcpyHostToDevice, c->st));
    }
    c->chunk_leaf = (int*)pb_alloc(c, sizeof(int) * cl.size());
    c->chunk_first = (int*)pb_alloc(c, sizeof(int) * cf.size());
    c->near_sp = (float4*)pb_alloc(c, sizeof(float4) * c->nt);
    c->near_sn = (float4*)pb_alloc(c, sizeof(float4) * c->nt);
    if (!c->chunk_leaf || !c->chunk_first || !c->near_sp || !c->near_sn)
        return pb_fail(c, PB_ERR_NOMEM, "near setup: out of memory");
    PB_CUDA(c, cudaMemcpyAsync(c->chunk_leaf, cl.data(), sizeof(int) * cl.size(), cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->chunk_first, cf.data(), sizeof(int) * cf.size(), cudaMemcpyHostToDevice, c->st));
    return near_flags(c, c->nchunks, c->chunk_leaf, c->chunk_first, lv.begin, c->e64p, c->near_nitems, c->near_items,
                      c->near_tiles);
}

// Mixed precision, one-point rule: before the near field of nr vectors, the packed densities and
// zero sums; xin: the vectors in element order (xs is then written), or nullptr.
int pb_near_pack(pb_ctx* c, const double* xin, double* xs, double* ys, int nr)
{
    const int nt = c->nt;
    const int* order = xin ? c->order : nullptr;
    const double* x = xin ? xin : xs;
    if (nr == 1) {
        k_near_pack<<<(nt + 255) / 256, 256, 0, c->st>>>(nt, c->e32p, c->e32n, order, x, xs, c->near_sp, c->near_sn, ys);
    } else {
        int rc = pb_near_reserve(c, nr);
        if (rc) return rc;
        k_near_dens<<<dim3((nt + 255) / 256, nr), 256, 0, c->st>>>(nt, c->e32p, order, x, xs, c->near_dens, ys);
    }
    PB_LAUNCH(c);
    return PB_OK;
}

// one vector; mixed: adds the bare sums into ys (after pb_near_pack), FP64: writes the rows
int pb_near_apply(pb_ctx* c, const double* xs, double* ys)
{
    const PbLevel& lv = c->lev[c->L];
    double eps = c->prm.eps_out / c->prm.eps_in;
    if (c->prm.precision == PB_MIXED) {
        k_near_tile<1><<<(c->near_nitems + NEAR_W - 1) / NEAR_W, 32 * NEAR_W, 0, c->st>>>(
            c->nt, c->near_nitems, c->near_items, c->near_tiles, c->chunk_leaf, c->chunk_first, lv.begin, c->near_sp,
            c->near_sn, c->e32l, eps, c->prm.kappa, ys);
    } else {
        Near64Tiles q = {c->near64_base, c->near64_first, lv.near_off, lv.near_idx, c->near64_pos, 0, 0};
        const std::vector<int>& cut = c->near64_cut;
        const std::vector<long long>& base = c->h_up_l64;
        for (size_t i = 0; i + 1 < cut.size(); ++i) {
            q.a0 = cut[i];
            q.a1 = cut[i + 1];
            const long long tiles = base[q.a1] - base[q.a0];
            k_near64<<<(unsigned)((tiles + 7) / 8), 256, 0, c->st>>>(c->nt, q, c->chunk_leaf, c->chunk_first, lv.begin,
                                                                     c->e64p, c->e64n, xs, eps, c->prm.kappa, c->near_part);
            PB_LAUNCH(c);
            k_near64_sum<<<(c->nchunks + 7) / 8, 256, 0, c->st>>>(c->nt, c->nchunks, q, c->chunk_leaf, c->chunk_first,
                                                                  lv.begin, c->e64p, c->near_part, xs, eps, i == 0,
                                                                  i + 2 == cut.size(), ys);
            PB_LAUNCH(c);
        }
        return PB_OK;
    }
    PB_LAUNCH(c);
    return PB_OK;
}

// Several right-hand sides: four per thread (blockIdx.y = group of four), so each correction
// is read once per four vectors instead of once per vector. Bound: the FP64 pipe, six operations per
// pair and vector (16 vectors on 81,920 elements: 236 us; chains of FMA, four operations, took 158 us, but
// round each row otherwise, and single entries of a batched solution then move by an FP32 ulp).
__global__ void k_corrections4(int nr, const int* __restrict__ toff, const int* __restrict__ tj,
                               const double* __restrict__ corr, MvEnd m)
{
    const int nt = m.nt;
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    const int q0 = 4 * blockIdx.y, nq = min(4, nr - q0);
    const long long vs = 2LL * nt;
    double y1[4] = {0, 0, 0, 0}, y2[4] = {0, 0, 0, 0};
    for (int t = toff[k]; t < toff[k + 1]; ++t) {
        const int j = tj[t];
        const double2 a = reinterpret_cast<const double2*>(corr)[2 * t];
        const double2 b = reinterpret_cast<const double2*>(corr)[2 * t + 1];
        const double c0 = a.x, c1 = a.y, c2 = b.x, c3 = b.y;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < nq) {
                const double* x = m.xs + (q0 + q) * vs;
                const double ph = x[j], dph = x[nt + j];
                y1[q] = __dadd_rn(y1[q], __fma_rn(c1, ph, __dmul_rn(c0, dph)));
                y2[q] = __dadd_rn(y2[q], __fma_rn(c3, ph, __dmul_rn(c2, dph)));
            }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nq) mv_end(m, (q0 + q) * vs, k, y1[q], y2[q]);
}

// corrections (with xs; without: the far field alone), far-field part and end of the product of nr
// vectors into y: in element order, or in tree order. sums: ys holds bare near-field sums.
int pb_corr_apply(pb_ctx* c, const double* xs, const double* ys, int nr, const double* yfar, bool sums, bool element_order,
                  double* y)
{
    const int nt = c->nt;
    const MvEnd m = {nt, sums ? c->e64p : nullptr, c->prm.eps_out / c->prm.eps_in, xs, ys, yfar,
                     element_order ? c->order : nullptr, y};
    if (!xs)
        k_mv_end<<<dim3((nt + 255) / 256, nr), 256, 0, c->st>>>(m);
    else if (nr > 1)
        k_corrections4<<<dim3((nt + 255) / 256, (nr + 3) / 4), 256, 0, c->st>>>(nr, c->touch_off, c->touch_j, c->corr, m);
    else
        k_corrections<<<(nt + 32 * CORR_W - 1) / (32 * CORR_W), 32 * CORR_W, 0, c->st>>>(c->touch_off, c->touch_j, c->corr,
                                                                                        m);
    PB_LAUNCH(c);
    return PB_OK;
}

template <int NR>
static int near_multi_launch(pb_ctx* c, const float2* dens, double* ys, double eps, int nvalid)
{
    const PbLevel& lv = c->lev[c->L];
    PB_CUDA(c, cudaFuncSetAttribute(k_near32m<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)NearM<NR>::smem));
    k_near32m<NR><<<(c->near_mitems * 32 + 255) / 256, 256, NearM<NR>::smem, c->st>>>(
        c->nt, c->near_mitems, c->near_mitem, c->near_mtiles, c->chunk_leaf, c->chunk_first, lv.begin, c->e32p,
        c->e32n, c->e32l, dens, eps, c->prm.kappa, ys, nvalid);
    PB_LAUNCH(c);
    return PB_OK;
}

// directed tiles for the several-vector kernel: every chunk of every neighbour leaf, cut into
// work items of at most NEAR_ITEM_M tiles of one target chunk
static int near_multi_items(pb_ctx* c)
{
    const PbLevel& lv = c->lev[c->L];
    const std::vector<int>& b = c->h_leaf_begin;
    const std::vector<int>& no = c->h_near_off;
    const std::vector<int>& ni = c->h_near_idx;
    std::vector<int> first_chunk(lv.ncl + 1, 0);
    for (int k = 0; k < lv.ncl; ++k) first_chunk[k + 1] = first_chunk[k] + (b[k + 1] - b[k] + 31) / 32;
    std::vector<int>& tm = c->h_up_i[5];
    std::vector<int4>& im = c->h_up_i4m;
    tm.clear();
    im.clear();
    for (int k = 0; k < lv.ncl; ++k)
        for (int a = first_chunk[k]; a < first_chunk[k + 1]; ++a) {
            int start = (int)tm.size();
            for (int t = no[k]; t < no[k + 1]; ++t)
                for (int bq = first_chunk[ni[t]]; bq < first_chunk[ni[t] + 1]; ++bq) {
                    tm.push_back(bq);
                    if ((int)tm.size() - start == NEAR_ITEM_M) {
                        im.push_back(make_int4(a, start, (int)tm.size(), 0));
                        start = (int)tm.size();
                    }
                }
            if ((int)tm.size() > start) im.push_back(make_int4(a, start, (int)tm.size(), 0));
        }
    c->near_mitems = (int)im.size();
    c->near_mitem = (int4*)pb_alloc(c, sizeof(int4) * (im.size() + 1));
    c->near_mtiles = (int*)pb_alloc(c, sizeof(int) * (tm.size() + 1));
    if (!c->near_mitem || !c->near_mtiles) return pb_fail(c, PB_ERR_NOMEM, "near setup: out of memory");
    PB_CUDA(c, cudaMemcpyAsync(c->near_mitem, im.data(), sizeof(int4) * im.size(), cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->near_mtiles, tm.data(), sizeof(int) * tm.size(), cudaMemcpyHostToDevice, c->st));
    return near_flags(c, c->nchunks, c->chunk_leaf, c->chunk_first, lv.begin, c->e64p, c->near_mitems, c->near_mitem,
                      c->near_mtiles);
}

// density buffer of the multi-vector near field and its work items (build lifetime, grown on
// demand)
int pb_near_reserve(pb_ctx* c, int nr)
{
    if (c->prm.precision != PB_MIXED || nr < 2) return PB_OK;
    if (!c->near_mitem) {
        int rc = near_multi_items(c);
        if (rc) return rc;
    }
    if (nr <= c->dens_nr) return PB_OK;
    nr = (nr + 15) / 16 * 16;  // groups read whole padded widths
    c->near_dens = (float2*)pb_alloc(c, sizeof(float2) * (size_t)c->nt * nr);
    if (!c->near_dens) return pb_fail(c, PB_ERR_NOMEM, "near field: out of memory");
    c->dens_nr = nr;
    return PB_OK;
}

// nr right-hand sides: xs and ys hold nr vectors of 2 nt (mixed: bare sums, after pb_near_pack); mixed
// precision evaluates each pair once for up to 16 of them, FP64 applies the single-vector kernel per right-hand side
int pb_near_apply_multi(pb_ctx* c, const double* xs, double* ys, int nr)
{
    const int nt = c->nt;
    const double eps = c->prm.eps_out / c->prm.eps_in;
    if (c->prm.precision != PB_MIXED) {
        for (int r = 0; r < nr; ++r) {
            int rc = pb_near_apply(c, xs + 2LL * nt * r, ys + 2LL * nt * r);
            if (rc) return rc;
        }
        return PB_OK;
    }
    // groups of up to 16 right-hand sides, each one launch of the smallest width that holds it
    // (the density buffer is padded to a multiple of 16 vectors)
    for (int r0 = 0; r0 < nr;) {
        const int v = std::min(16, nr - r0);
        const int g = v > 8 ? 16 : v > 4 ? 8 : v > 2 ? 4 : v > 1 ? 2 : 1;
        const float2* d = c->near_dens + (size_t)nt * r0;
        double* y = ys + 2LL * nt * r0;
        const int rc = g == 16  ? near_multi_launch<16>(c, d, y, eps, v)
                       : g == 8 ? near_multi_launch<8>(c, d, y, eps, v)
                       : g == 4 ? near_multi_launch<4>(c, d, y, eps, v)
                       : g == 2 ? near_multi_launch<2>(c, d, y, eps, v)
                                : near_multi_launch<1>(c, d, y, eps, v);
        if (rc) return rc;
        r0 += v;
    }
    return PB_OK;
}

// ---------- the near field on the points of a regular rule (mixed precision) ----------
// The same pair-tile kernel over the q2 points of every element (q2 = 4 or 16), so the order-q
// rule's near field (both bases) runs at the element kernel's rate: point chunks of 32 within
// each leaf's point range, the tiles of the element plan's neighbour lists, FP32 hi/lo point
// records built once per build.
__global__ void k_pts32(long long np, const double4_32a* __restrict__ pp, const double4_32a* __restrict__ pn,
                        float4* __restrict__ p32, float4* __restrict__ l32, float4* __restrict__ n32)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double4_32a x = pp[p], n = pn[p];
    const float hx = (float)x.x, hy = (float)x.y, hz = (float)x.z;
    p32[p] = make_float4(hx, hy, hz, (float)x.w);
    l32[p] = make_float4((float)(x.x - (double)hx), (float)(x.y - (double)hy), (float)(x.z - (double)hz), 0.f);
    n32[p] = make_float4((float)n.x, (float)n.y, (float)n.z, 0.f);
}

// point records with densities: W_p times the point's values, from the element values xs
// (piecewise constant: every point of element p / q2) or from per-point values xq
__global__ void k_pts_pack(long long np, int q2, int nt, const float4* __restrict__ p32, const float4* __restrict__ n32,
                           const double4_32a* __restrict__ pp, const double* __restrict__ xs,
                           const double* __restrict__ xq, float4* __restrict__ sp, float4* __restrict__ sn)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double W = pp[p].w;
    double u1, u2;
    if (xq) {
        u1 = xq[p];
        u2 = xq[np + p];
    } else {
        const int k = (int)(p / q2);
        u1 = xs[k];
        u2 = xs[nt + k];
    }
    const float4 a = p32[p], b = n32[p];
    sp[p] = make_float4(a.x, a.y, a.z, (float)(W * u1));
    sn[p] = make_float4(b.x, b.y, b.z, (float)(W * u2));
}

// ys[k] = mass - sum over element k's points of W_a y_a (both halves), y the point sums
__global__ void k_pts_finish_elem(int nt, int q2, const double4_32a* __restrict__ ep,
                                  const double4_32a* __restrict__ pp, const double* __restrict__ xs,
                                  const double* __restrict__ ypt, double eps, double* __restrict__ ys)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    const long long np = (long long)nt * q2;
    double s1 = 0.0, s2 = 0.0;
    for (int a = 0; a < q2; ++a) {
        const long long p = (long long)k * q2 + a;
        const double W = pp[p].w;
        s1 += W * ypt[p];
        s2 += W * ypt[np + p];
    }
    const double A = ep[k].w;
    ys[k] = 0.5 * (1.0 + eps) * A * xs[k] - s1;
    ys[nt + k] = 0.5 * (1.0 + 1.0 / eps) * A * xs[nt + k] - s2;
}

bool pb_near_points_ok(const pb_ctx* c) { return c->prm.precision == PB_MIXED && (c->q2 == 4 || c->q2 == 16); }

int pb_near_points_setup(pb_ctx* c)
{
    if (!pb_near_points_ok(c)) return PB_OK;
    const PbLevel& lv = c->lev[c->L];
    const int q2 = c->q2;
    const long long np = (long long)c->nt * q2;
    const std::vector<int>& b = c->h_leaf_begin;
    std::vector<int> cl, cf, tl;
    std::vector<int4> it;
    std::vector<int> first_chunk(lv.ncl + 1, 0);
    for (int k = 0; k < lv.ncl; ++k) {
        const long long s0 = (long long)b[k] * q2, s1 = (long long)b[k + 1] * q2;
        for (long long s = s0; s < s1; s += 32) {
            cl.push_back(k);
            cf.push_back((int)s);
        }
        first_chunk[k + 1] = (int)cl.size();
    }
    const std::vector<int>& no = c->h_near_off;
    const std::vector<int>& ni = c->h_near_idx;
    near_pair_items(lv.ncl, first_chunk, no, ni, tl, it);
    c->pn_nitems = (int)it.size();
    c->h_pn_i[0].swap(cl);
    c->h_pn_i[1].swap(cf);
    c->h_pn_i[2].swap(tl);
    c->h_pn_i4.swap(it);
    c->pn_items = (int4*)pb_alloc(c, sizeof(int4) * (c->h_pn_i4.size() + 1));
    c->pn_tiles = (int*)pb_alloc(c, sizeof(int) * (c->h_pn_i[2].size() + 1));
    c->pn_chunk_leaf = (int*)pb_alloc(c, sizeof(int) * (c->h_pn_i[0].size() + 1));
    c->pn_chunk_first = (int*)pb_alloc(c, sizeof(int) * (c->h_pn_i[1].size() + 1));
    c->pn_begin = (int*)pb_alloc(c, sizeof(int) * (lv.ncl + 1));
    c->pn_p32 = (float4*)pb_alloc(c, sizeof(float4) * np);
    c->pn_l32 = (float4*)pb_alloc(c, sizeof(float4) * np);
    c->pn_n32 = (float4*)pb_alloc(c, sizeof(float4) * np);
    c->pn_sp = (float4*)pb_alloc(c, sizeof(float4) * np);
    c->pn_sn = (float4*)pb_alloc(c, sizeof(float4) * np);
    c->pn_y = (double*)pb_alloc(c, sizeof(double) * 2 * np);
    if (!c->pn_items || !c->pn_tiles || !c->pn_chunk_leaf || !c->pn_chunk_first || !c->pn_begin || !c->pn_p32 ||
        !c->pn_l32 || !c->pn_n32 || !c->pn_sp || !c->pn_sn || !c->pn_y)
        return pb_fail(c, PB_ERR_NOMEM, "point near field: out of memory");
    // (the host vectors live in the context until the next build: no synchronisation needed)
    PB_CUDA(c, cudaMemcpyAsync(c->pn_items, c->h_pn_i4.data(), sizeof(int4) * c->h_pn_i4.size(),
                               cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->pn_tiles, c->h_pn_i[2].data(), sizeof(int) * c->h_pn_i[2].size(),
                               cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->pn_chunk_leaf, c->h_pn_i[0].data(), sizeof(int) * c->h_pn_i[0].size(),
                               cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->pn_chunk_first, c->h_pn_i[1].data(), sizeof(int) * c->h_pn_i[1].size(),
                               cudaMemcpyHostToDevice, c->st));
    PB_CUDA(c, cudaMemcpyAsync(c->pn_begin, c->begin_q, sizeof(int) * (lv.ncl + 1), cudaMemcpyDeviceToDevice, c->st));
    k_pts32<<<(unsigned)((np + 255) / 256), 256, 0, c->st>>>(np, c->pts_p, c->pts_n, c->pn_p32, c->pn_l32, c->pn_n32);
    PB_LAUNCH(c);
    return near_flags(c, (int)c->h_pn_i[0].size(), c->pn_chunk_leaf, c->pn_chunk_first, c->pn_begin, c->pts_p,
                      c->pn_nitems, c->pn_items, c->pn_tiles);
}

// ypt (2 np) = per point sum over the near points of other elements of K (W u), in FP64; the
// densities from element values xs or point values xq (one of them null)
int pb_near_points_apply(pb_ctx* c, const double* xs, const double* xq, double* ypt)
{
    const long long np = (long long)c->nt * c->q2;
    const double eps = c->prm.eps_out / c->prm.eps_in;
    k_pts_pack<<<(unsigned)((np + 255) / 256), 256, 0, c->st>>>(np, c->q2, c->nt, c->pn_p32, c->pn_n32, c->pts_p, xs,
                                                                 xq, c->pn_sp, c->pn_sn);
    PB_LAUNCH(c);
    PB_CUDA(c, cudaMemsetAsync(ypt, 0, sizeof(double) * 2 * np, c->st));
    const unsigned nb = (unsigned)((c->pn_nitems + NEAR_W - 1) / NEAR_W);
    if (c->q2 == 4)
        k_near_tile<4><<<nb, 32 * NEAR_W, 0, c->st>>>((int)np, c->pn_nitems, c->pn_items, c->pn_tiles, c->pn_chunk_leaf,
                                               c->pn_chunk_first, c->pn_begin, c->pn_sp, c->pn_sn, c->pn_l32, eps,
                                               c->prm.kappa, ypt);
    else
        k_near_tile<16><<<nb, 32 * NEAR_W, 0, c->st>>>((int)np, c->pn_nitems, c->pn_items, c->pn_tiles, c->pn_chunk_leaf,
                                                c->pn_chunk_first, c->pn_begin, c->pn_sp, c->pn_sn, c->pn_l32, eps,
                                                c->prm.kappa, ypt);
    PB_LAUNCH(c);
    return PB_OK;
}

// the piecewise-constant order-q near field with the mass terms from the point tiles
int pb_near_points_elem(pb_ctx* c, const double* xs, double* ys)
{
    int rc;
    if ((rc = pb_near_points_apply(c, xs, nullptr, c->pn_y))) return rc;
    const double eps = c->prm.eps_out / c->prm.eps_in;
    k_pts_finish_elem<<<(c->nt + 255) / 256, 256, 0, c->st>>>(c->nt, c->q2, c->e64p, c->pts_p, xs, c->pn_y, eps, ys);
    PB_LAUNCH(c);
    return PB_OK;
}
