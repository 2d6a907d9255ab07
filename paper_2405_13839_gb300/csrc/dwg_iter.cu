// dwg_iter.cu -- the per-iteration steps after the GWN evaluation
// (paper Alg. 1, Sec. 4.3, Sec. 5.1):
//   k_iso          iso-value w_bar = mean of w over the input points (Eq. 6,
//                  averaged over the inputs), FP64, fixed summation order;
//   k_mc_faces     level set of w - w_bar in every octree leaf, realised as
//                  the six-tetrahedron split of the leaf cube; one face per
//                  cut tetrahedron with its vector area (the cross-product
//                  gradient of Sec. 4.3) oriented toward increasing w;
//   k_knn_lists, k_knn_far  each face adds its vector to its k nearest input
//                  points (Eq. 7), from its leaf's candidate list or, in a
//                  leaf without one, by a warp's search of the bucket tree;
//                  sums are 64-bit fixed point, so the result does not depend
//                  on the order of the atomic additions (k_knn_scatter: k
//                  other than 10, or no lists at all);
//   k_normal_update  n_i <- -sum / |sum| (a point no face chose keeps its
//                  normal), the per-point change in degrees, next sources;
//   k_sel_*        convergence statistic of Sec. 5.1: mean of the
//                  ceil(n / 100) largest changes, by an exact multi-CTA radix
//                  select on the float bits, then the loop condition.
// and the once-per-cloud steps around it:
//   k_cell_radius, k_cell_lists  per-leaf candidate lists of the faces'
//                  k-nearest search (exact; built once per discretisation);
//   k_init_pca, k_init_gauss     PCA and Gauss-map initial normals (Sec. 5.1);
//   k_voronoi_area              local-Voronoi area weights (Sec. 5.1);
//   k_clamp_delta               clamp radii of the modified kernel (Sec. 5.2);
//   k_mc_tris                   the level set as triangles (the output);
//   k_features                  patch features of the learned warm start.
#include <algorithm>

#include <string.h>

#include "dwg_internal.cuh"

namespace dwg {

// ---------------------------------------------------------------------------
// iso-value
// ---------------------------------------------------------------------------
__device__ __forceinline__ void iso_body(const double *__restrict__ wsum_blocks, int nb,
                                         int64_t n, IterState *st)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    __shared__ double sh[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += wsum_blocks[b];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        st->iso = sh[0] / (double)n;
        st->nfaces = 0;
        st->ndefer = 0;
        st->nfar = 0;
    }
}

__global__ void k_iso(const double *__restrict__ wsum_blocks, int nb, int64_t n, IterState *st)
{
    iso_body(wsum_blocks, nb, n, st);
}

// ---------------------------------------------------------------------------
// level-set faces
// ---------------------------------------------------------------------------
__constant__ int c_tets[6][4] = {{0, 1, 3, 7}, {0, 3, 2, 7}, {0, 2, 6, 7},
                                 {0, 6, 4, 7}, {0, 4, 5, 7}, {0, 5, 1, 7}};

struct F3 {
    float x, y, z;
};
__device__ __forceinline__ F3 f3(float4 v) { return {v.x, v.y, v.z}; }
__device__ __forceinline__ F3 operator-(F3 a, F3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ F3 cross(F3 a, F3 b)
{
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ F3 lerp0(F3 xa, float fa, F3 xb, float fb)
{
    float t = fa / (fa - fb);
    return {xa.x + t * (xb.x - xa.x), xa.y + t * (xb.y - xa.y), xa.z + t * (xb.z - xa.z)};
}

// Polygon of a tetrahedron that the level set cuts; m has bit i where vertex i
// is above.  The vertices are first put in the order lone vertex, others (one
// on its own side) or two above, two below: by selects over all four, so that
// nothing is indexed and everything stays in registers.
__device__ __forceinline__ void tet_face(const F3 (&x)[4], const float (&f)[4], int m, F3 &area,
                                         F3 &cen)
{
    // per mask, 2 bits a place: which vertex comes first, second, ...
    // (mask 0 and 15 do not occur)
    const int na = __popc(m);
    const int mm = na == 3 ? 15 - m : m;  // the lone vertex's bit
    // orders of the masks 1 2 3 4 5 6 8 9 10 12, 8 bits each, at 8 * mask
    const unsigned long long t0 = 0xe4ull << 8 | 0xe1ull << 16 | 0xe4ull << 24 | 0xd2ull << 32 |
                                  0xd8ull << 40 | 0xc9ull << 48;
    const unsigned long long t1 = 0x93ull | 0x9cull << 8 | 0x8dull << 16 | 0x4eull << 32;
    const unsigned perm = (unsigned)((mm < 8 ? t0 : t1) >> (8 * (mm & 7)));
    F3 v[4];
    float g[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = (perm >> (2 * i)) & 3;
        v[i] = j == 0 ? x[0] : j == 1 ? x[1] : j == 2 ? x[2] : x[3];
        g[i] = j == 0 ? f[0] : j == 1 ? f[1] : j == 2 ? f[2] : f[3];
    }
    F3 P[4];
    F3 ca = {0, 0, 0}, cb = {0, 0, 0};
    auto add = [](F3 &a, F3 p) { a.x += p.x; a.y += p.y; a.z += p.z; };
    const bool quad = na == 2;
    P[0] = lerp0(v[0], g[0], quad ? v[2] : v[1], quad ? g[2] : g[1]);
    P[1] = lerp0(v[0], g[0], quad ? v[3] : v[2], quad ? g[3] : g[2]);
    P[2] = lerp0(quad ? v[1] : v[0], quad ? g[1] : g[0], v[3], g[3]);
    P[3] = lerp0(v[1], g[1], v[2], g[2]);  // of a quadrilateral
    F3 s = {0, 0, 0};
    if (quad) {
        area = cross(P[2] - P[0], P[3] - P[1]);
        add(ca, v[0]);
        add(ca, v[1]);
        add(cb, v[2]);
        add(cb, v[3]);
    } else {
        area = cross(P[1] - P[0], P[2] - P[0]);
        add(ca, v[0]);
        add(cb, v[1]);
        add(cb, v[2]);
        add(cb, v[3]);
        if (na == 3) {
            const F3 t = ca;
            ca = cb;
            cb = t;
        }
    }
    area.x *= 0.5f; area.y *= 0.5f; area.z *= 0.5f;
    const float ia = 1.f / na, ib = 1.f / (4 - na);
    F3 dir = {ca.x * ia - cb.x * ib, ca.y * ia - cb.y * ib, ca.z * ia - cb.z * ib};
    if (area.x * dir.x + area.y * dir.y + area.z * dir.z < 0.f) {
        area.x = -area.x; area.y = -area.y; area.z = -area.z;
    }
    add(s, P[0]);
    add(s, P[1]);
    add(s, P[2]);
    if (quad) add(s, P[3]);
    const float inv = quad ? 0.25f : 1.f / 3;
    cen = {s.x * inv, s.y * inv, s.z * inv};
}

// Triangles of one tetrahedron's piece of the level set (0, 1 or 2), on the
// same edge points as tet_face, wound so that (v1 - v0) x (v2 - v0) points
// toward decreasing w (outward for outward normals).
__device__ __forceinline__ int tet_tris(const F3 x[4], const float f[4], const bool ab[4],
                                        F3 T[2][3])
{
    int na = (int)ab[0] + (int)ab[1] + (int)ab[2] + (int)ab[3];
    if (na == 0 || na == 4) return 0;
    F3 P[4];
    int nt;
    if (na == 1 || na == 3) {
        bool want = (na == 1);
        int lone = 0;
        for (int i = 0; i < 4; ++i)
            if (ab[i] == want) lone = i;
        int np = 0;
        for (int i = 0; i < 4; ++i)
            if (i != lone) P[np++] = lerp0(x[lone], f[lone], x[i], f[i]);
        T[0][0] = P[0]; T[0][1] = P[1]; T[0][2] = P[2];
        nt = 1;
    } else {
        int a0 = -1, a1 = -1, b0 = -1, b1 = -1;
        for (int i = 0; i < 4; ++i) {
            if (ab[i]) { if (a0 < 0) a0 = i; else a1 = i; }
            else { if (b0 < 0) b0 = i; else b1 = i; }
        }
        P[0] = lerp0(x[a0], f[a0], x[b0], f[b0]);  // a cycle of the quad
        P[1] = lerp0(x[a0], f[a0], x[b1], f[b1]);
        P[2] = lerp0(x[a1], f[a1], x[b1], f[b1]);
        P[3] = lerp0(x[a1], f[a1], x[b0], f[b0]);
        T[0][0] = P[0]; T[0][1] = P[1]; T[0][2] = P[2];
        T[1][0] = P[0]; T[1][1] = P[2]; T[1][2] = P[3];
        nt = 2;
    }
    F3 ca = {0, 0, 0}, cb = {0, 0, 0};
    for (int i = 0; i < 4; ++i) {
        if (ab[i]) { ca.x += x[i].x; ca.y += x[i].y; ca.z += x[i].z; }
        else { cb.x += x[i].x; cb.y += x[i].y; cb.z += x[i].z; }
    }
    float ia = 1.f / na, ib = 1.f / (4 - na);
    F3 down = {cb.x * ib - ca.x * ia, cb.y * ib - ca.y * ia, cb.z * ib - ca.z * ia};
    F3 nrm = nt == 1 ? cross(P[1] - P[0], P[2] - P[0]) : cross(P[2] - P[0], P[3] - P[1]);
    if (nrm.x * down.x + nrm.y * down.y + nrm.z * down.z < 0.f)
        for (int t = 0; t < nt; ++t) {
            F3 v = T[t][1];
            T[t][1] = T[t][2];
            T[t][2] = v;
        }
    return nt;
}

// The level set as triangles: the same corner values and decisions as
// k_mc_faces.  Without FILL only the count; with FILL each leaf writes its
// triangles (9 floats) at an index from the counter, those below cap.
template <bool FILL>
__global__ void __launch_bounds__(256)
    k_mc_tris(const int *__restrict__ leaf_corners, int64_t nl, const float4 *__restrict__ cpos,
              const float *__restrict__ wc, const IterState *st, float *__restrict__ out,
              int64_t cap, unsigned long long *counter)
{
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nl) return;
    const double iso = st->iso;
    F3 x[8];
    float f[8];
    bool ab[8];
    for (int v = 0; v < 8; ++v) {
        int ci = leaf_corners[l * 8 + v];
        x[v] = f3(cpos[ci]);
        double df = (double)wc[ci] - iso;
        f[v] = (float)df;
        ab[v] = df > 0.0;
    }
    F3 T[12][3];
    int nt = 0;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        F3 xt[4];
        float ft[4];
        bool at[4];
        for (int i = 0; i < 4; ++i) {
            int v = c_tets[t][i];
            xt[i] = x[v];
            ft[i] = f[v];
            at[i] = ab[v];
        }
        F3 tt[2][3];
        const int k = tet_tris(xt, ft, at, tt);
        for (int j = 0; j < k; ++j) {
            T[nt][0] = tt[j][0];
            T[nt][1] = tt[j][1];
            T[nt][2] = tt[j][2];
            ++nt;
        }
    }
    if (nt == 0) return;
    const unsigned long long base = atomicAdd(counter, (unsigned long long)nt);
    if (!FILL) return;
    for (int j = 0; j < nt; ++j) {
        const unsigned long long o = base + j;
        if (o >= (unsigned long long)cap) break;
        float *r = out + 9 * o;
        for (int v = 0; v < 3; ++v) {
            r[3 * v + 0] = T[j][v].x;
            r[3 * v + 1] = T[j][v].y;
            r[3 * v + 2] = T[j][v].z;
        }
    }
}

cudaError_t launch_mc_tris(Ctx *c, float *out, int64_t cap, unsigned long long *counter)
{
    const unsigned g = (unsigned)ceil_div(c->nleaves, 256);
    if (out)
        k_mc_tris<true><<<g, 256, 0, c->stream>>>(c->d_leaf_corners, c->nleaves, c->d_corner_pos,
                                                  c->d_wc, c->d_state, out, cap, counter);
    else
        k_mc_tris<false><<<g, 256, 0, c->stream>>>(c->d_leaf_corners, c->nleaves,
                                                   c->d_corner_pos, c->d_wc, c->d_state, nullptr,
                                                   0, counter);
    return cudaGetLastError();
}

// Faces of the level set.  Each face record also carries its leaf's index
// (in the area's w) and, in the centroid's w, the position in the
// Morton-sorted points of the face's leaf cell (found once per cut leaf):
// the k-nearest search of its faces starts there.  The signs at the eight
// corners say how many faces a leaf has, so a leaf that is not cut reads
// nothing else and the faces are written as they are computed.  Bound by the
// latency of the gathers on a small octree, by their L2 traffic on a large
// one: 22.5 -> 16.4 us on a 2,000-point sphere and 2.92 -> 2.37 ms on a 4M
// union (random normals) against vertices indexed in local memory and all
// positions read.
__device__ __forceinline__ void mc_faces_body(const int *__restrict__ leaf_corners,
                                              const int4 *__restrict__ leaves, int64_t nl,
                                              const float4 *__restrict__ cpos,
                                              const float *__restrict__ wc,
                                              const uint64_t *__restrict__ codes, int64_t n,
                                              IterState *st, float4 *__restrict__ faces,
                                              int64_t max_faces, int *err, int64_t bid)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    int64_t l = bid * blockDim.x + threadIdx.x;
    const double iso = st->iso;
    // corner masks of the six tetrahedra (corners 0 and 7 and two more)
    constexpr int tets[6][4] = {{0, 1, 3, 7}, {0, 3, 2, 7}, {0, 2, 6, 7},
                                {0, 6, 4, 7}, {0, 4, 5, 7}, {0, 5, 1, 7}};
    int cnt = 0;
    int ci[8];
    float f[8];
    bool ab[8];
    if (l < nl) {
        const int4 c0 = reinterpret_cast<const int4 *>(leaf_corners)[2 * l];
        const int4 c1 = reinterpret_cast<const int4 *>(leaf_corners)[2 * l + 1];
        ci[0] = c0.x; ci[1] = c0.y; ci[2] = c0.z; ci[3] = c0.w;
        ci[4] = c1.x; ci[5] = c1.y; ci[6] = c1.z; ci[7] = c1.w;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            double df = (double)wc[ci[v]] - iso;
            f[v] = (float)df;
            ab[v] = df > 0.0;
        }
#pragma unroll
        for (int t = 0; t < 6; ++t) {
            const int na = (int)ab[0] + (int)ab[tets[t][1]] + (int)ab[tets[t][2]] + (int)ab[7];
            cnt += (na & 3) != 0;
        }
    }
    int seed = 0;
    if (cnt > 0) {
        const int4 L = leaves[l];
        const uint64_t code = ((uint64_t)(uint32_t)L.y | ((uint64_t)(uint32_t)L.z << 32))
                              << (3 * (kMortonBits - L.x));
        int64_t lo = 0, hi = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (__ldg(&codes[mid]) < code) lo = mid + 1; else hi = mid;
        }
        seed = (int)lo;
    }
    // warp-aggregated append
    const int lane = threadIdx.x & 31;
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    int total = __shfl_sync(0xffffffffu, incl, 31);
    int base = 0;
    if (lane == 31 && total > 0) base = atomicAdd(&st->nfaces, total);
    base = __shfl_sync(0xffffffffu, base, 31);
    int64_t o = (int64_t)base + incl - cnt;
    if (cnt == 0) return;
    F3 x[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) x[v] = f3(cpos[ci[v]]);
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        const int m = (int)ab[0] | (int)ab[tets[t][1]] << 1 | (int)ab[tets[t][2]] << 2 |
                      (int)ab[7] << 3;
        if (m == 0 || m == 15) continue;
        if (o >= max_faces) {
            atomicOr(err, kErrOverflow);
            break;
        }
        const F3 xt[4] = {x[0], x[tets[t][1]], x[tets[t][2]], x[7]};
        const float ft[4] = {f[0], f[tets[t][1]], f[tets[t][2]], f[7]};
        F3 area, cen;
        tet_face(xt, ft, m, area, cen);
        faces[2 * o] = make_float4(area.x, area.y, area.z, __int_as_float((int)l));
        faces[2 * o + 1] = make_float4(cen.x, cen.y, cen.z, __int_as_float(seed));
        ++o;
    }
}

__global__ void __launch_bounds__(256)
    k_mc_faces(const int *__restrict__ leaf_corners, const int4 *__restrict__ leaves, int64_t nl,
               const float4 *__restrict__ cpos, const float *__restrict__ wc,
               const uint64_t *__restrict__ codes, int64_t n, IterState *st,
               float4 *__restrict__ faces, int64_t max_faces, int *err)
{
    mc_faces_body(leaf_corners, leaves, nl, cpos, wc, codes, n, st, faces, max_faces, err,
                  blockIdx.x);
}

// ---------------------------------------------------------------------------
// exact k nearest points over the bucket tree
// ---------------------------------------------------------------------------
__device__ __forceinline__ float box_d2(float4 lo, float4 hi, F3 q)
{
    float dx = fmaxf(fmaxf(lo.x - q.x, q.x - hi.x), 0.f);
    float dy = fmaxf(fmaxf(lo.y - q.y, q.y - hi.y), 0.f);
    float dz = fmaxf(fmaxf(lo.z - q.z, q.z - hi.z), 0.f);
    return fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
}
__device__ __forceinline__ float pt_d2(float4 p, F3 q)
{
    float dx = __fsub_rn(p.x, q.x), dy = __fsub_rn(p.y, q.y), dz = __fsub_rn(p.z, q.z);
    return fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
}

// Candidate order: squared float32 distance, ties to the smaller input index,
// as one 64-bit key (the bits of a non-negative float order like the float).
__device__ __forceinline__ uint64_t knn_key(float d, int64_t o)
{
    return ((uint64_t)__float_as_uint(d) << 32) | (uint64_t)(uint32_t)o;
}

template <int KMAX, bool FIXED>
__device__ __forceinline__ void knn_insert(uint64_t key, int j, int k, uint64_t *best, int *bj)
{
#pragma unroll
    for (int t = KMAX - 1; t >= 0; --t) {
        if (!FIXED && t >= k) continue;
        bool prev = t > 0 && key < best[t > 0 ? t - 1 : 0];
        bool cur = key < best[t];
        if (prev) {
            best[t] = best[t - 1];
            bj[t] = bj[t - 1];
        } else if (cur) {
            best[t] = key;
            bj[t] = j;
        }
    }
}

// Exact k nearest points of q.  KMAX is the array size; with FIXED the
// runtime k equals KMAX and every index is a compile-time constant (the
// arrays stay in registers).  The list is seeded with the points next to q's
// Morton code in the sorted order, which bounds the search ball before the
// depth-first descent (nearer child first) prunes the bucket tree.
// With budget >= 0 the search gives up after that many node visits and
// point distances, returns false and leaves in *bound the k-th smallest
// distance (squared) found so far: an upper bound of q's k-th nearest.
template <int KMAX, bool FIXED>
__device__ __forceinline__ bool knn_search(const KnnTree &T, F3 q, int k, int *bj, int *err,
                                           int64_t seed = -1, int budget = -1,
                                           float *bound = nullptr)
{
    uint64_t best[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
        best[t] = ~0ull;
        bj[t] = -1;
    }
    const int kk = FIXED ? KMAX : k;
    // seed: the sorted neighbours of q's position on the Morton curve (or a
    // given position near q)
    int64_t lo = seed;
    if (lo < 0) {
        uint64_t code = morton3((uint64_t)quant21(q.x, T.cube_lo[0], T.inv_h21),
                                (uint64_t)quant21(q.y, T.cube_lo[1], T.inv_h21),
                                (uint64_t)quant21(q.z, T.cube_lo[2], T.inv_h21));
        int64_t hi = T.n;
        lo = 0;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (__ldg(&T.codes[mid]) < code) lo = mid + 1; else hi = mid;
        }
    }
    const int64_t s0 = max((int64_t)0, lo - kk), s1 = min(T.n, lo + kk);
    for (int64_t j = s0; j < s1; ++j) {
        float d = pt_d2(__ldg(&T.p4[j]), q);
        uint64_t key = knn_key(d, __ldg(&T.perm[j]));
        if (key < best[kk - 1]) knn_insert<KMAX, FIXED>(key, (int)j, k, best, bj);
    }
    const int64_t nleaf = (int64_t)1 << T.levels;
    int stack[64];
    int sp = 0;
    int work = 0;
    stack[sp++] = 1;
    while (sp > 0) {
        int node = stack[--sp];
        const float worst = best[kk - 1] == ~0ull ? INFINITY : __uint_as_float((uint32_t)(best[kk - 1] >> 32));
        if (budget >= 0 && work > budget) {
            *bound = worst;
            return false;
        }
        ++work;
        if (box_d2(__ldg(&T.lo[node]), __ldg(&T.hi[node]), q) > worst) continue;
        if (node >= nleaf) {
            int64_t j0 = (int64_t)(node - nleaf) * kBucket;
            int64_t j1 = min(j0 + kBucket, T.n);
            work += (int)(j1 - j0);
            for (int64_t j = j0; j < j1; ++j) {
                if (j >= s0 && j < s1) continue;  // already seeded
                float d = pt_d2(__ldg(&T.p4[j]), q);
                if (d > worst) continue;
                uint64_t key = knn_key(d, __ldg(&T.perm[j]));
                if (key < best[kk - 1]) knn_insert<KMAX, FIXED>(key, (int)j, k, best, bj);
            }
        } else {
            int a = 2 * node, b = 2 * node + 1;
            float da = box_d2(__ldg(&T.lo[a]), __ldg(&T.hi[a]), q);
            float db = box_d2(__ldg(&T.lo[b]), __ldg(&T.hi[b]), q);
            if (sp + 2 > 64) {
                atomicOr(err, kErrStack);
                break;
            }
            // push the farther child first so that the nearer one is visited first
            if (da <= db) {
                if (db <= worst) stack[sp++] = b;
                if (da <= worst) stack[sp++] = a;
            } else {
                if (da <= worst) stack[sp++] = a;
                if (db <= worst) stack[sp++] = b;
            }
        }
    }
    return true;
}

// The k nearest of q among a candidate list that is known to contain them:
// the same keys and insertion as knn_search, so the same result.
template <int KMAX, bool FIXED>
__device__ __forceinline__ void knn_scan(const KnnTree &T, F3 q, int k, const int *__restrict__ cand,
                                         int64_t c0, int64_t c1, int *bj)
{
    uint64_t best[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
        best[t] = ~0ull;
        bj[t] = -1;
    }
    const int kk = FIXED ? KMAX : k;
    float worst = INFINITY;
    for (int64_t t = c0; t < c1; ++t) {
        const int j = __ldg(&cand[t]);
        const float d = pt_d2(__ldg(&T.p4[j]), q);
        if (d > worst) continue;  // the tie-break index is only needed from here
        const uint64_t key = knn_key(d, __ldg(&T.perm[j]));
        if (key < best[kk - 1]) {
            knn_insert<KMAX, FIXED>(key, j, k, best, bj);
            if (best[kk - 1] != ~0ull) worst = __uint_as_float((uint32_t)(best[kk - 1] >> 32));
        }
    }
}

static KnnTree knn_tree(const Ctx *c);

// ---------------------------------------------------------------------------
// the same search by a whole warp
// ---------------------------------------------------------------------------
// The list is one (key, index) pair per lane, ascending over the lanes.
__device__ __forceinline__ void warp_cmp_swap(uint64_t &key, int &j, int lane, int mask, bool up)
{
    const uint64_t ok = __shfl_xor_sync(0xffffffffu, key, mask);
    const int oj = __shfl_xor_sync(0xffffffffu, j, mask);
    // `up`: the lower lane of the pair keeps the smaller key
    if (((lane & mask) == 0) == up ? ok < key : ok > key) {
        key = ok;
        j = oj;
    }
}

// bitonic sort of the warp's 32 pairs, ascending over the lanes
__device__ __forceinline__ void warp_sort(uint64_t &key, int &j, int lane)
{
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int m = size >> 1; m > 0; m >>= 1)
            warp_cmp_swap(key, j, lane, m, (lane & size) == 0 || size == 32);
}

// The batch (nk, nj), one pair per lane (~0: none), merged into the sorted
// list: one pair at a time while few are below the k-th key, else by sorting
// the batch and a bitonic merge of the two lists' 32 smallest (the line between
// them at 6, 12, 20 or all 32: within 1 % of each other).
__device__ __forceinline__ void warp_merge(uint64_t &key, int &j, uint64_t &kth, uint64_t nk, int nj,
                                           int k, int lane)
{
    unsigned m = __ballot_sync(0xffffffffu, nk < kth);
    if (__popc(m) > 12) {
        warp_sort(nk, nj, lane);
        const uint64_t rk = __shfl_sync(0xffffffffu, nk, 31 - lane);
        const int rj = __shfl_sync(0xffffffffu, nj, 31 - lane);
        if (rk < key) {
            key = rk;
            j = rj;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) warp_cmp_swap(key, j, lane, d, true);
        kth = __shfl_sync(0xffffffffu, key, k - 1);
        return;
    }
    while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const uint64_t ck = __shfl_sync(0xffffffffu, nk, src);
        const int cj = __shfl_sync(0xffffffffu, nj, src);
        const uint64_t pk = __shfl_up_sync(0xffffffffu, key, 1);
        const int pj = __shfl_up_sync(0xffffffffu, j, 1);
        if (key > ck) {
            const bool shift = lane > 0 && pk > ck;
            key = shift ? pk : ck;
            j = shift ? pj : cj;
        }
        kth = __shfl_sync(0xffffffffu, key, k - 1);
        m &= __ballot_sync(0xffffffffu, nk < kth);
    }
}

constexpr int kWarpStack = 160;  // 31 siblings stay on the stack per five levels of the tree

// Exact k nearest points of q (k <= 32) by one warp, the keys of knn_search:
// lane t ends with the t-th nearest point in j (-1: fewer points).  A step
// tests the up to 32 descendants five levels below a node at once (they are
// consecutive in the heap: one coalesced load), the nearest of those within
// the k-th distance is taken next; two buckets are scanned at a time, a lane
// per point.  The list starts from the 32 points around `seed`, a position
// in the sorted points.  Budget and *bound as in knn_search.
__device__ __forceinline__ bool warp_knn(const KnnTree &T, F3 q, int k, int64_t seed, int lane,
                                         int2 *stack, int &j, int *err, int budget, float *bound)
{
    const int64_t s0 = max((int64_t)0, min(seed - 16, T.n - 32)), s1 = min(T.n, s0 + 32);
    uint64_t key = ~0ull;
    j = -1;
    if (s0 + lane < s1) {
        j = (int)(s0 + lane);
        key = knn_key(pt_d2(__ldg(&T.p4[j]), q), __ldg(&T.perm[j]));
    }
    warp_sort(key, j, lane);
    uint64_t kth = __shfl_sync(0xffffffffu, key, k - 1);
    auto worst_of = [](uint64_t kk) {
        return kk == ~0ull ? INFINITY : __uint_as_float((uint32_t)(kk >> 32));
    };
    float worst = worst_of(kth);
    const unsigned lt = (1u << lane) - 1u;
    const int nleaf = 1 << T.levels;
    int sp = 1, work = 0;
    __syncwarp();
    if (lane == 0) stack[0] = make_int2(1, 0);
    __syncwarp();
    while (sp > 0) {
        const int2 e = stack[--sp];
        if (__int_as_float(e.y) > worst) continue;
        if (budget >= 0 && work > budget) {
            *bound = worst;
            return false;
        }
        const int lv = 31 - __clz(e.x), step = min(5, T.levels - lv);
        const int child = (e.x << step) + lane;
        float cd = INFINITY;
        const bool in = lane < (1 << step);
        if (in) cd = box_d2(__ldg(&T.lo[child]), __ldg(&T.hi[child]), q);
        work += 1 << step;
        unsigned keep = __ballot_sync(0xffffffffu, in && cd <= worst);
        if (keep == 0) continue;
        // the nearest of the kept nodes
        const unsigned cb = (keep >> lane) & 1u ? __float_as_uint(cd) : 0xffffffffu;
        const unsigned mn = __reduce_min_sync(0xffffffffu, cb);
        const int first = __ffs(__ballot_sync(0xffffffffu, cb == mn) & keep) - 1;
        if (lv + step < T.levels) {  // inner nodes: the nearest on top of the stack
            const int cnt = __popc(keep);
            if (sp + cnt > kWarpStack) {
                if (lane == 0) atomicOr(err, kErrStack);
                break;
            }
            if ((keep >> lane) & 1u) {
                const int pos = lane == first ? cnt - 1
                                              : __popc(keep & lt) - (lane > first ? 1 : 0);
                stack[sp + pos] = make_int2(child, __float_as_int(cd));
            }
            sp += cnt;
            __syncwarp();
            continue;
        }
        // buckets, two at a time, the nearest first
        const int child0 = child - lane;
        int a = first;
        keep &= ~(1u << first);
        while (a >= 0) {
            const int b = keep ? __ffs(keep) - 1 : -1;
            if (b >= 0) keep &= keep - 1;
            const int mine = lane < 16 ? a : b;
            const int64_t p = (int64_t)(child0 + mine - nleaf) * kBucket + (lane & 15);
            uint64_t nk = ~0ull;
            if (mine >= 0 && p < T.n && !(p >= s0 && p < s1)) {
                const float d = pt_d2(__ldg(&T.p4[p]), q);
                if (d <= worst) nk = knn_key(d, __ldg(&T.perm[p]));
            }
            work += 32;
            warp_merge(key, j, kth, nk, (int)p, k, lane);
            worst = worst_of(kth);
            keep &= __ballot_sync(0xffffffffu, cd <= worst);
            a = keep ? __ffs(keep) - 1 : -1;
            if (a >= 0) keep &= keep - 1;
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// the same search for a warp of neighbouring queries, one per lane
// ---------------------------------------------------------------------------
// The lanes' queries lie together (consecutive sorted points, consecutive
// octree leaves), so their searches visit nearly the same nodes: the warp
// walks the tree once, each node's box tested by every lane against its own
// query and radius, four descendants two levels down a step (consecutive in
// the heap); a node no lane needs is dropped.  A bucket that some lane needs
// is read once, every point a broadcast, and each lane keeps its K smallest
// distances with floating-point minima and maxima only.  A second pass over
// the buckets read collects the points within the K-th distance, which are
// then ordered by the (distance, input index) keys.  (A test of the box
// around all the queries prunes 32 nodes at once, but one outlier among
// them, or a jump of the Morton order, makes it keep most of the tree.)
constexpr int kShWarps = 4;       // warps per CTA of the kernels that use it
constexpr int kShStack = 96;      // at most 3 siblings per two levels stay behind
// A warp stops after this many buckets: the lanes that still need a node (an
// outlier, a cell far from the points) are searched by a warp each instead,
// so that one such query does not hold its 31 neighbours.  With 32 buckets the
// features of a 1M blob take 2.28 ms, with 64 1.77, with 128 1.91 (1 % outliers;
// 200,000 points 541, 538 and 700 us).
constexpr int kShBuckets = 64;

struct ShSmem {
    int stack[kShStack];
    int visited[kShBuckets];
};

// Walks the tree for the warp's queries.  worst(): this lane's radius
// (squared; negative: nothing needed); on_bucket(b) is called by every lane
// for each bucket within some lane's radius, the nearest subtree first.  When
// on_bucket gives up (false), the lanes that need it or a node still on the
// stack get true.
template <class WorstFn, class BucketFn>
__device__ __forceinline__ bool sh_walk(const KnnTree &T, F3 q, int lane, int *stack,
                                        WorstFn &&worst, BucketFn &&on_bucket)
{
    const int nleaf = 1 << T.levels;
    // the least distance at which a lane needs the node (float bits), ~0: none
    auto need = [&](int node) {
        const float d = box_d2(__ldg(&T.lo[node]), __ldg(&T.hi[node]), q);
        return __reduce_min_sync(0xffffffffu, d <= worst() ? __float_as_uint(d) : 0xffffffffu);
    };
    int sp = 1;
    __syncwarp();
    if (lane == 0) stack[0] = 1;
    __syncwarp();
    while (sp > 0) {
        const int node = stack[--sp];
        if (need(node) == 0xffffffffu) continue;
        if (node >= nleaf) {
            if (on_bucket(node - nleaf)) continue;
            bool more = false;
            for (++sp; sp > 0 && !more;) {
                const int nd = stack[--sp];
                more = box_d2(__ldg(&T.lo[nd]), __ldg(&T.hi[nd]), q) <= worst();
            }
            __syncwarp();
            return more;
        }
        const int step = node >= nleaf / 2 ? 1 : 2;
        const int c0 = node << step, nc = 1 << step;
        unsigned dd[4];
        int cc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cc[i] = c0 + i;
            dd[i] = i < nc ? need(c0 + i) : 0xffffffffu;
        }
        // farthest first onto the stack
        auto order = [&](int i, int j) {
            if (dd[i] < dd[j]) {
                const unsigned t = dd[i]; dd[i] = dd[j]; dd[j] = t;
                const int u = cc[i]; cc[i] = cc[j]; cc[j] = u;
            }
        };
        order(0, 1); order(2, 3); order(0, 2); order(1, 3); order(1, 2);
        __syncwarp();  // the pop above is read by every lane
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (dd[i] != 0xffffffffu) {
                if (lane == 0) stack[sp] = cc[i];
                ++sp;
            }
        __syncwarp();
    }
    return false;
}

// The K smallest distances (squared) of each lane's query in b, ascending,
// INFINITY where the cloud has fewer points.  `seed`: a sorted position near
// the queries (the same in every lane), whose four buckets are read first.
// S.visited holds the *nvis buckets read.  True for a lane whose search did
// not end within kShBuckets buckets.
template <int K>
__device__ __forceinline__ bool sh_smallest(const KnnTree &T, F3 q, int64_t seed, int lane,
                                            ShSmem &S, int *nvis, float (&b)[K])
{
#pragma unroll
    for (int t = 0; t < K; ++t) b[t] = INFINITY;
    int nv = 0;
    auto read = [&](int64_t bucket) {
        if (lane == 0) S.visited[nv] = (int)bucket;
        ++nv;
        const int64_t j0 = bucket * kBucket;
        const int cnt = (int)min((int64_t)kBucket, T.n - j0);
#pragma unroll 4
        for (int u = 0; u < cnt; ++u) {
            const float d = pt_d2(__ldg(&T.p4[j0 + u]), q);
            if (d < b[K - 1]) {
#pragma unroll
                for (int t = K - 1; t > 0; --t) b[t] = fmaxf(b[t - 1], fminf(b[t], d));
                b[0] = fminf(b[0], d);
            }
        }
    };
    const int64_t nb = (T.n + kBucket - 1) / kBucket;
    const int64_t s0 = max((int64_t)0, min(seed / kBucket - 1, nb - 4)), s1 = min(nb, s0 + 4);
    for (int64_t s = s0; s < s1; ++s) read(s);
    const bool more = sh_walk(
        T, q, lane, S.stack, [&]() { return b[K - 1]; },
        [&](int bucket) {
            if (bucket >= s0 && bucket < s1) return true;
            if ((int64_t)bucket >= nb) return true;  // an empty leaf of the complete tree
            if (nv == kShBuckets) return false;
            read(bucket);
            return true;
        });
    *nvis = nv;
    __syncwarp();
    return more;
}

// ---------------------------------------------------------------------------
// the K nearest points of every point, itself among them
// ---------------------------------------------------------------------------
// idx[t * stride + r]: the t-th nearest (ascending keys, sorted position, -1:
// fewer points) of sorted point i0 + r, r < cnt, as knn_search<K, true>
// gives it.  Points whose search does not end within the warp's buckets, or
// whose K-th distance ties with others beyond the K, go to the queue.
template <int K>
__global__ void __launch_bounds__(32 * kShWarps)
    k_knn_points(KnnTree T, int64_t i0, int cnt, int64_t stride, int *__restrict__ idx,
                 int *__restrict__ queue, int *nqueue)
{
    __shared__ ShSmem S_all[kShWarps];
    __shared__ int cols_all[kShWarps][K][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r - lane >= cnt) return;  // the whole warp
    ShSmem &S = S_all[wid];
    int (*cols)[32] = cols_all[wid];
    const bool valid = r < cnt;
    const int64_t i = i0 + (valid ? r : cnt - 1);
    const float4 p = T.p4[i];
    const F3 q{p.x, p.y, p.z};
    int nv = 0, found = 0;
    bool far;
    {
        float b[K];
        far = sh_smallest<K>(T, q, i0 + r - lane + 16, lane, S, &nv, b);
        const float dk = far ? -1.f : b[K - 1];
        for (int v = 0; v < nv; ++v) {
            const int bucket = S.visited[v];
            const int node = (1 << T.levels) + bucket;
            const float d = box_d2(__ldg(&T.lo[node]), __ldg(&T.hi[node]), q);
            if (!__any_sync(0xffffffffu, d <= dk)) continue;
            const int64_t j0 = (int64_t)bucket * kBucket;
            const int c = (int)min((int64_t)kBucket, T.n - j0);
#pragma unroll 4
            for (int u = 0; u < c; ++u)
                if (pt_d2(__ldg(&T.p4[j0 + u]), q) <= dk) {
                    if (found < K) cols[found][lane] = (int)j0 + u;
                    ++found;
                }
        }
    }
    far = valid && (far || found > K);
    const unsigned fm = __ballot_sync(0xffffffffu, far);
    if (fm) {
        int base = 0;
        if (lane == 0) base = atomicAdd(nqueue, __popc(fm));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (far) queue[base + __popc(fm & ((1u << lane) - 1u))] = r;
    }
    if (!valid || far) return;
    uint64_t key[K];
    int bj[K];
#pragma unroll
    for (int t = 0; t < K; ++t) {
        bj[t] = t < found ? cols[t][lane] : -1;
        key[t] = bj[t] >= 0 ? knn_key(pt_d2(__ldg(&T.p4[bj[t]]), q), __ldg(&T.perm[bj[t]])) : ~0ull;
    }
#pragma unroll
    for (int u = 0; u < K; ++u)
#pragma unroll
        for (int t = u & 1; t + 1 < K; t += 2)
            if (key[t + 1] < key[t]) {
                const uint64_t k = key[t];
                key[t] = key[t + 1];
                key[t + 1] = k;
                const int j = bj[t];
                bj[t] = bj[t + 1];
                bj[t + 1] = j;
            }
#pragma unroll
    for (int t = 0; t < K; ++t) idx[t * stride + r] = bj[t];
}

// the queued points, a warp each
__global__ void __launch_bounds__(32 * kShWarps)
    k_knn_points_far(KnnTree T, int64_t i0, int64_t stride, int k, int *__restrict__ idx,
                     const int *__restrict__ queue, const int *__restrict__ nqueue, int *err)
{
    __shared__ int2 s_stack[kShWarps][kWarpStack];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nq = *nqueue;
    for (int u = blockIdx.x * kShWarps + wid; u < nq; u += gridDim.x * kShWarps) {
        const int r = queue[u];
        const float4 p = T.p4[i0 + r];
        int j;
        float bound;
        warp_knn(T, F3{p.x, p.y, p.z}, k, i0 + r, lane, s_stack[wid], j, err, -1, &bound);
        if (lane < k) idx[(int64_t)lane * stride + r] = j;
    }
}

constexpr int kShFarBlocks = kSMs * 8;

// A table of the K nearest points, filled for one range of points at a time
// (at most kKnnRange, so that the table stays small beside a large cloud;
// fewer where memory is short): `use(i0, cnt, stride, table)` launches the
// kernel that reads it.  A cloud of at most kKnnDirect points gets none: there
// the launches that fill a table are the time, and the kernel that would read
// it searches by itself (features of 10 points: 67 us by a table, 47 by itself;
// of 100 points 74 by a table, 99).
constexpr int64_t kKnnRange = (int64_t)3 << 20;
constexpr int64_t kKnnRangeMin = 4096;
constexpr int64_t kKnnDirect = 48;

template <int K, class UseFn>
static cudaError_t points_nearest(Ctx *c, UseFn &&use)
{
    if (c->n <= kKnnDirect) {
        use(0, (int)c->n, 0, (const int *)nullptr);
        return cudaGetLastError();
    }
    const KnnTree T = knn_tree(c);
    int64_t stride = std::min<int64_t>(c->n, kKnnRange);
    ScratchScope scope(c);
    int *buf = nullptr;  // K * stride table, queue, its length
    cudaError_t e;
    while ((e = scratch_get(c, &buf, ((K + 1) * stride + 1) * sizeof(int))) ==
               cudaErrorMemoryAllocation &&
           stride > kKnnRangeMin)
        stride = std::max(kKnnRangeMin, ceil_div(stride, 2));
    if (e != cudaSuccess) return e;
    int *queue = buf + K * stride, *nq = queue + stride;
    for (int64_t i0 = 0; i0 < c->n && e == cudaSuccess; i0 += stride) {
        const int cnt = (int)std::min<int64_t>(stride, c->n - i0);
        e = cudaMemsetAsync(nq, 0, sizeof(int), c->stream);
        if (e != cudaSuccess) break;
        k_knn_points<K><<<(unsigned)ceil_div(cnt, 32 * kShWarps), 32 * kShWarps, 0, c->stream>>>(
            T, i0, cnt, stride, buf, queue, nq);
        k_knn_points_far<<<(unsigned)std::min<int64_t>(ceil_div(cnt, kShWarps), kShFarBlocks),
                           32 * kShWarps, 0, c->stream>>>(T, i0, stride, K, buf, queue, nq,
                                                          c->d_err);
        use(i0, cnt, stride, (const int *)buf);
        e = cudaGetLastError();
    }
    return e;
}

// the neighbours of a point, from its column of the table or by a search
template <int K, bool TABLE>
__device__ __forceinline__ void point_neighbours(const KnnTree &T, float4 p, int64_t stride,
                                                 const int *__restrict__ nbr, int r, int (&bj)[K],
                                                 int *err)
{
    if constexpr (TABLE) {
#pragma unroll
        for (int t = 0; t < K; ++t) bj[t] = __ldg(&nbr[t * stride + r]);
    } else {
        knn_search<K, true>(T, F3{p.x, p.y, p.z}, K, bj, err);
    }
}

__device__ __forceinline__ uint64_t point_code(const KnnTree &T, F3 q)
{
    return morton3((uint64_t)quant21(q.x, T.cube_lo[0], T.inv_h21),
                   (uint64_t)quant21(q.y, T.cube_lo[1], T.inv_h21),
                   (uint64_t)quant21(q.z, T.cube_lo[2], T.inv_h21));
}

// position of the first code not below `code`, by the warp
__device__ __forceinline__ int64_t warp_lower_bound(const uint64_t *__restrict__ codes, int64_t n,
                                                    uint64_t code, int lane)
{
    int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
    while (hi - lo > 32) {
        const int64_t s = (hi - lo) >> 5;
        const int c = __popc(__ballot_sync(0xffffffffu, __ldg(&codes[lo + s * (lane + 1) - 1]) < code));
        if (c < 32) hi = lo + s * (c + 1) - 1;
        lo += s * c;
    }
    return lo + __popc(__ballot_sync(0xffffffffu, lo + lane < hi && __ldg(&codes[lo + lane]) < code));
}

// The scatter's additions are first summed per warp in a shared-memory
// table keyed by point (open addressing, a few probes), then each distinct
// point of the warp takes one global addition per component.  Neighbouring
// faces share most of their nearest points, and where the level set lies
// away from the points many faces share the same few; summing them in the
// warp first keeps the global atomics few and uncontended.  A table per warp
// (not per block) lets each warp leave as soon as its own faces are done.
// The sums are 64-bit fixed-point integers, so the grouping changes no bit.
// The tables take 28 KB of shared memory per block, which the SM takes from
// its L1 cache: on clouds of millions of points the searches' gathers lose
// more to the smaller cache than the tables save (a 3M-point union: 80.8 ->
// 40.7 ms with them; a 15M-point union: 49 -> 70 ms), so in k_knn_scatter
// clouds above kAggMaxPoints add straight to the points' sums.
constexpr int kAggBits = 8;
constexpr int kAggSlots = 1 << kAggBits;  // table entries per warp of 32 faces
constexpr int kAggWarps = 4;              // warps of a 128-thread block
constexpr int kAggProbes = 8;    // entries tried before adding to global memory directly
constexpr int64_t kAggMaxPoints = 4000000;
constexpr size_t kAggSmem =
    (size_t)kAggWarps * kAggSlots * (3 * sizeof(unsigned long long) + sizeof(int));

// Faces whose leaf cell has a candidate list, k = 10: a thread per face.  A
// candidate is one 32-bit key, its squared distance's bits with the low 8
// replaced by its place in the list (at most kCellCap = 256 entries), and
// the 11 smallest keys are kept sorted with integer minima and maxima alone
// (21 instructions a candidate that enters, no 64-bit compares and no index
// to move).  Cutting 8 bits can only matter when the tenth and the eleventh
// key agree above them; that face is scanned again with the full (distance,
// input index) keys.  Faces without a list are queued for k_knn_far.
// The sums per warp are 32-bit here: a face vector is below 2^25 units (8
// finest-cell areas) or goes straight to the points' sums.  At 16 KB a block
// the tables pay at every size (15M points: 37.4 / 15.4 ms straight to the
// points' sums, 36.4 / 14.9 with them).
// Bound: the gathers of the candidates (L1 wavefronts 81-85 % of their peak)
// and the integer pipe.  With k_knn_far against the one thread per face with
// 64-bit keys and its own tree search (random normals / 3rd-16th iteration):
// 2,000-point sphere 0.63 / 0.19 -> 0.10 / 0.05 ms, 100k torus 2.8 / 1.9 ->
// 0.33 / 0.18 ms, 1M blob 13.5 / 10.2 -> 5.5 / 3.8 ms, 4M union 29 / 14.5 ->
// 12.1 / 5.2 ms.  On a small cloud one face's chain of dependent loads (index,
// point, four at a time) is the time: with the next indices loading beside the
// points, and six CTAs an SM asked for rather than eight, 94 / 49 -> 84 / 41 us at 2,000
// points and 12.1 / 5.2 -> 11.5 / 4.9 ms on the 4M union; eight at a time 80 /
// 37 us but 11.9 / 5.1 ms.
constexpr int kScanK = 10;
constexpr int kTabBits = 8;
constexpr int kTabSlots = 1 << kTabBits;
constexpr int kScanWarps = 4;
constexpr size_t kTabSmem = (size_t)kScanWarps * kTabSlots * 4 * sizeof(int);
constexpr long long kTabMax = 1 << 25;

__device__ __forceinline__ void knn_lists_body(const float4 *__restrict__ faces, IterState *st,
                                               int64_t max_faces, const KnnTree &T,
                                               const int64_t *__restrict__ cell_off,
                                               const int *__restrict__ cell_idx, double scale,
                                               unsigned long long *acc, int *far_q, int64_t bid)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    const int64_t nf = min((int64_t)st->nfaces, max_faces);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (bid * blockDim.x + wid * 32 >= nf) return;  // the whole warp is past the faces
    extern __shared__ int s_tab[];
    int *s_key = s_tab + wid * 4 * kTabSlots;
    int *s_v = s_key + kTabSlots;
    for (int i = lane; i < kTabSlots; i += 32) {
        s_key[i] = -1;
        s_v[i] = s_v[kTabSlots + i] = s_v[2 * kTabSlots + i] = 0;
    }
    const int64_t f = bid * blockDim.x + threadIdx.x;
    int bj[kScanK];
#pragma unroll
    for (int t = 0; t < kScanK; ++t) bj[t] = -1;
    long long vx = 0, vy = 0, vz = 0;
    bool far = false;
    if (f < nf) {
        const float4 A = faces[2 * f], C = faces[2 * f + 1];
        const int leaf = __float_as_int(A.w);
        const int64_t c0 = __ldg(&cell_off[leaf]);
        const int len = (int)(__ldg(&cell_off[leaf + 1]) - c0);
        vx = llrint((double)A.x * scale);
        vy = llrint((double)A.y * scale);
        vz = llrint((double)A.z * scale);
        far = len <= 0;
        if (!far) {
            const int *cand = cell_idx + c0;
            const F3 q{C.x, C.y, C.z};
            unsigned b[kScanK + 1];
#pragma unroll
            for (int t = 0; t <= kScanK; ++t) b[t] = 0xffffffffu;
            // the indices of the next four load beside these four points
            int jn[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) jn[u] = __ldg(&cand[min(u, len - 1)]);
            for (int t = 0; t < len; t += 4) {
                unsigned ky[4];
                float4 pp[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) pp[u] = __ldg(&T.p4[jn[u]]);
#pragma unroll
                for (int u = 0; u < 4; ++u) jn[u] = __ldg(&cand[min(t + 4 + u, len - 1)]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float d = pt_d2(pp[u], q);
                    ky[u] = t + u < len ? (__float_as_uint(d) & 0xffffff00u) | (unsigned)(t + u)
                                        : 0xffffffffu;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (ky[u] < b[kScanK]) {
#pragma unroll
                        for (int i = kScanK; i > 0; --i) b[i] = max(b[i - 1], min(b[i], ky[u]));
                        b[0] = min(b[0], ky[u]);
                    }
                }
            }
            if ((b[kScanK - 1] >> 8) == (b[kScanK] >> 8) && b[kScanK] != 0xffffffffu) {
                knn_scan<kScanK, true>(T, q, kScanK, cell_idx, c0, c0 + len, bj);
            } else {
#pragma unroll
                for (int t = 0; t < kScanK; ++t)
                    if (b[t] != 0xffffffffu) bj[t] = __ldg(&cand[b[t] & 255u]);
            }
        }
    }
    const unsigned fm = __ballot_sync(0xffffffffu, far);
    if (fm) {
        int base = 0;
        if (lane == 0) base = atomicAdd(&st->nfar, __popc(fm));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (far) far_q[base + __popc(fm & ((1u << lane) - 1u))] = (int)f;
    }
    auto direct = [&](int j) {
        unsigned long long *a = acc + 3 * (int64_t)j;
        atomicAdd(a + 0, (unsigned long long)vx);
        atomicAdd(a + 1, (unsigned long long)vy);
        atomicAdd(a + 2, (unsigned long long)vz);
    };
    const bool small = llabs(vx) < kTabMax && llabs(vy) < kTabMax && llabs(vz) < kTabMax;
    __syncwarp();  // the table is cleared
#pragma unroll
    for (int t = 0; t < kScanK; ++t) {
        const int j = bj[t];
        if (j < 0) continue;
        bool added = false;
        if (small) {
            unsigned h = ((unsigned)j * 2654435761u) >> (32 - kTabBits);
            for (int p = 0; p < kAggProbes; ++p, h = (h + 1) & (kTabSlots - 1)) {
                const int prev = atomicCAS(&s_key[h], -1, j);
                if (prev == -1 || prev == j) {
                    atomicAdd(&s_v[h], (int)vx);
                    atomicAdd(&s_v[kTabSlots + h], (int)vy);
                    atomicAdd(&s_v[2 * kTabSlots + h], (int)vz);
                    added = true;
                    break;
                }
            }
        }
        if (!added) direct(j);  // a large vector, or a crowded table
    }
    __syncwarp();  // every addition is in the table
    for (int i = lane; i < kTabSlots; i += 32) {
        const int j = s_key[i];
        if (j < 0) continue;
        unsigned long long *a = acc + 3 * (int64_t)j;
        atomicAdd(a + 0, (unsigned long long)(long long)s_v[i]);
        atomicAdd(a + 1, (unsigned long long)(long long)s_v[kTabSlots + i]);
        atomicAdd(a + 2, (unsigned long long)(long long)s_v[2 * kTabSlots + i]);
    }
}

__global__ void __launch_bounds__(32 * kScanWarps, 6)
    k_knn_lists(const float4 *__restrict__ faces, IterState *st, int64_t max_faces, KnnTree T,
                const int64_t *__restrict__ cell_off, const int *__restrict__ cell_idx,
                double scale, unsigned long long *acc, int *far_q)
{
    knn_lists_body(faces, st, max_faces, T, cell_off, cell_idx, scale, acc, far_q, blockIdx.x);
}

// The queued faces (in cells far from the points, over kCellCap candidates),
// a warp per face: as threads of a warp their searches, of very different
// length, waited for each other and were one chain of dependent loads each.
constexpr int kFarWarps = 4;

__device__ __forceinline__ void knn_far_body(const float4 *__restrict__ faces, IterState *st,
                                             const KnnTree &T, const int *__restrict__ far_q,
                                             double scale, unsigned long long *acc, int2 *defer,
                                             int budget, int *err, int64_t bid, int64_t nblk)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    __shared__ int2 s_stack[kFarWarps][kWarpStack];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nq = st->nfar;
    for (int64_t i = bid * kFarWarps + wid; i < nq; i += nblk * kFarWarps) {
        const int f = far_q[i];
        const float4 A = faces[2 * (int64_t)f], C = faces[2 * (int64_t)f + 1];
        const F3 q{C.x, C.y, C.z};
        const int64_t seed = (int64_t)__float_as_int(C.w);
        int j, bud = budget;
        float bound = INFINITY;
        bool own = true;
        while (!warp_knn(T, q, kScanK, seed, lane, s_stack[wid], j, err, bud, &bound)) {
            int slot = 0;
            if (lane == 0) slot = atomicAdd(&st->ndefer, 1);
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if (slot < kDeferCap) {
                if (lane == 0) defer[slot] = make_int2(f, __float_as_int(bound));
                own = false;  // added by k_knn_deferred
                break;
            }
            bud = -1;
        }
        if (own && lane < kScanK && j >= 0) {
            unsigned long long *a = acc + 3 * (int64_t)j;
            atomicAdd(a + 0, (unsigned long long)llrint((double)A.x * scale));
            atomicAdd(a + 1, (unsigned long long)llrint((double)A.y * scale));
            atomicAdd(a + 2, (unsigned long long)llrint((double)A.z * scale));
        }
    }
}

__global__ void __launch_bounds__(32 * kFarWarps)
    k_knn_far(const float4 *__restrict__ faces, IterState *st, KnnTree T,
              const int *__restrict__ far_q, double scale, unsigned long long *acc, int2 *defer,
              int budget, int *err)
{
    knn_far_body(faces, st, T, far_q, scale, acc, defer, budget, err, blockIdx.x, gridDim.x);
}

// blocks of the far search's launch for a queue of at most cap faces
static int far_blocks(int64_t cap, int most)
{
    return (int)std::min<int64_t>(ceil_div(cap, kFarWarps), most);
}
constexpr int kFarBlocks = kSMs * 8;      // one cloud
constexpr int kFarBlocksBatch = 64;      // a cloud's part of a batch

// A face whose own search (no candidate list for its cell) runs past
// kSearchBudget -- a face far from the points, about as far from many of
// them, as near the centre of a sphere -- is deferred: its index and the
// bound its partial search reached go to a list that k_knn_deferred finishes
// with a whole block per face, so that no single thread holds the launch.
template <int KMAX, bool FIXED>
__device__ __forceinline__ void knn_scatter_body(const float4 *__restrict__ faces,
                                                 IterState *st, int64_t max_faces,
                                                 const KnnTree &T, int k,
                                                 const int64_t *__restrict__ cell_off,
                                                 const int *__restrict__ cell_idx, double scale,
                                                 unsigned long long *acc, int2 *defer,
                                                 int budget, bool agg, int *err, int64_t bid)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    const int64_t nf = min((int64_t)st->nfaces, max_faces);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (bid * blockDim.x + wid * 32 >= nf) return;  // the whole warp is past the faces
    // agg: kAggSmem bytes of dynamic shared memory, per warp 3 x kAggSlots
    // sums, then every warp's kAggSlots keys
    extern __shared__ unsigned long long s_agg[];
    unsigned long long *s_v = s_agg + (size_t)wid * 3 * kAggSlots;
    int *s_key = reinterpret_cast<int *>(s_agg + (size_t)kAggWarps * 3 * kAggSlots) +
                 wid * kAggSlots;
    if (agg) {
        for (int i = lane; i < kAggSlots; i += 32) {
            s_key[i] = -1;
            s_v[i] = s_v[kAggSlots + i] = s_v[2 * kAggSlots + i] = 0ull;
        }
    }
    const int64_t f = bid * blockDim.x + threadIdx.x;
    const bool active = f < nf;
    int bj[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) bj[t] = -1;
    long long vx = 0, vy = 0, vz = 0;
    if (active) {
        float4 A = faces[2 * f], C = faces[2 * f + 1];
        int64_t c0 = 0, c1 = 0;
        if (cell_off) {
            const int leaf = __float_as_int(A.w);
            c0 = __ldg(&cell_off[leaf]);
            c1 = __ldg(&cell_off[leaf + 1]);
        }
        if (c1 > c0) {
            knn_scan<KMAX, FIXED>(T, F3{C.x, C.y, C.z}, k, cell_idx, c0, c1, bj);
        } else {
            // one inlined search: budgeted first, unbounded when the list is full
            const F3 q{C.x, C.y, C.z};
            const int64_t seed = (int64_t)__float_as_int(C.w);
            int bud = budget;
            float bound = INFINITY;
            while (!knn_search<KMAX, FIXED>(T, q, k, bj, err, seed, bud, &bound)) {
                const int slot = atomicAdd(&st->ndefer, 1);
                if (slot < kDeferCap) {
                    defer[slot] = make_int2((int)f, __float_as_int(bound));
#pragma unroll
                    for (int t = 0; t < KMAX; ++t) bj[t] = -1;  // added by k_knn_deferred
                    break;
                }
                bud = -1;
            }
        }
        vx = llrint((double)A.x * scale);
        vy = llrint((double)A.y * scale);
        vz = llrint((double)A.z * scale);
    }
    if (!agg) {  // straight to the points' sums
#pragma unroll
        for (int t = 0; t < KMAX; ++t) {
            if (t >= k || bj[t] < 0) continue;
            unsigned long long *a = acc + 3 * (int64_t)bj[t];
            atomicAdd(a + 0, (unsigned long long)vx);
            atomicAdd(a + 1, (unsigned long long)vy);
            atomicAdd(a + 2, (unsigned long long)vz);
        }
        return;
    }
    __syncwarp();  // the table is cleared
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
        if (t >= k || bj[t] < 0) continue;
        const int j = bj[t];
        unsigned h = ((unsigned)j * 2654435761u) >> (32 - kAggBits);
        bool added = false;
        for (int p = 0; p < kAggProbes; ++p, h = (h + 1) & (kAggSlots - 1)) {
            const int prev = atomicCAS(&s_key[h], -1, j);
            if (prev == -1 || prev == j) {
                atomicAdd(&s_v[h], (unsigned long long)vx);
                atomicAdd(&s_v[kAggSlots + h], (unsigned long long)vy);
                atomicAdd(&s_v[2 * kAggSlots + h], (unsigned long long)vz);
                added = true;
                break;
            }
        }
        if (!added) {  // the table is crowded: straight to the point's sums
            unsigned long long *a = acc + 3 * (int64_t)j;
            atomicAdd(a + 0, (unsigned long long)vx);
            atomicAdd(a + 1, (unsigned long long)vy);
            atomicAdd(a + 2, (unsigned long long)vz);
        }
    }
    __syncwarp();  // every addition is in the table
    for (int i = lane; i < kAggSlots; i += 32) {
        const int j = s_key[i];
        if (j < 0) continue;
        unsigned long long *a = acc + 3 * (int64_t)j;
        atomicAdd(a + 0, s_v[i]);
        atomicAdd(a + 1, s_v[kAggSlots + i]);
        atomicAdd(a + 2, s_v[2 * kAggSlots + i]);
    }
}

// 8 resident blocks per SM (64 registers): the search is a chain of
// dependent loads that wants the warps
template <int KMAX, bool FIXED>
__global__ void __launch_bounds__(128, KMAX > 16 ? 1 : 8)
    k_knn_scatter(const float4 *__restrict__ faces, IterState *st, int64_t max_faces,
                  KnnTree T, int k, const int64_t *__restrict__ cell_off,
                  const int *__restrict__ cell_idx, double scale, unsigned long long *acc,
                  int2 *defer, int budget, int agg, int *err)
{
    knn_scatter_body<KMAX, FIXED>(faces, st, max_faces, T, k, cell_off, cell_idx, scale, acc,
                                  defer, budget, agg != 0, err, blockIdx.x);
}

// The deferred faces, one block per face (the blocks take the list in
// turn; 128 threads for k <= 16, 64 for up to 32 so that the lists fit the
// static shared memory).  The threads first test the bucket tree's nodes at
// one level of at most 2,048 nodes against the bound of the face's partial
// search (an upper bound of its k-th nearest distance), then split the
// buckets under the nodes that pass, skipping buckets whose box lies beyond
// the bound; each thread keeps its own k nearest under the search's
// (distance, input index) keys; thread 0 takes the k smallest of the
// block's lists -- the k points the full search finds -- and adds the
// face's vector to them.
template <int KMAX>
__host__ __device__ constexpr int defer_threads() { return KMAX > 16 ? 64 : 128; }

template <int KMAX, bool FIXED>
__device__ __forceinline__ void knn_deferred_body(const float4 *__restrict__ faces,
                                                  const IterState *st,
                                                  const int2 *__restrict__ defer,
                                                  const KnnTree &T, int k, double scale,
                                                  unsigned long long *acc, int64_t bid,
                                                  int64_t nblk)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    const int nd = min(st->ndefer, kDeferCap);
    if (bid >= nd) return;  // the same for every thread of the block
    constexpr int NT = defer_threads<KMAX>();
    __shared__ uint64_t s_key[NT * KMAX];
    __shared__ int s_j[NT * KMAX];
    __shared__ int s_head[NT];
    constexpr int kCoarseBits = 11;
    __shared__ int s_pass[1 << kCoarseBits];
    __shared__ int s_npass;
    const int kk = FIXED ? KMAX : k;
    const int64_t nleaf = (int64_t)1 << T.levels;
    const int64_t nb = (T.n + kBucket - 1) / kBucket;
    const int lc = min(T.levels, kCoarseBits);      // the coarse level
    const int64_t span = (int64_t)1 << (T.levels - lc);  // buckets under a coarse node
    for (int64_t d = bid; d < nd; d += nblk) {
        const int2 e = defer[d];
        const int64_t f = e.x;
        const float4 C = faces[2 * f + 1];
        const F3 q{C.x, C.y, C.z};
        uint64_t best[KMAX];
        int bj[KMAX];
#pragma unroll
        for (int t = 0; t < KMAX; ++t) {
            best[t] = ~0ull;
            bj[t] = -1;
        }
        float worst = __int_as_float(e.y);
        if (threadIdx.x == 0) s_npass = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < (1 << lc); i += NT) {
            const int node = (1 << lc) + i;
            if ((int64_t)i * span < nb &&
                box_d2(__ldg(&T.lo[node]), __ldg(&T.hi[node]), q) <= worst)
                s_pass[atomicAdd(&s_npass, 1)] = i;
        }
        __syncthreads();
        const int64_t total = (int64_t)s_npass * span;
        for (int64_t u = threadIdx.x; u < total; u += NT) {
            const int64_t b = (int64_t)s_pass[u / span] * span + u % span;
            if (b >= nb) continue;
            const int64_t node = nleaf + b;
            if (box_d2(__ldg(&T.lo[node]), __ldg(&T.hi[node]), q) > worst) continue;
            const int64_t j0 = b * kBucket, j1 = min(j0 + kBucket, T.n);
            for (int64_t j = j0; j < j1; ++j) {
                const float d2 = pt_d2(__ldg(&T.p4[j]), q);
                if (d2 > worst) continue;
                const uint64_t key = knn_key(d2, __ldg(&T.perm[j]));
                if (key < best[kk - 1]) {
                    knn_insert<KMAX, FIXED>(key, (int)j, k, best, bj);
                    if (best[kk - 1] != ~0ull)
                        worst = fminf(worst, __uint_as_float((uint32_t)(best[kk - 1] >> 32)));
                }
            }
        }
#pragma unroll
        for (int t = 0; t < KMAX; ++t) {
            s_key[threadIdx.x * KMAX + t] = best[t];
            s_j[threadIdx.x * KMAX + t] = bj[t];
        }
        s_head[threadIdx.x] = 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            const float4 A = faces[2 * f];
            const long long vx = llrint((double)A.x * scale);
            const long long vy = llrint((double)A.y * scale);
            const long long vz = llrint((double)A.z * scale);
            for (int r = 0; r < kk; ++r) {  // the r-th smallest key of the block
                uint64_t m = ~0ull;
                int win = -1;
                for (int t = 0; t < NT; ++t) {
                    const int hd = s_head[t];
                    if (hd < kk && s_key[t * KMAX + hd] < m) {
                        m = s_key[t * KMAX + hd];
                        win = t;
                    }
                }
                if (win < 0 || m == ~0ull) break;  // fewer than k points
                const int j = s_j[win * KMAX + s_head[win]];
                s_head[win] += 1;
                unsigned long long *a = acc + 3 * (int64_t)j;
                atomicAdd(a + 0, (unsigned long long)vx);
                atomicAdd(a + 1, (unsigned long long)vy);
                atomicAdd(a + 2, (unsigned long long)vz);
            }
        }
        __syncthreads();  // the lists are read before the next face reuses them
    }
}

template <int KMAX, bool FIXED>
__global__ void __launch_bounds__(defer_threads<KMAX>())
    k_knn_deferred(const float4 *__restrict__ faces, const IterState *st,
                   const int2 *__restrict__ defer, KnnTree T, int k, double scale,
                   unsigned long long *acc)
{
    knn_deferred_body<KMAX, FIXED>(faces, st, defer, T, k, scale, acc, blockIdx.x, gridDim.x);
}

template <int KMAX, bool FIXED>
__global__ void k_knn_query(const float4 *__restrict__ q, int64_t m, KnnTree T, int k,
                            int64_t *idx_out, int *err)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    float4 v = q[i];
    int bj[KMAX];
    knn_search<KMAX, FIXED>(T, F3{v.x, v.y, v.z}, k, bj, err);
    for (int t = 0; t < k; ++t) idx_out[i * k + t] = bj[t] >= 0 ? T.perm[bj[t]] : -1;
}

// distance from each of m sampled points (sorted indices, strided) to its
// 11th nearest point (itself included: the 10th nearest other point)
__global__ void k_spacing(KnnTree T, int64_t m, int64_t stride, float *d_out, int *err)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const float4 v = T.p4[min(i * stride, T.n - 1)];
    const F3 q = {v.x, v.y, v.z};
    int bj[11];
    knn_search<11, true>(T, q, 11, bj, err);
    d_out[i] = bj[10] >= 0 ? sqrtf(pt_d2(T.p4[bj[10]], q)) : 0.f;
}

cudaError_t launch_spacing(Ctx *c, int64_t m, float *d_out)
{
    const int64_t stride = std::max<int64_t>(1, c->n / std::max<int64_t>(m, 1));
    k_spacing<<<(unsigned)ceil_div(m, 128), 128, 0, c->stream>>>(knn_tree(c), m, stride, d_out,
                                                                 c->d_err);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// learned warm start: patch features from the 16 nearest other points
// ---------------------------------------------------------------------------
// Centroid and RMS radius about it, in FP64 relative to the bounding-box
// centre b (so that mean |p - c|^2 = mean |p - b|^2 - |c - b|^2 loses nothing):
// per-block sums in a fixed order, then one block over the blocks' sums.  As
// one block over all points it was a chain of loads: 913 us for 200,000
// points, 23 us as two launches.  Up to kSumOne points one block is enough.
constexpr int64_t kSumOne = 512;
constexpr int kSumBlocks = 2 * kSMs;

__device__ __forceinline__ double block_sum(double v, double *sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// mean offset m[0..2] from b and mean squared distance m[3] -> cx, cy, cz, R
__device__ __forceinline__ void centroid_out(const double (&m)[4], double bx, double by, double bz,
                                             double *out)
{
    out[0] = bx + m[0];
    out[1] = by + m[1];
    out[2] = bz + m[2];
    out[3] = sqrt(fmax(0.0, m[3] - (m[0] * m[0] + m[1] * m[1] + m[2] * m[2])));
}

// (one block: the result at once)
__global__ void __launch_bounds__(256)
    k_centroid_part(const float4 *__restrict__ p4, int64_t n, double bx, double by, double bz,
                    double *__restrict__ part, double *__restrict__ out)
{
    __shared__ double sh[256];
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float4 p = p4[i];
        const double dx = p.x - bx, dy = p.y - by, dz = p.z - bz;
        s[0] += dx;
        s[1] += dy;
        s[2] += dz;
        s[3] += dx * dx + dy * dy + dz * dz;
    }
    for (int k = 0; k < 4; ++k) {
        s[k] = block_sum(s[k], sh);
        if (threadIdx.x == 0) part[4 * blockIdx.x + k] = s[k];
    }
    // (the divisions by one thread: by every thread of 304 blocks they took 5 us)
    if (gridDim.x == 1 && threadIdx.x == 0) {
        for (int k = 0; k < 4; ++k) s[k] /= n;
        centroid_out(s, bx, by, bz, out);
    }
}

__global__ void __launch_bounds__(256)
    k_centroid(const double *__restrict__ part, int nb, int64_t n, double bx, double by, double bz,
               double *out)
{
    __shared__ double sh[256];
    double m[4];
    for (int k = 0; k < 4; ++k) {
        double v = 0.0;
        for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[4 * b + k];
        m[k] = block_sum(v, sh) / n;
    }
    if (threadIdx.x == 0) centroid_out(m, bx, by, bz, out);
}

// Feature row of sorted point i: offsets to its 16 nearest other points (in
// ascending order) divided by their RMS length, then (p - c) / R, zero
// padding to 64.  Rows go to row index perm[i] when by_input is set.  A thread
// makes its point's row in shared memory and the warp writes its 32 rows one
// after the other, 128 bytes a store: written a float at a time by each
// thread (32 sectors a store) 200,000 rows took 99 us, now 31.
constexpr int kFeatWarps = 4;
constexpr int kFeatRow = 51;

template <bool TABLE>
__global__ void __launch_bounds__(32 * kFeatWarps)
    k_features(KnnTree T, int64_t i0, int cnt_i, int64_t stride, const int *__restrict__ nbr,
               const double *__restrict__ cR, float *__restrict__ X, int by_input, int *err)
{
    __shared__ float rows[kFeatWarps][32][kFeatRow];
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int r0 = r - lane;
    if (r0 >= cnt_i) return;  // the whole warp
    float (*S)[kFeatRow] = rows[threadIdx.x >> 5];
    int cnt = 0;
    float inv = 0.f;
    int64_t to = 0;
    if (r < cnt_i) {
        const int64_t i = i0 + r;
        const float4 pi = T.p4[i];
        int bj[17];
        point_neighbours<17, TABLE>(T, pi, stride, nbr, r, bj, err);
        float ss = 0.f;
#pragma unroll
        for (int t = 0; t < 17; ++t) {
            const int j = bj[t];
            if (j < 0 || j == (int)i || cnt == 16) continue;
            float4 pj = T.p4[j];
            float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
            S[lane][3 * cnt] = dx;
            S[lane][3 * cnt + 1] = dy;
            S[lane][3 * cnt + 2] = dz;
            ss += dx * dx + dy * dy + dz * dz;
            ++cnt;
        }
        float s = cnt > 0 ? sqrtf(ss / cnt) : 0.f;
        inv = s > 0.f ? 1.f / s : 0.f;
        double R = cR[3];
        S[lane][48] = R > 0.0 ? (float)((pi.x - cR[0]) / R) : 0.f;
        S[lane][49] = R > 0.0 ? (float)((pi.y - cR[1]) / R) : 0.f;
        S[lane][50] = R > 0.0 ? (float)((pi.z - cR[2]) / R) : 0.f;
        to = by_input ? T.perm[i] : i;
    }
    __syncwarp();
    const int nr = min(32, cnt_i - r0);
    for (int w = 0; w < nr; ++w) {
        const int len = 3 * __shfl_sync(0xffffffffu, cnt, w);
        const float iw = __shfl_sync(0xffffffffu, inv, w);
        float *row = X + __shfl_sync(0xffffffffu, to, w) * 64;
        row[lane] = lane < len ? S[w][lane] * iw : 0.f;
        const int k = 32 + lane;
        row[k] = k < 48 ? (k < len ? S[w][k] * iw : 0.f) : k < kFeatRow ? S[w][k] : 0.f;
    }
}

// network outputs (sorted order) -> unit initial normals; an output that is
// zero or not finite keeps the random normal already in nrm
__global__ void k_normals_from_y(const float *__restrict__ Y, int64_t n, float4 *nrm)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x = Y[3 * i], y = Y[3 * i + 1], z = Y[3 * i + 2];
    float l = sqrtf(x * x + y * y + z * z);
    if (l > 1e-12f && isfinite(l)) nrm[i] = make_float4(x / l, y / l, z / l, 0.f);
}

cudaError_t launch_features(Ctx *c, float *X, bool by_input, double *cR)
{
    const int nb = c->n <= kSumOne ? 1 : (int)std::min<int64_t>(ceil_div(c->n, 256), kSumBlocks);
    k_centroid_part<<<nb, 256, 0, c->stream>>>(c->d_p4, c->n, c->bbox_c[0], c->bbox_c[1],
                                               c->bbox_c[2], cR + 4, cR);
    if (nb > 1)
        k_centroid<<<1, 256, 0, c->stream>>>(cR + 4, nb, c->n, c->bbox_c[0], c->bbox_c[1],
                                             c->bbox_c[2], cR);
    return points_nearest<17>(c, [&](int64_t i0, int cnt, int64_t stride, const int *nbr) {
        auto k = nbr ? k_features<true> : k_features<false>;
        k<<<(unsigned)ceil_div(cnt, 32 * kFeatWarps), 32 * kFeatWarps, 0, c->stream>>>(
            knn_tree(c), i0, cnt, stride, nbr, cR, X, by_input ? 1 : 0, c->d_err);
    });
}

cudaError_t launch_normals_from_y(Ctx *c, const float *Y)
{
    k_normals_from_y<<<(unsigned)ceil_div(c->n, 256), 256, 0, c->stream>>>(Y, c->n, c->d_nrm);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// PCA and Gauss-map initial normals (Sec. 5.1, "Normal Initialization")
// ---------------------------------------------------------------------------
// Unit eigenvector of the smallest eigenvalue of the symmetric 3 x 3 matrix a
// (destroyed), by cyclic Jacobi rotations: each rotation is the symmetric
// 2 x 2 Schur decomposition of Golub and Van Loan (Matrix Computations,
// Sec. 8.5) applied to the (p, q) plane.  False for the zero matrix or a
// non-finite result.
__device__ bool sym3_min_eigvec(double a[3][3], double out[3])
{
    double fro = 0.0;
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) fro += a[r][k] * a[r][k];
    if (!(fro > 0.0) || !isfinite(fro)) return false;
    double v[3][3] = {{1.0, 0.0, 0.0}, {0.0, 1.0, 0.0}, {0.0, 0.0, 1.0}};
    for (int sweep = 0; sweep < 16; ++sweep) {
        const double off = a[0][1] * a[0][1] + a[0][2] * a[0][2] + a[1][2] * a[1][2];
        if (off <= 1e-36 * fro) break;  // off-diagonal below double rounding of the entries
        for (int r = 0; r < 3; ++r) {
            const int p = r == 2 ? 1 : 0, q = r == 0 ? 1 : 2;  // (0,1), (0,2), (1,2)
            if (a[p][q] == 0.0) continue;
            const double tau = (a[q][q] - a[p][p]) / (2.0 * a[p][q]);
            const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            const double c = 1.0 / sqrt(1.0 + t * t), s = t * c;
            // A <- J^T A J and V <- V J, J the identity but for J_pp = J_qq = c,
            // J_pq = s, J_qp = -s
            for (int k = 0; k < 3; ++k) {
                const double x = a[k][p], y = a[k][q];
                a[k][p] = c * x - s * y;
                a[k][q] = s * x + c * y;
            }
            for (int k = 0; k < 3; ++k) {
                const double x = a[p][k], y = a[q][k];
                a[p][k] = c * x - s * y;
                a[q][k] = s * x + c * y;
            }
            for (int k = 0; k < 3; ++k) {
                const double x = v[k][p], y = v[k][q];
                v[k][p] = c * x - s * y;
                v[k][q] = s * x + c * y;
            }
        }
    }
    int m = 0;
    if (a[1][1] < a[m][m]) m = 1;
    if (a[2][2] < a[m][m]) m = 2;
    const double l = sqrt(v[0][m] * v[0][m] + v[1][m] * v[1][m] + v[2][m] * v[2][m]);
    if (!(l > 0.0) || !isfinite(l)) return false;
    for (int k = 0; k < 3; ++k) out[k] = v[k][m] / l;
    return true;
}

// PCA normal of sorted point i: the smallest-eigenvalue eigenvector of the
// covariance of its kPcaK nearest points (itself included), in FP64 on the
// offsets from p_i.  PCA fixes the line only; the direction is the one away
// from the bounding-box centre c (the Gauss-map side, n . (p_i - c) > 0),
// and +z, then +y, then +x where that dot product is zero.  Where the
// covariance is zero the random normal already in nrm stays.
template <bool TABLE>
__global__ void __launch_bounds__(128)
    k_init_pca(KnnTree T, int64_t i0, int cnt_i, int64_t stride, const int *__restrict__ nbr,
               double cx, double cy, double cz, float4 *__restrict__ nrm, int *err)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= cnt_i) return;
    const int64_t i = i0 + r;
    const float4 pi = T.p4[i];
    int bj[kPcaK];
    point_neighbours<kPcaK, TABLE>(T, pi, stride, nbr, r, bj, err);
    double d[kPcaK][3], mean[3] = {0.0, 0.0, 0.0};
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < kPcaK; ++t) {
        const int j = bj[t];
        if (j < 0) continue;
        const float4 pj = T.p4[j];
        d[cnt][0] = (double)pj.x - (double)pi.x;
        d[cnt][1] = (double)pj.y - (double)pi.y;
        d[cnt][2] = (double)pj.z - (double)pi.z;
        for (int k = 0; k < 3; ++k) mean[k] += d[cnt][k];
        ++cnt;
    }
    if (cnt < 1) return;
    for (int k = 0; k < 3; ++k) mean[k] /= cnt;
    double C[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
    for (int t = 0; t < cnt; ++t) {
        const double e0 = d[t][0] - mean[0], e1 = d[t][1] - mean[1], e2 = d[t][2] - mean[2];
        C[0][0] += e0 * e0; C[0][1] += e0 * e1; C[0][2] += e0 * e2;
        C[1][1] += e1 * e1; C[1][2] += e1 * e2; C[2][2] += e2 * e2;
    }
    C[1][0] = C[0][1]; C[2][0] = C[0][2]; C[2][1] = C[1][2];
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) C[r][k] /= cnt;
    double e[3];
    if (!sym3_min_eigvec(C, e)) return;
    const double side = e[0] * ((double)pi.x - cx) + e[1] * ((double)pi.y - cy) +
                        e[2] * ((double)pi.z - cz);
    const bool flip = side != 0.0
                          ? side < 0.0
                          : (e[2] < 0.0 || (e[2] == 0.0 && (e[1] < 0.0 || (e[1] == 0.0 && e[0] < 0.0))));
    const double sg = flip ? -1.0 : 1.0;
    nrm[i] = make_float4((float)(sg * e[0]), (float)(sg * e[1]), (float)(sg * e[2]), 0.f);
}

// Gauss-map normal: the direction from the bounding-box centre c to p_i, in
// FP64; a point at c keeps its random normal.
__global__ void k_init_gauss(const float4 *__restrict__ p4, int64_t n, double cx, double cy,
                             double cz, float4 *__restrict__ nrm)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 p = p4[i];
    const double dx = (double)p.x - cx, dy = (double)p.y - cy, dz = (double)p.z - cz;
    const double l = sqrt(dx * dx + dy * dy + dz * dz);
    if (l > 0.0) nrm[i] = make_float4((float)(dx / l), (float)(dy / l), (float)(dz / l), 0.f);
}

cudaError_t launch_init_pca(Ctx *c)
{
    return points_nearest<kPcaK>(c, [&](int64_t i0, int cnt, int64_t stride, const int *nbr) {
        auto k = nbr ? k_init_pca<true> : k_init_pca<false>;
        k<<<(unsigned)ceil_div(cnt, 128), 128, 0, c->stream>>>(knn_tree(c), i0, cnt, stride, nbr,
                                                               c->bbox_c[0], c->bbox_c[1],
                                                               c->bbox_c[2], c->d_nrm, c->d_err);
    });
}

cudaError_t launch_init_gauss(Ctx *c)
{
    k_init_gauss<<<(unsigned)ceil_div(c->n, 256), 256, 0, c->stream>>>(
        c->d_p4, c->n, c->bbox_c[0], c->bbox_c[1], c->bbox_c[2], c->d_nrm);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// local-Voronoi area weights (Sec. 5.1, "Computing Area Weights")
// ---------------------------------------------------------------------------
// A convex polygon of k vertices (counter-clockwise) clipped in place by the
// half-plane ax x + ay y <= b; at most CAP output vertices (a convex polygon
// gains at most one per clip; *over is set if rounding asked for more).
// FP64 runs at 1/64 of the FP32 rate here and bounds the whole kernel, so each
// vertex is tested once.  Keeping the tests' values, or the farthest vertex's
// distance to pass over seeds that cut nothing, costs more in local memory and
// conversions than it saves: with both, 1M points took 11.6 ms at m = 15 (10.7
// now), 14.5 at m = 8 (12.2) and 25.8 at m = 20 (20.6).
template <int CAP>
__device__ __forceinline__ int vor_clip(double (&px)[CAP], double (&py)[CAP], int k, double ax,
                                        double ay, double b, bool *over)
{
    double ox[CAP], oy[CAP];
    const double first = ax * px[0] + ay * py[0] - b;
    double fp = first;
    int o = 0;
    for (int t = 0; t < k; ++t) {
        const int u = t + 1 == k ? 0 : t + 1;
        const double fq = u == 0 ? first : ax * px[u] + ay * py[u] - b;
        if (fp <= 0.0) {
            if (o < CAP) { ox[o] = px[t]; oy[o] = py[t]; ++o; } else *over = true;
        }
        if ((fp < 0.0 && fq > 0.0) || (fq < 0.0 && fp > 0.0)) {
            const double s = fp / (fp - fq);
            if (o < CAP) {
                ox[o] = px[t] + s * (px[u] - px[t]);
                oy[o] = py[t] + s * (py[u] - py[t]);
                ++o;
            } else {
                *over = true;
            }
        }
        fp = fq;
    }
    for (int v = 0; v < o; ++v) {
        px[v] = ox[v];
        py[v] = oy[v];
    }
    return o;
}

// Area of a convex polygon containing the origin intersected with the disk of
// radius R about the origin: each edge (A, B) spans the triangle (0, A, B);
// the part of the edge inside the circle adds its triangle, the parts outside
// add circular sectors R^2 * angle / 2.
__device__ double vor_disk_area(const double *px, const double *py, int k, double R)
{
    double total = 0.0;
    const double R2 = R * R;
    for (int t = 0; t < k; ++t) {
        const int u = t + 1 == k ? 0 : t + 1;
        const double ax = px[t], ay = py[t], dx = px[u] - ax, dy = py[u] - ay;
        const double a = dx * dx + dy * dy, b = ax * dx + ay * dy, c = ax * ax + ay * ay - R2;
        if (a == 0.0) continue;
        const double bx = px[u], by = py[u];
        // both ends well inside the circle: so is the edge (the roots below
        // would be clamped to 0 and 1), and there are no sectors
        bool inside = c < -1e-9 * R2 && bx * bx + by * by - R2 < -1e-9 * R2;
        double s1 = 0.0, s2 = 0.0;
        if (!inside) {
            const double disc = b * b - a * c;
            if (disc > 0.0) {
                const double r = sqrt(disc);
                s1 = fmin(fmax((-b - r) / a, 0.0), 1.0);
                s2 = fmin(fmax((-b + r) / a, 0.0), 1.0);
            }
            inside = s1 == 0.0 && s2 == 1.0;
        }
        if (inside) {
            const double x2 = ax + dx, y2 = ay + dy;
            total += 0.5 * (ax * y2 - ay * x2);
            continue;
        }
        const double x1 = ax + s1 * dx, y1 = ay + s1 * dy, x2 = ax + s2 * dx, y2 = ay + s2 * dy;
        // no crossing: s1 = s2 = 0, one sector from A to B
        total += 0.5 * R2 * atan2(ax * y1 - ay * x1, ax * x1 + ay * y1);
        total += 0.5 * (x1 * y2 - y1 * x2);
        total += 0.5 * R2 * atan2(x2 * by - y2 * bx, x2 * bx + y2 * by);
    }
    return total;
}

// Cell area of sorted point i: its m nearest other points, the PCA tangent
// plane through it, the projected neighbours as Voronoi seeds, the cell of
// the origin cut to the disk of half the largest projected distance.  A
// neighbourhood with no extent gives 0 (the caller substitutes the mean).
template <int KMAX, bool FIXED, bool TABLE>
__global__ void __launch_bounds__(128)
    k_voronoi_area(KnnTree T, int64_t i0, int cnt_i, int64_t stride, const int *__restrict__ nbr,
                   int m, double *__restrict__ area, int *err)
{
    constexpr int CAP = KMAX + 4;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= cnt_i) return;
    const int64_t i = i0 + r;
    const float4 pi = T.p4[i];
    int bj[KMAX];
    if constexpr (FIXED)
        point_neighbours<KMAX, TABLE>(T, pi, stride, nbr, r, bj, err);
    else
        knn_search<KMAX, false>(T, F3{pi.x, pi.y, pi.z}, m + 1, bj, err);
    double d[KMAX][3];
    double mean[3] = {0.0, 0.0, 0.0};
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
        const int j = bj[t];
        if (t > m || j < 0 || j == (int)i || cnt == m) continue;
        const float4 pj = T.p4[j];
        d[cnt][0] = (double)pj.x - (double)pi.x;
        d[cnt][1] = (double)pj.y - (double)pi.y;
        d[cnt][2] = (double)pj.z - (double)pi.z;
        for (int k = 0; k < 3; ++k) mean[k] += d[cnt][k];
        ++cnt;
    }
    area[i] = 0.0;
    if (cnt < 1) return;
    for (int k = 0; k < 3; ++k) mean[k] /= (cnt + 1);  // p_i itself is the zero offset
    double C[3][3];
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) C[r][k] = mean[r] * mean[k];  // the zero offset's term
    for (int t = 0; t < cnt; ++t)
        for (int r = 0; r < 3; ++r)
            for (int k = 0; k < 3; ++k) C[r][k] += (d[t][r] - mean[r]) * (d[t][k] - mean[k]);
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) C[r][k] /= (cnt + 1);
    double nv[3];
    if (!sym3_min_eigvec(C, nv)) return;
    // tangent basis: e1 = normalise(n x axis least aligned with n), e2 = n x e1
    int ax = 0;
    if (fabs(nv[1]) < fabs(nv[ax])) ax = 1;
    if (fabs(nv[2]) < fabs(nv[ax])) ax = 2;
    double e1[3] = {ax == 2 ? nv[1] : (ax == 1 ? -nv[2] : 0.0),
                    ax == 0 ? nv[2] : (ax == 2 ? -nv[0] : 0.0),
                    ax == 1 ? nv[0] : (ax == 0 ? -nv[1] : 0.0)};
    const double l1 = sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
    for (int k = 0; k < 3; ++k) e1[k] /= l1;
    const double e2[3] = {nv[1] * e1[2] - nv[2] * e1[1], nv[2] * e1[0] - nv[0] * e1[2],
                          nv[0] * e1[1] - nv[1] * e1[0]};
    double qx[KMAX], qy[KMAX], R2m = 0.0;
    for (int t = 0; t < cnt; ++t) {
        qx[t] = d[t][0] * e1[0] + d[t][1] * e1[1] + d[t][2] * e1[2];
        qy[t] = d[t][0] * e2[0] + d[t][1] * e2[1] + d[t][2] * e2[2];
        R2m = fmax(R2m, qx[t] * qx[t] + qy[t] * qy[t]);
    }
    const double R = 0.5 * sqrt(R2m);
    if (!(R > 0.0)) return;
    double ax0[CAP], ay0[CAP];
    ax0[0] = -R; ay0[0] = -R; ax0[1] = R; ay0[1] = -R;
    ax0[2] = R;  ay0[2] = R;  ax0[3] = -R; ay0[3] = R;
    int k = 4;
    bool over = false;
    for (int t = 0; t < cnt && k >= 3; ++t) {
        const double r2 = qx[t] * qx[t] + qy[t] * qy[t];
        if (!(r2 > 0.0)) continue;  // a seed on the origin imposes nothing
        k = vor_clip<CAP>(ax0, ay0, k, qx[t], qy[t], 0.5 * r2, &over);
    }
    if (over) atomicOr(err, kErrGeometry);
    if (k >= 3) area[i] = vor_disk_area(ax0, ay0, k, R);
}

// mean of the positive areas: per-block sums in a fixed order, then one
// block over them (1,050 us for 1M points as one block); up to kAreaOne points
// one block is enough.  No positive area at all (a cloud of one point, or all
// copies of one): the paper's default weight 1.
constexpr int64_t kAreaOne = 2048;

__global__ void __launch_bounds__(256)
    k_area_part(const double *__restrict__ area, int64_t n, double *__restrict__ part,
                double *__restrict__ out)
{
    __shared__ double sh[256];
    double s = 0.0, c = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double a = area[i];
        if (a > 0.0) { s += a; c += 1.0; }
    }
    const double ss = block_sum(s, sh), sc = block_sum(c, sh);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = ss;
        part[2 * blockIdx.x + 1] = sc;
        if (gridDim.x == 1) out[0] = sc > 0.0 ? ss / sc : 1.0;
    }
}

__global__ void __launch_bounds__(256)
    k_area_mean(const double *__restrict__ part, int nb, double *out)
{
    __shared__ double sh[256];
    double s = 0.0, c = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        s += part[2 * b];
        c += part[2 * b + 1];
    }
    const double ss = block_sum(s, sh), sc = block_sum(c, sh);
    if (threadIdx.x == 0) out[0] = sc > 0.0 ? ss / sc : 1.0;
}

// install a_i (zero areas take the mean) into p4.w; optionally write them in
// input order
__global__ void k_area_install(const double *__restrict__ area, const double *__restrict__ mean,
                               const int64_t *__restrict__ perm, int64_t n, float4 *p4,
                               float *a_out, int *err)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = area[i] > 0.0 ? area[i] : mean[0];
    const float f = (float)a;
    if (!(f > 0.f) || !isfinite(f)) atomicOr(err, kErrNonfinite);
    p4[i].w = f;
    if (a_out) a_out[perm[i]] = f;
}

cudaError_t launch_voronoi_weights(Ctx *c, int m, double *scratch, float *a_out)
{
    cudaError_t e = cudaSuccess;
    if (m == 15)
        e = points_nearest<16>(c, [&](int64_t i0, int cnt, int64_t stride, const int *nbr) {
            auto k = nbr ? k_voronoi_area<16, true, true> : k_voronoi_area<16, true, false>;
            k<<<(unsigned)ceil_div(cnt, 128), 128, 0, c->stream>>>(knn_tree(c), i0, cnt, stride,
                                                                   nbr, m, scratch, c->d_err);
        });
    else
        k_voronoi_area<32, false, false><<<(unsigned)ceil_div(c->n, 128), 128, 0, c->stream>>>(
            knn_tree(c), 0, (int)c->n, 0, nullptr, m, scratch, c->d_err);
    if (e != cudaSuccess) return e;
    const int nb = c->n <= kAreaOne ? 1 : (int)std::min<int64_t>(ceil_div(c->n, 256), kSumBlocks);
    double *mean = scratch + c->n;
    k_area_part<<<nb, 256, 0, c->stream>>>(scratch, c->n, mean + 1, mean);
    if (nb > 1) k_area_mean<<<1, 256, 0, c->stream>>>(mean + 1, nb, mean);
    k_area_install<<<(unsigned)ceil_div(c->n, 256), 256, 0, c->stream>>>(
        scratch, scratch + c->n, c->d_perm, c->n, c->d_p4, a_out, c->d_err);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// clamp radii of the modified Poisson kernel (Sec. 5.2, "Poisson Kernels")
// ---------------------------------------------------------------------------
// delta_i = mean distance (FP64) from p_i to those of its k nearest other
// points whose distance lies in [vmin, vmax]; if none does, the mean of all
// k distances clamped to [vmin, vmax].  Stored as delta^2 in float32 (sorted
// order) and, when asked, delta in input order.
template <int KMAX, bool FIXED, bool TABLE>
__global__ void __launch_bounds__(128)
    k_clamp_delta(KnnTree T, int64_t i0, int cnt_i, int64_t stride, const int *__restrict__ nbr,
                  int k, double vmin, double vmax, float *__restrict__ delta2,
                  float *__restrict__ delta_out, int *err)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= cnt_i) return;
    const int64_t i = i0 + r;
    const float4 pi = T.p4[i];
    int bj[KMAX];
    if constexpr (FIXED)
        point_neighbours<KMAX, TABLE>(T, pi, stride, nbr, r, bj, err);
    else
        knn_search<KMAX, false>(T, F3{pi.x, pi.y, pi.z}, k + 1, bj, err);
    double sum_in = 0.0, sum_all = 0.0;
    int n_in = 0, cnt = 0;
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
        const int j = bj[t];
        if (t > k || j < 0 || j == (int)i || cnt == k) continue;
        const float4 pj = T.p4[j];
        const double dx = (double)pj.x - (double)pi.x, dy = (double)pj.y - (double)pi.y,
                     dz = (double)pj.z - (double)pi.z;
        const double d = sqrt(dx * dx + dy * dy + dz * dz);
        sum_all += d;
        ++cnt;
        if (d >= vmin && d <= vmax) {
            sum_in += d;
            ++n_in;
        }
    }
    double delta = vmin;
    if (n_in > 0) delta = sum_in / n_in;
    else if (cnt > 0) delta = fmin(fmax(sum_all / cnt, vmin), vmax);
    delta2[i] = (float)(delta * delta);
    if (delta_out) delta_out[T.perm[i]] = (float)delta;
}

cudaError_t launch_clamp_delta(Ctx *c, int k, double vmin, double vmax, float *delta_out)
{
    if (k == 10)
        return points_nearest<11>(c, [&](int64_t i0, int cnt, int64_t stride, const int *nbr) {
            auto kern = nbr ? k_clamp_delta<11, true, true> : k_clamp_delta<11, true, false>;
            kern<<<(unsigned)ceil_div(cnt, 128), 128, 0, c->stream>>>(
                knn_tree(c), i0, cnt, stride, nbr, k, vmin, vmax, c->d_delta2, delta_out, c->d_err);
        });
    k_clamp_delta<32, false, false><<<(unsigned)ceil_div(c->n, 128), 128, 0, c->stream>>>(
        knn_tree(c), 0, (int)c->n, 0, nullptr, k, vmin, vmax, c->d_delta2, delta_out, c->d_err);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// normal update (Eq. 7) and per-point change
// ---------------------------------------------------------------------------
__device__ __forceinline__ void normal_update_body(int mode, int64_t n,
                                                   unsigned long long *__restrict__ acc,
                                                   const float4 *__restrict__ wg,
                                                   const float4 *__restrict__ p4,
                                                   float4 *__restrict__ nrm,
                                                   float *__restrict__ src,
                                                   float *__restrict__ src16,
                                                   float *__restrict__ dtheta,
                                                   double *__restrict__ dn_blocks,
                                                   const IterState *st, int64_t bid)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch: normals stay
    int64_t i = bid * blockDim.x + threadIdx.x;
    double dn = 0.0;
    if (i < n) {
        float4 o = nrm[i];
        float nx = o.x, ny = o.y, nz = o.z;
        if (mode == DWG_UPDATE_LEVELSET) {
            // -sum / |sum| does not depend on the fixed-point scale: the
            // integer sums go to float (relative rounding 2^-24) and are
            // normalised in FP32 (FP64 runs at a small fraction of FP32 here)
            unsigned long long *a = acc + 3 * i;
            const float ax = __ll2float_rn((long long)a[0]);
            const float ay = __ll2float_rn((long long)a[1]);
            const float az = __ll2float_rn((long long)a[2]);
            a[0] = 0ull; a[1] = 0ull; a[2] = 0ull;
            const float len = sqrtf(fmaf(az, az, fmaf(ay, ay, ax * ax)));
            if (len > 0.f && isfinite(len)) {
                nx = -ax / len;
                ny = -ay / len;
                nz = -az / len;
            }
        } else {
            float4 g = wg[i];
            float len = sqrtf(g.x * g.x + g.y * g.y + g.z * g.z);
            if (len > 0.f && isfinite(len)) {
                nx = -g.x / len;
                ny = -g.y / len;
                nz = -g.z / len;
            }
        }
        float cx = o.y * nz - o.z * ny, cy = o.z * nx - o.x * nz, cz = o.x * ny - o.y * nx;
        float sn = sqrtf(cx * cx + cy * cy + cz * cz);
        float cs = o.x * nx + o.y * ny + o.z * nz;
        dtheta[i] = atan2f(sn, cs) * (float)(180.0 / kPi);
        float ex = nx - o.x, ey = ny - o.y, ez = nz - o.z;
        dn = (double)sqrtf(ex * ex + ey * ey + ez * ez);
        nrm[i] = make_float4(nx, ny, nz, 0.f);
        float c = p4[i].w * (float)(1.0 / (4.0 * kPi));
        float mx = c * nx, my = c * ny, mz = c * nz;
        // only the moment words of the record change: (mx, mx) as one 8-byte
        // store (no read of the position words), then (my, my, mz, mz)
        float *r = src + i * kSrcFloats;
        *reinterpret_cast<float2 *>(r + 6) = make_float2(mx, mx);
        *reinterpret_cast<float4 *>(r + 8) = make_float4(my, my, mz, mz);
        if (src16) {  // the modified kernel's records (same first 12 floats)
            float *r16 = src16 + i * kSrcFloatsClamp;
            *reinterpret_cast<float2 *>(r16 + 6) = make_float2(mx, mx);
            *reinterpret_cast<float4 *>(r16 + 8) = make_float4(my, my, mz, mz);
        }
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = dn;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) dn_blocks[bid] = sh[0];
}

__global__ void __launch_bounds__(256)
    k_normal_update(int mode, int64_t n, unsigned long long *__restrict__ acc,
                    const float4 *__restrict__ wg, const float4 *__restrict__ p4,
                    float4 *__restrict__ nrm, float *__restrict__ src,
                    float *__restrict__ src16, float *__restrict__ dtheta,
                    double *__restrict__ dn_blocks, const IterState *st)
{
    normal_update_body(mode, n, acc, wg, p4, nrm, src, src16, dtheta, dn_blocks, st, blockIdx.x);
}

// ---------------------------------------------------------------------------
// convergence: exact mean of the ceil(n/100) largest changes
// ---------------------------------------------------------------------------
constexpr int kSelThreads = 1024;

// exclusive block scan of one unsigned per thread (1024 threads)
__device__ unsigned block_scan_u(unsigned v, unsigned *warp_sums, unsigned &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    if (w == 0) {
        unsigned s = warp_sums[lane];
        unsigned si = s;
        for (int o = 1; o < 32; o <<= 1) {
            unsigned x = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += x;
        }
        warp_sums[lane] = si - s;
        if (lane == 31) warp_sums[32] = si;
    }
    __syncthreads();
    unsigned r = warp_sums[w] + incl - v;
    total = warp_sums[32];
    __syncthreads();
    return r;
}

// Among the bins of hist (nb bins, 4 per thread), find b with
// suffix(b) >= k > suffix(b + 1); returns b and the count strictly above.
__device__ void find_bin(const unsigned *hist, int nb, unsigned k, unsigned *warp_sums,
                         int *s_bin, unsigned *s_above)
{
    unsigned loc[4];
    unsigned s = 0;
    int b0 = threadIdx.x * 4;
    for (int t = 0; t < 4; ++t) {
        loc[t] = (b0 + t < nb) ? hist[b0 + t] : 0u;
        s += loc[t];
    }
    unsigned total;
    unsigned ex = block_scan_u(s, warp_sums, total);
    for (int t = 0; t < 4; ++t) {
        int b = b0 + t;
        unsigned suffix = total - ex;  // count in bins >= b
        if (b < nb && suffix >= k && suffix - loc[t] < k) {
            *s_bin = b;
            *s_above = suffix - loc[t];
        }
        ex += loc[t];
    }
    __syncthreads();
}

// The exact k-th largest change by a three-level radix select on the float
// bits (non-negative floats order like their bit patterns): bits 31..20,
// 19..8, 7..0.  Each level is a histogram over all changes by many CTAs
// (shared-memory bins, then integer atomics into the global bins: exact)
// and one CTA that finds the bin holding the k-th largest; then a grid sums
// the changes strictly above the threshold into per-block FP64 partials
// and one CTA adds the partials in a fixed order and takes the decision.
constexpr int kSelGridThreads = 256;

__device__ __forceinline__ void sel_hist_body(const float *__restrict__ dtheta, int64_t n,
                                              int level, const SelState *__restrict__ ss,
                                              unsigned *__restrict__ hist, const IterState *st,
                                              int64_t bid, int64_t nblk)
{
    if (cloud_idle(st)) return;
    __shared__ unsigned h[kSelBins];
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) h[b] = 0;
    __syncthreads();
    const unsigned *bits = reinterpret_cast<const unsigned *>(dtheta);
    const int shift = level == 0 ? 20 : (level == 1 ? 8 : 0);
    const unsigned mask = level == 2 ? 255u : 4095u;
    const int sh_hi = level == 1 ? 20 : 8;  // bits above this level's field (levels 1, 2)
    const unsigned prefix = ss->prefix;
    for (int64_t i = bid * blockDim.x + threadIdx.x; i < n; i += nblk * blockDim.x) {
        const unsigned v = bits[i];
        if (level > 0 && (v >> sh_hi) != prefix) continue;
        atomicAdd(&h[(v >> shift) & mask], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x)
        if (h[b]) atomicAdd(&hist[b], h[b]);
}

__global__ void __launch_bounds__(kSelGridThreads)
    k_sel_hist(const float *__restrict__ dtheta, int64_t n, int level,
               const SelState *__restrict__ ss, unsigned *__restrict__ hist, const IterState *st)
{
    sel_hist_body(dtheta, n, level, ss, hist, st, blockIdx.x, gridDim.x);
}

__device__ __forceinline__ void sel_find_body(int64_t n, int level, SelState *__restrict__ ss,
                                              unsigned *__restrict__ hist, const IterState *st)
{
    if (cloud_idle(st)) return;
    __shared__ unsigned warp_sums[33];
    __shared__ int s_bin;
    __shared__ unsigned s_above;
    const int nb = level == 2 ? 256 : 4096;
    if (level == 0 && threadIdx.x == 0) {
        ss->krem = (unsigned)((n + 99) / 100);
        ss->above = 0;
        ss->prefix = 0;
    }
    __syncthreads();
    find_bin(hist, nb, ss->krem, warp_sums, &s_bin, &s_above);
    if (threadIdx.x == 0) {
        ss->prefix = (ss->prefix << (level == 2 ? 8 : 12)) | (unsigned)s_bin;
        ss->above += s_above;
        ss->krem -= s_above;
    }
    for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) hist[b] = 0;  // for the next level
}

__global__ void __launch_bounds__(kSelThreads)
    k_sel_find(int64_t n, int level, SelState *__restrict__ ss, unsigned *__restrict__ hist,
               const IterState *st)
{
    sel_find_body(n, level, ss, hist, st);
}

__device__ __forceinline__ void sel_sum_body(const float *__restrict__ dtheta, int64_t n,
                                             const SelState *__restrict__ ss,
                                             double *__restrict__ part, const IterState *st,
                                             int64_t bid, int64_t nblk)
{
    if (cloud_idle(st)) return;
    __shared__ double sh[kSelGridThreads];
    const unsigned *bits = reinterpret_cast<const unsigned *>(dtheta);
    const unsigned tbits = ss->prefix;
    double s = 0.0;
    for (int64_t i = bid * blockDim.x + threadIdx.x; i < n; i += nblk * blockDim.x)
        if (bits[i] > tbits) s += (double)dtheta[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[bid] = sh[0];
}

__global__ void __launch_bounds__(kSelGridThreads)
    k_sel_sum(const float *__restrict__ dtheta, int64_t n, const SelState *__restrict__ ss,
              double *__restrict__ part, const IterState *st)
{
    sel_sum_body(dtheta, n, ss, part, st, blockIdx.x, gridDim.x);
}

// the statistic, the trace and the loop condition (one thread)
__device__ __forceinline__ void sel_decide(int64_t n, float tol, int rule, unsigned prefix,
                                           unsigned above, double sum_above, double sum_dn,
                                           IterState *st, double *tr_iso, double *tr_stat,
                                           double *tr_dn, long long *tr_faces,
                                           cudaGraphConditionalHandle cond, int use_cond)
{
    const unsigned k = (unsigned)((n + 99) / 100);
    const float tval = __uint_as_float(prefix);
    double stat = (sum_above + (double)(k - above) * (double)tval) / (double)k;
    int it = st->iter;
    st->stat = stat;
    if (tr_iso && it < st->max_iters) {
        tr_iso[it] = st->iso;
        tr_stat[it] = stat;
        tr_dn[it] = sum_dn / (double)n;
        tr_faces[it] = st->nfaces;
    }
    it += 1;
    st->iter = it;
    // rule 0: mean of the largest 1 % of the changes <= tol degrees (Sec. 5.1);
    // rule 1: mean |n_new - n_old| over all points <= 2 sin(tol / 2), the
    // chord of tol degrees (the measure plotted in Fig. 6)
    int done;
    if (rule == 1) {
        const double chord = 2.0 * sin((double)tol * (kPi / 360.0));
        done = sum_dn / (double)n <= chord;
    } else {
        done = stat <= (double)tol;
    }
    st->done = done;
    if (use_cond) cudaGraphSetConditional(cond, (!done && it < st->max_iters) ? 1u : 0u);
}

__device__ __forceinline__ void sel_final_body(int64_t n, float tol, int rule,
                                               const SelState *__restrict__ ss,
                                               const double *__restrict__ part, int npart,
                                               IterState *st,
                                               const double *__restrict__ dn_blocks, int ndn,
                                               double *tr_iso, double *tr_stat, double *tr_dn,
                                               long long *tr_faces,
                                               cudaGraphConditionalHandle cond, int use_cond)
{
    if (cloud_idle(st)) return;  // finished cloud of a batch
    __shared__ double sh[kSelThreads];
    double s = 0.0;
    for (int b = threadIdx.x; b < npart; b += blockDim.x) s += part[b];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    const double sum_above = sh[0];
    __syncthreads();
    double dn = 0.0;
    for (int b = threadIdx.x; b < ndn; b += blockDim.x) dn += dn_blocks[b];
    sh[threadIdx.x] = dn;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        sel_decide(n, tol, rule, ss->prefix, ss->above, sum_above, sh[0], st, tr_iso, tr_stat,
                   tr_dn, tr_faces, cond, use_cond);
}

__global__ void __launch_bounds__(kSelThreads)
    k_sel_final(int64_t n, float tol, int rule, const SelState *__restrict__ ss,
                const double *__restrict__ part, int npart, IterState *st,
                const double *__restrict__ dn_blocks, int ndn, double *tr_iso, double *tr_stat,
                double *tr_dn, long long *tr_faces, cudaGraphConditionalHandle cond, int use_cond)
{
    sel_final_body(n, tol, rule, ss, part, npart, st, dn_blocks, ndn, tr_iso, tr_stat, tr_dn,
                   tr_faces, cond, use_cond);
}

// The whole selection of a small cloud in one CTA: the changes in registers,
// the bins in shared memory, no launch between the levels.  The sum's
// partials are those of k_sel_sum's blocks, a warp each, added in the order
// of its tree, so the statistic is the same bits either way.  It is bound by
// the chain of barriers and by the adds of one SM: 12 us in place of 39 for the
// eight launches at 2,000 points, 18 at 16,384, where a cloud's other phases
// take 580; the limit is what a thread holds in registers.
constexpr int kSelSmallPer = 16;
constexpr int64_t kSelSmallMax = kSelSmallPer * kSelThreads;

__device__ __forceinline__ void sel_small_body(const float *__restrict__ dtheta, int64_t n,
                                               float tol, int rule, IterState *st,
                                               const double *__restrict__ dn_blocks,
                                               double *tr_iso, double *tr_stat, double *tr_dn,
                                               long long *tr_faces,
                                               cudaGraphConditionalHandle cond, int use_cond)
{
    if (cloud_idle(st)) return;
    __shared__ unsigned h[2 * kSelBins + 256];  // the three levels' bins
    __shared__ unsigned warp_sums[33];
    __shared__ int s_bin;
    __shared__ unsigned s_above;
    __shared__ double part[32];
    static_assert(kSelSmallMax <= 32 * 4 * kSelGridThreads && kSelSmallMax <= 64 * 256, "sums");
    const unsigned *bits = reinterpret_cast<const unsigned *>(dtheta);
    unsigned v[kSelSmallPer];
#pragma unroll
    for (int j = 0; j < kSelSmallPer; ++j) {
        const int64_t i = threadIdx.x + (int64_t)j * kSelThreads;
        v[j] = i < n ? bits[i] : 0u;
    }
    for (int b = threadIdx.x; b < 2 * kSelBins + 256; b += kSelThreads) h[b] = 0;
    __syncthreads();
    unsigned prefix = 0, above = 0, krem = (unsigned)((n + 99) / 100);
    for (int level = 0; level < 3; ++level) {
        unsigned *hl = h + level * kSelBins;
        const int shift = level == 0 ? 20 : (level == 1 ? 8 : 0);
        const unsigned mask = level == 2 ? 255u : 4095u;
        const int sh_hi = level == 1 ? 20 : 8;
#pragma unroll
        for (int j = 0; j < kSelSmallPer; ++j)
            if (threadIdx.x + (int64_t)j * kSelThreads < n &&
                (level == 0 || (v[j] >> sh_hi) == prefix))
                atomicAdd(&hl[(v[j] >> shift) & mask], 1u);
        __syncthreads();
        find_bin(hl, level == 2 ? 256 : 4096, krem, warp_sums, &s_bin, &s_above);
        prefix = (prefix << (level == 2 ? 8 : 12)) | (unsigned)s_bin;
        above += s_above;
        krem -= s_above;  // (written again behind the next level's first barrier)
    }
    const int nblk = (int)((n + 4 * kSelGridThreads - 1) / (4 * kSelGridThreads));
    const int lane = threadIdx.x & 31;
    for (int b = threadIdx.x >> 5; b < nblk; b += kSelThreads / 32) {
        double p[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            p[q] = 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t i =
                    ((int64_t)k * nblk + b) * kSelGridThreads + 32 * q + lane;
                const unsigned u = i < n ? bits[i] : 0u;
                // one change in a hundred counts: most warps skip the add
                if (__any_sync(0xffffffffu, u > prefix))
                    if (u > prefix) p[q] += (double)__uint_as_float(u);
            }
        }
        double t = ((p[0] + p[4]) + (p[2] + p[6])) + ((p[1] + p[5]) + (p[3] + p[7]));
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) part[b] = t;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    // k_sel_final's trees, whose other entries are zero
    const int ndn = (int)((n + 255) / 256);
    double sum = lane < nblk ? part[lane] : 0.0;
    double dn = (lane < ndn ? dn_blocks[lane] : 0.0) + (lane + 32 < ndn ? dn_blocks[lane + 32] : 0.0);
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_down_sync(0xffffffffu, sum, o);
        dn += __shfl_down_sync(0xffffffffu, dn, o);
    }
    if (lane == 0)
        sel_decide(n, tol, rule, prefix, above, sum, dn, st, tr_iso, tr_stat, tr_dn, tr_faces, cond,
                   use_cond);
}

__global__ void __launch_bounds__(kSelThreads)
    k_sel_small(const float *__restrict__ dtheta, int64_t n, float tol, int rule, IterState *st,
                const double *__restrict__ dn_blocks, double *tr_iso, double *tr_stat,
                double *tr_dn, long long *tr_faces, cudaGraphConditionalHandle cond, int use_cond)
{
    sel_small_body(dtheta, n, tol, rule, st, dn_blocks, tr_iso, tr_stat, tr_dn, tr_faces, cond,
                   use_cond);
}

// ---------------------------------------------------------------------------
// random unit normals from splitmix64 (stream 7)
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_random_normals(float4 *nrm, const int64_t *perm, int64_t n, uint64_t key)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t j = (uint64_t)perm[i];
    const uint64_t G = 0x9E3779B97F4A7C15ull;
    uint64_t a = mix64(key + (2 * j + 1) * G), b = mix64(key + (2 * j + 2) * G);
    double u0 = (double)(a >> 11) * 0x1.0p-53, u1 = (double)(b >> 11) * 0x1.0p-53;
    double z = 1.0 - 2.0 * u0;
    double phi = 2.0 * kPi * u1;
    double s = sqrt(fmax(0.0, 1.0 - z * z));
    nrm[i] = make_float4((float)(s * cos(phi)), (float)(s * sin(phi)), (float)z, 0.f);
}

cudaError_t launch_random_normals(float4 *nrm, const int64_t *perm, int64_t n, uint64_t seed,
                                  cudaStream_t s)
{
    uint64_t key = mix64(((seed & 0xFFFFFFFFull) << 32) | 7ull);
    k_random_normals<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(nrm, perm, n, key);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static KnnTree knn_tree(const Ctx *c)
{
    KnnTree T;
    T.p4 = c->d_p4;
    T.perm = c->d_perm;
    T.n = c->n;
    T.lo = c->d_bvh_lo;
    T.hi = c->d_bvh_hi;
    T.levels = c->knn_levels;
    T.codes = c->d_codes;
    for (int k = 0; k < 3; ++k) T.cube_lo[k] = c->cube_lo[k];
    T.inv_h21 = (double)(1 << kMortonBits) / c->cube_L;
    return T;
}

cudaError_t launch_iso(Ctx *c)
{
    k_iso<<<1, 256, 0, c->stream>>>(c->d_wsum_blocks, c->wsum_blocks, c->n, c->d_state);
    return cudaGetLastError();
}

bool cell_lists_ready(const Ctx *c)
{
    return c->knn_lists && c->cells_k == c->knn && c->d_cell_off;
}

int knn_phase_blocks(const Ctx *c, int phase)
{
    if (!cell_lists_ready(c)) return 0;
    if (phase == kPhKnnLists) return (int)ceil_div(c->max_faces, 32 * kScanWarps);
    return far_blocks(c->far_cap, kFarBlocksBatch);
}

// A cloud's entry of the batched iteration's table: the same arguments its
// own launches pass (launch_reduce_points with the points as queries,
// launch_iso, launch_reduce_w, launch_mc_faces, launch_knn_scatter,
// launch_normal_update, launch_select, launch_tree_moments, the list
// evaluation); valid while the cloud's buffers stay (the batch graph's
// generation covers them).
void fill_cloud_iter(const Ctx *c, CloudIter *o)
{
    memset(o, 0, sizeof *o);
    o->st = c->d_state;
    o->err = c->d_err;
    o->counter = c->d_counter;
    o->n = c->n;
    o->ep = make_eval_params(c);
    o->part_p = c->d_part_p;
    o->nchunks_p = c->nchunks_p;
    o->p4 = c->d_p4;
    o->src = c->d_src;
    o->codes = c->d_codes;
    for (int k = 0; k < 3; ++k) o->cq.lo[k] = c->cube_lo[k];
    o->cq.inv_h21 = (double)(1 << kMortonBits) / c->cube_L;
    o->wg = c->d_wg;
    o->wsum_blocks = c->d_wsum_blocks;
    o->wsum_nb = c->wsum_blocks;
    o->part_c = c->d_part_c;
    o->nchunks_c = c->nchunks_c;
    o->ncorners = c->ncorners;
    const bool lat = !use_tree(c) && corners_on_lattice(c);
    o->lat_corner = lat ? c->d_lat_corner : nullptr;
    o->lat_slots = lat ? corners_slots(c) : 0;
    o->wc = c->d_wc;
    o->leaf_corners = c->d_leaf_corners;
    o->leaves = c->d_leaves;
    o->nleaves = c->nleaves;
    o->corner_pos = c->d_corner_pos;
    o->faces = c->d_faces;
    o->max_faces = c->max_faces;
    o->defer = c->d_defer;
    o->knn_budget = c->knn_budget;
    o->T = knn_tree(c);
    o->k = c->knn;
    const bool lists = cell_lists_ready(c);
    o->cell_off = lists ? c->d_cell_off : nullptr;
    o->cell_idx = lists ? c->d_cell_idx : nullptr;
    o->far_q = lists ? c->d_far_q : nullptr;
    o->acc_scale = c->acc_scale;
    o->acc = c->d_acc;
    o->mode = c->mode;
    o->nrm = c->d_nrm;
    o->nrm_c = c->d_nrm;
    o->src_rw = c->d_src;
    o->dtheta = c->d_dtheta;
    o->dn_blocks = c->d_dn_blocks;
    o->sel = c->d_sel;
    o->sel_hist = c->d_sel_hist;
    o->sel_part = c->d_sel_part;
    o->sel_nb = select_blocks(c->n);
    o->tol = c->tol;
    o->conv_rule = c->conv_rule;
    o->tr_iso = c->d_tr_iso;
    o->tr_stat = c->d_tr_stat;
    o->tr_dn = c->d_tr_dn;
    o->tr_faces = c->d_tr_faces;
    o->tree = use_tree(c) ? 1 : 0;
    o->levels = c->tree_levels;
    o->bucket = c->tree_leaf;
    o->tree_M = c->d_tree_M;
    o->tree_rec = c->d_tree_rec;
    o->tree_mrec = c->d_tree_mrec;
    o->tree_frec = c->d_tree_frec;
    const TreeLists *L[2] = {&c->lists_p, &c->lists_c};
    float *lp[2] = {c->d_part_p, c->d_part_c};
    for (int w = 0; w < 2; ++w) {
        o->lq[w] = L[w]->q;
        o->lm[w] = L[w]->m;
        o->far_off[w] = L[w]->d_far_off;
        o->near_off[w] = L[w]->d_near_off;
        o->item_off[w] = L[w]->d_item_off;
        o->far_ids[w] = L[w]->d_far;
        o->near_ids[w] = L[w]->d_near;
        o->items[w] = L[w]->d_items;
        o->nitems[w] = L[w]->nitems;
        o->irec[w] = L[w]->irec;
        o->ipart[w] = L[w]->d_ipart;
        o->lpart[w] = lp[w];
    }
}

cudaError_t launch_mc_faces(Ctx *c)
{
    k_mc_faces<<<(unsigned)ceil_div(c->nleaves, 256), 256, 0, c->stream>>>(
        c->d_leaf_corners, c->d_leaves, c->nleaves, c->d_corner_pos, c->d_wc, c->d_codes, c->n,
        c->d_state, c->d_faces, c->max_faces, c->d_err);
    return cudaGetLastError();
}

cudaError_t launch_knn_scatter(Ctx *c)
{
    // one thread per possible face; threads past the emitted count exit
    unsigned blocks = (unsigned)ceil_div(c->max_faces, 128);
    KnnTree T = knn_tree(c);
    const bool lists = cell_lists_ready(c);
    const int64_t *off = lists ? c->d_cell_off : nullptr;
    const int *idx = lists ? c->d_cell_idx : nullptr;
    // k_knn_scatter's per-warp sum tables (dynamic shared memory) on clouds up
    // to kAggMaxPoints; batched clouds always take them
    const int agg = c->n <= kAggMaxPoints ? 1 : 0;
    const size_t smem = agg ? kAggSmem : 0;
    if (lists && c->knn == kScanK) {
        k_knn_lists<<<blocks, 32 * kScanWarps, kTabSmem, c->stream>>>(
            c->d_faces, c->d_state, c->max_faces, T, off, idx, c->acc_scale, c->d_acc, c->d_far_q);
        if (c->far_cap > 0) {
            k_knn_far<<<far_blocks(c->far_cap, kFarBlocks), 32 * kFarWarps, 0, c->stream>>>(
                c->d_faces, c->d_state, T, c->d_far_q, c->acc_scale, c->d_acc, c->d_defer,
                c->knn_budget, c->d_err);
            k_knn_deferred<10, true><<<kDeferBlocks, defer_threads<10>(), 0, c->stream>>>(
                c->d_faces, c->d_state, c->d_defer, T, c->knn, c->acc_scale, c->d_acc);
        }
    } else if (c->knn == 10) {
        k_knn_scatter<10, true><<<blocks, 128, smem, c->stream>>>(
            c->d_faces, c->d_state, c->max_faces, T, c->knn, off, idx, c->acc_scale, c->d_acc,
            c->d_defer, c->knn_budget, agg, c->d_err);
        k_knn_deferred<10, true><<<kDeferBlocks, defer_threads<10>(), 0, c->stream>>>(
            c->d_faces, c->d_state, c->d_defer, T, c->knn, c->acc_scale, c->d_acc);
    } else {
        k_knn_scatter<32, false><<<blocks, 128, smem, c->stream>>>(
            c->d_faces, c->d_state, c->max_faces, T, c->knn, off, idx, c->acc_scale, c->d_acc,
            c->d_defer, c->knn_budget, agg, c->d_err);
        k_knn_deferred<32, false><<<kDeferBlocks, defer_threads<32>(), 0, c->stream>>>(
            c->d_faces, c->d_state, c->d_defer, T, c->knn, c->acc_scale, c->d_acc);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// per-leaf candidate lists of the faces' k nearest points
// ---------------------------------------------------------------------------
// A face lies in its leaf cell.  With c' the cell centre rounded to float and
// h' >= |x - c'| for every x of the cell (half-diagonal plus the rounding of
// c' and of a face centroid), the k nearest points of c' lie within r_k(c')
// of c', so within r_k(c') + h' of any x: x's k nearest lie within
// R = r_k(c') + 2 h' of c'.  R is widened by a relative 1e-4 and an absolute
// 2^-17 of the coordinates so that float32 distance rounding cannot drop a
// point; extra candidates cost time, never the result.
constexpr int kCellCap = 256;

__device__ __forceinline__ void cell_centre(int4 L, int d, const KnnTree &T, double cube_L,
                                            F3 &cf, double &hp)
{
    const uint64_t code = (uint64_t)(uint32_t)L.y | ((uint64_t)(uint32_t)L.z << 32);
    const double hd = cube_L / (double)(1ll << d);  // finest cell edge
    const double e = hd * (double)(1ll << (d - L.x)); // this cell's edge
    const double cx = T.cube_lo[0] + (double)(compact3(code) << (d - L.x)) * hd + 0.5 * e;
    const double cy = T.cube_lo[1] + (double)(compact3(code >> 1) << (d - L.x)) * hd + 0.5 * e;
    const double cz = T.cube_lo[2] + (double)(compact3(code >> 2) << (d - L.x)) * hd + 0.5 * e;
    cf = F3{(float)cx, (float)cy, (float)cz};
    const double mag = fabs(cx) + fabs(cy) + fabs(cz) + e;
    hp = 0.5 * e * 1.7320508075688772 + ldexp(mag, -17);
}

// A warp's leaf centres (consecutive leaves, neighbours in space) and a
// sorted position near them; past the last leaf the last one is repeated.
__device__ __forceinline__ bool cell_warp(const int4 *__restrict__ leaves, int64_t nl, int d,
                                          const KnnTree &T, double cube_L, int lane, int64_t &l,
                                          F3 &cf, double &hp)
{
    l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l - lane >= nl) return false;  // the whole warp
    cell_centre(leaves[min(l, nl - 1)], d, T, cube_L, cf, hp);
    return true;
}

// R^2 of a leaf from the squared distance of its centre's k-th nearest point
// (INFINITY: fewer than k points, every point is a candidate)
__device__ __forceinline__ float cell_r2(float dk, F3 cf, double hp)
{
    if (dk == INFINITY) return INFINITY;
    const double rk = sqrt((double)dk);
    const double R = (rk + 2.0 * hp) * (1.0 + 1e-4) + ldexp(fabs((double)cf.x) + fabs((double)cf.y) +
                                                             fabs((double)cf.z) + rk, -17);
    return __double2float_ru(R * R);
}

// k = 10: the leaves whose search does not end within the warp's buckets go
// to the queue (a warp each, k_cell_radius_far)
__global__ void __launch_bounds__(32 * kShWarps)
    k_cell_radius(const int4 *__restrict__ leaves, int64_t nl, int d, double cube_L, KnnTree T,
                  float *__restrict__ R2, int *__restrict__ queue, int *nqueue)
{
    __shared__ ShSmem S[kShWarps];
    const int lane = threadIdx.x & 31;
    int64_t l;
    F3 cf;
    double hp;
    if (!cell_warp(leaves, nl, d, T, cube_L, lane, l, cf, hp)) return;
    const F3 c0{__shfl_sync(0xffffffffu, cf.x, 16), __shfl_sync(0xffffffffu, cf.y, 16),
                __shfl_sync(0xffffffffu, cf.z, 16)};
    const int64_t seed = warp_lower_bound(T.codes, T.n, point_code(T, c0), lane);
    float b[kScanK];
    int nv;
    const bool far = sh_smallest<kScanK>(T, cf, seed, lane, S[threadIdx.x >> 5], &nv, b) && l < nl;
    const unsigned fm = __ballot_sync(0xffffffffu, far);
    if (fm) {
        int base = 0;
        if (lane == 0) base = atomicAdd(nqueue, __popc(fm));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (far) queue[base + __popc(fm & ((1u << lane) - 1u))] = (int)l;
    }
    if (l < nl && !far) R2[l] = cell_r2(b[kScanK - 1], cf, hp);
}

__global__ void __launch_bounds__(32 * kShWarps)
    k_cell_radius_far(const int4 *__restrict__ leaves, int d, double cube_L, KnnTree T,
                      float *__restrict__ R2, const int *__restrict__ queue,
                      const int *__restrict__ nqueue, int *err)
{
    __shared__ int2 s_stack[kShWarps][kWarpStack];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nq = *nqueue;
    for (int u = blockIdx.x * kShWarps + wid; u < nq; u += gridDim.x * kShWarps) {
        const int l = queue[u];
        F3 cf;
        double hp;
        cell_centre(leaves[l], d, T, cube_L, cf, hp);
        int j;
        float bound;
        warp_knn(T, cf, kScanK, warp_lower_bound(T.codes, T.n, point_code(T, cf), lane), lane,
                 s_stack[wid], j, err, -1, &bound);
        const int last = __shfl_sync(0xffffffffu, j, kScanK - 1);
        if (lane == 0) R2[l] = cell_r2(last < 0 ? INFINITY : pt_d2(T.p4[last], cf), cf, hp);
    }
}

// any k, a thread per leaf
template <int KMAX>
__global__ void __launch_bounds__(128)
    k_cell_radius_k(const int4 *__restrict__ leaves, int64_t nl, int d, double cube_L, KnnTree T,
                    int k, float *__restrict__ R2, int *err)
{
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nl) return;
    F3 cf;
    double hp;
    cell_centre(leaves[l], d, T, cube_L, cf, hp);
    int bj[KMAX];
    knn_search<KMAX, false>(T, cf, k, bj, err);
    const int last = bj[k - 1];
    R2[l] = cell_r2(last < 0 ? INFINITY : pt_d2(T.p4[last], cf), cf, hp);
}

// points within the radius (FILL: write them; otherwise count, 0 above the
// cap), one walk of the tree per warp of leaves
template <bool FILL>
__global__ void __launch_bounds__(32 * kShWarps)
    k_cell_lists(const int4 *__restrict__ leaves, int64_t nl, int d, double cube_L, KnnTree T,
                 const float *__restrict__ R2, const int64_t *__restrict__ off,
                 int *__restrict__ idx, int64_t *__restrict__ cnt, int *err)
{
    __shared__ int stack[kShWarps][kShStack];
    const int lane = threadIdx.x & 31;
    int64_t l;
    F3 cf;
    double hp;
    if (!cell_warp(leaves, nl, d, T, cube_L, lane, l, cf, hp)) return;
    const bool valid = l < nl;
    float r2 = valid ? R2[l] : -1.f;  // -1: this lane needs nothing (more)
    int64_t o0 = 0;
    int room = kCellCap;
    if (FILL) {
        o0 = valid ? off[l] : 0;
        room = valid ? (int)(off[l + 1] - o0) : 0;
        if (room <= 0) r2 = -1.f;
    }
    if (!__any_sync(0xffffffffu, r2 >= 0.f)) {
        if (!FILL && valid) cnt[l] = 0;
        return;
    }
    int count = 0;
    sh_walk(
        T, cf, lane, stack[threadIdx.x >> 5], [&]() { return r2; },
        [&](int bucket) {
            const int64_t j0 = (int64_t)bucket * kBucket;
            if (j0 >= T.n) return true;  // an empty leaf of the complete tree
            const int c = (int)min((int64_t)kBucket, T.n - j0);
#pragma unroll 4
            for (int u = 0; u < c; ++u)
                if (pt_d2(__ldg(&T.p4[j0 + u]), cf) <= r2) {
                    if (FILL && count < room) idx[o0 + count] = (int)j0 + u;
                    ++count;
                }
            if (!FILL && count > kCellCap) r2 = -1.f;  // over the cap: no list
            return true;
        });
    if (!valid) return;
    if (!FILL) cnt[l] = count > kCellCap ? 0 : count;
    else if (room > 0 && count != room) atomicOr(err, kErrOverflow);  // the two passes must agree
}

// leaves without a list (their faces go to the far queue, up to six a leaf)
__global__ void __launch_bounds__(256)
    k_cells_without(const int64_t *__restrict__ cnt, int64_t nl, unsigned long long *out)
{
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int none = __syncthreads_count(l < nl && cnt[l] == 0);
    if (threadIdx.x == 0 && none) atomicAdd(out, (unsigned long long)none);
}

void free_cell_lists(Ctx *c)
{
    cudaFree(c->d_cell_off);
    cudaFree(c->d_cell_idx);
    cudaFree(c->d_far_q);
    c->d_cell_off = nullptr;
    c->d_cell_idx = nullptr;
    c->d_far_q = nullptr;
    c->far_cap = 0;
    c->cells_k = 0;
}

int build_cell_lists(Ctx *c)
{
    if (!c->knn_lists || c->nleaves < 1) return DWG_OK;
    if (c->cells_k == c->knn && c->d_cell_off) return DWG_OK;
    free_cell_lists(c);
    ++c->bufgen;  // a captured graph holds the old pointers
    const int64_t nl = c->nleaves;
    const int d = c->built_depth;
    KnnTree T = knn_tree(c);
    float *R2 = nullptr;
    int64_t *cnt = nullptr, *tot = nullptr;
    int *queue = nullptr;
    auto body = [&]() -> int {
        DWG_CUDA_TRY(c, cudaMalloc(&R2, nl * sizeof(float)));
        DWG_CUDA_TRY(c, cudaMalloc(&cnt, nl * sizeof(int64_t)));
        DWG_CUDA_TRY(c, cudaMalloc(&tot, 2 * sizeof(int64_t)));
        DWG_CUDA_TRY(c, cudaMalloc(&c->d_cell_off, (nl + 1) * sizeof(int64_t)));
        const unsigned g = (unsigned)ceil_div(nl, 128);
        if (c->knn == kScanK) {
            DWG_CUDA_TRY(c, cudaMalloc(&queue, (nl + 1) * sizeof(int)));
            DWG_CUDA_TRY(c, cudaMemsetAsync(queue + nl, 0, sizeof(int), c->stream));
            k_cell_radius<<<g, 128, 0, c->stream>>>(c->d_leaves, nl, d, c->cube_L, T, R2, queue,
                                                    queue + nl);
            k_cell_radius_far<<<(unsigned)std::min<int64_t>(ceil_div(nl, kShWarps), kShFarBlocks),
                                32 * kShWarps, 0, c->stream>>>(c->d_leaves, d, c->cube_L, T, R2,
                                                               queue, queue + nl, c->d_err);
        } else {
            k_cell_radius_k<32><<<g, 128, 0, c->stream>>>(c->d_leaves, nl, d, c->cube_L, T, c->knn,
                                                          R2, c->d_err);
        }
        k_cell_lists<false><<<g, 128, 0, c->stream>>>(c->d_leaves, nl, d, c->cube_L, T, R2,
                                                      nullptr, nullptr, cnt, c->d_err);
        int rc = scan_i64(c, cnt, c->d_cell_off, nl, tot);
        if (rc) return rc;
        DWG_CUDA_TRY(c, cudaMemsetAsync(tot + 1, 0, sizeof(int64_t), c->stream));
        k_cells_without<<<(unsigned)ceil_div(nl, 256), 256, 0, c->stream>>>(
            cnt, nl, reinterpret_cast<unsigned long long *>(tot + 1));
        int64_t ht[2] = {0, 0};
        DWG_CUDA_TRY(c, cudaMemcpyAsync(ht, tot, sizeof ht, cudaMemcpyDeviceToHost, c->stream));
        DWG_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        const int64_t total = ht[0];
        c->far_cap = 6 * ht[1];
        DWG_CUDA_TRY(c, cudaMalloc(&c->d_far_q, std::max<int64_t>(c->far_cap, 1) * sizeof(int)));
        DWG_CUDA_TRY(c, cudaMemcpyAsync(c->d_cell_off + nl, tot, sizeof(int64_t),
                                        cudaMemcpyDeviceToDevice, c->stream));
        // lists only where they fit comfortably (a quarter of the free memory)
        size_t fr = 0, tt = 0;
        cudaMemGetInfo(&fr, &tt);
        if ((size_t)total * sizeof(int) > fr / 4) return DWG_ERR_OOM;
        DWG_CUDA_TRY(c, cudaMalloc(&c->d_cell_idx, std::max<int64_t>(total, 1) * sizeof(int)));
        k_cell_lists<true><<<g, 128, 0, c->stream>>>(c->d_leaves, nl, d, c->cube_L, T, R2,
                                                     c->d_cell_off, c->d_cell_idx, nullptr,
                                                     c->d_err);
        DWG_CUDA_TRY(c, cudaGetLastError());
        DWG_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        c->cells_k = c->knn;
        return DWG_OK;
    };
    int rc = body();
    cudaFree(R2);
    cudaFree(cnt);
    cudaFree(tot);
    cudaFree(queue);
    if (rc) {
        free_cell_lists(c);  // the tree search serves every face
        if (rc == DWG_ERR_OOM) rc = DWG_OK;
    }
    return rc;
}

cudaError_t launch_knn_query(Ctx *c, const float4 *q, int64_t m, int k, int64_t *idx_out)
{
    KnnTree T = knn_tree(c);
    unsigned blocks = (unsigned)ceil_div(m, 128);
    if (k == 10)
        k_knn_query<10, true><<<blocks, 128, 0, c->stream>>>(q, m, T, k, idx_out, c->d_err);
    else
        k_knn_query<32, false><<<blocks, 128, 0, c->stream>>>(q, m, T, k, idx_out, c->d_err);
    return cudaGetLastError();
}

cudaError_t launch_normal_update(Ctx *c)
{
    k_normal_update<<<(unsigned)ceil_div(c->n, 256), 256, 0, c->stream>>>(
        c->mode, c->n, c->d_acc, c->d_wg, c->d_p4, c->d_nrm, c->d_src,
        c->reg_mode == DWG_REG_CLAMP ? c->d_src16 : nullptr, c->d_dtheta, c->d_dn_blocks,
        c->d_state);
    return cudaGetLastError();
}

int select_blocks(int64_t n)
{
    return (int)std::min<int64_t>(std::max<int64_t>(ceil_div(n, 4 * kSelGridThreads), 1), 1024);
}

bool select_small(int64_t n) { return n <= kSelSmallMax; }

cudaError_t launch_select(Ctx *c, cudaGraphConditionalHandle cond, int use_cond)
{
    if (select_small(c->n)) {
        k_sel_small<<<1, kSelThreads, 0, c->stream>>>(
            c->d_dtheta, c->n, c->tol, c->conv_rule, c->d_state, c->d_dn_blocks, c->d_tr_iso,
            c->d_tr_stat, c->d_tr_dn, c->d_tr_faces, cond, use_cond);
        return cudaGetLastError();
    }
    const int nb = select_blocks(c->n);
    for (int level = 0; level < 3; ++level) {
        k_sel_hist<<<nb, kSelGridThreads, 0, c->stream>>>(c->d_dtheta, c->n, level, c->d_sel,
                                                          c->d_sel_hist, c->d_state);
        k_sel_find<<<1, kSelThreads, 0, c->stream>>>(c->n, level, c->d_sel, c->d_sel_hist,
                                                     c->d_state);
    }
    k_sel_sum<<<nb, kSelGridThreads, 0, c->stream>>>(c->d_dtheta, c->n, c->d_sel, c->d_sel_part,
                                                     c->d_state);
    k_sel_final<<<1, kSelThreads, 0, c->stream>>>(
        c->n, c->tol, c->conv_rule, c->d_sel, c->d_sel_part, nb, c->d_state, c->d_dn_blocks,
        (int)ceil_div(c->n, 256), c->d_tr_iso, c->d_tr_stat, c->d_tr_dn, c->d_tr_faces, cond,
        use_cond);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// batched iteration phases: every cloud of a batch in one launch (each
// cloud's blocks as in its own launch, so its results are the same bits)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_iso_b(const CloudIter *__restrict__ cl)
{
    const CloudIter &c = cl[blockIdx.x];
    iso_body(c.wsum_blocks, c.wsum_nb, c.n, c.st);
}

__global__ void __launch_bounds__(256)
    k_mc_faces_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    mc_faces_body(c.leaf_corners, c.leaves, c.nleaves, c.corner_pos, c.wc, c.codes, c.n, c.st,
                  c.faces, c.max_faces, c.err, (int64_t)blockIdx.x - off[ci]);
}

// a batch has k = 10; clouds without candidate lists search the tree
__global__ void __launch_bounds__(32 * kScanWarps, 6)
    k_knn_lists_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    knn_lists_body(c.faces, c.st, c.max_faces, c.T, c.cell_off, c.cell_idx, c.acc_scale, c.acc,
                   c.far_q, (int64_t)blockIdx.x - off[ci]);
}

__global__ void __launch_bounds__(32 * kFarWarps)
    k_knn_far_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    knn_far_body(c.faces, c.st, c.T, c.far_q, c.acc_scale, c.acc, c.defer, c.knn_budget, c.err,
                 (int64_t)blockIdx.x - off[ci], (int64_t)off[ci + 1] - off[ci]);
}

template <int KMAX, bool FIXED>
__global__ void __launch_bounds__(128)
    k_knn_scatter_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    knn_scatter_body<KMAX, FIXED>(c.faces, c.st, c.max_faces, c.T, c.k, c.cell_off, c.cell_idx,
                                  c.acc_scale, c.acc, c.defer, c.knn_budget, true, c.err,
                                  (int64_t)blockIdx.x - off[ci]);
}

__global__ void __launch_bounds__(defer_threads<10>())
    k_knn_deferred_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    knn_deferred_body<10, true>(c.faces, c.st, c.defer, c.T, c.k, c.acc_scale, c.acc,
                                (int64_t)blockIdx.x - off[ci], (int64_t)(off[ci + 1] - off[ci]));
}

__global__ void __launch_bounds__(256)
    k_normal_update_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    normal_update_body(c.mode, c.n, c.acc, c.wg, c.p4, c.nrm, c.src_rw, nullptr, c.dtheta,
                       c.dn_blocks, c.st, (int64_t)blockIdx.x - off[ci]);
}

__global__ void __launch_bounds__(kSelGridThreads)
    k_sel_hist_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl, int level)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    sel_hist_body(c.dtheta, c.n, level, c.sel, c.sel_hist, c.st, (int64_t)blockIdx.x - off[ci],
                  (int64_t)off[ci + 1] - off[ci]);
}

// small clouds (select_small): the whole selection in one block
__global__ void __launch_bounds__(kSelThreads)
    k_sel_small_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const CloudIter &c = cl[seg_cloud(off, ncl)];
    sel_small_body(c.dtheta, c.n, c.tol, c.conv_rule, c.st, c.dn_blocks, c.tr_iso, c.tr_stat,
                   c.tr_dn, c.tr_faces, 0, 0);
}

__global__ void __launch_bounds__(kSelThreads)
    k_sel_find_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl, int level)
{
    const CloudIter &c = cl[seg_cloud(off, ncl)];
    sel_find_body(c.n, level, c.sel, c.sel_hist, c.st);
}

__global__ void __launch_bounds__(kSelGridThreads)
    k_sel_sum_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const int ci = seg_cloud(off, ncl);
    const CloudIter &c = cl[ci];
    sel_sum_body(c.dtheta, c.n, c.sel, c.sel_part, c.st, (int64_t)blockIdx.x - off[ci],
                 (int64_t)off[ci + 1] - off[ci]);
}

__global__ void __launch_bounds__(kSelThreads)
    k_sel_final_b(const CloudIter *__restrict__ cl, const int *__restrict__ off, int ncl)
{
    const CloudIter &c = cl[seg_cloud(off, ncl)];
    sel_final_body(c.n, c.tol, c.conv_rule, c.sel, c.sel_part, c.sel_nb, c.st, c.dn_blocks,
                   (int)((c.n + 255) / 256), c.tr_iso, c.tr_stat, c.tr_dn, c.tr_faces, 0, 0);
}

cudaError_t launch_iter_batch(int phase, const CloudIter *cl, const int *off, int ncl,
                              int blocks, int arg, cudaStream_t s)
{
    if (blocks <= 0) return cudaSuccess;
    const unsigned g = (unsigned)blocks;
    switch (phase) {
    case kPhIso: k_iso_b<<<(unsigned)ncl, 256, 0, s>>>(cl); break;
    case kPhMcFaces: k_mc_faces_b<<<g, 256, 0, s>>>(cl, off, ncl); break;
    case kPhKnn: k_knn_scatter_b<10, true><<<g, 128, kAggSmem, s>>>(cl, off, ncl); break;
    case kPhKnnLists: k_knn_lists_b<<<g, 32 * kScanWarps, kTabSmem, s>>>(cl, off, ncl); break;
    case kPhKnnFar: k_knn_far_b<<<g, 32 * kFarWarps, 0, s>>>(cl, off, ncl); break;
    case kPhKnnDefer:
        k_knn_deferred_b<<<g, defer_threads<10>(), 0, s>>>(cl, off, ncl);
        break;
    case kPhUpdate: k_normal_update_b<<<g, 256, 0, s>>>(cl, off, ncl); break;
    case kPhSelSmall: k_sel_small_b<<<g, kSelThreads, 0, s>>>(cl, off, ncl); break;
    case kPhSelHist: k_sel_hist_b<<<g, kSelGridThreads, 0, s>>>(cl, off, ncl, arg); break;
    case kPhSelFind: k_sel_find_b<<<g, kSelThreads, 0, s>>>(cl, off, ncl, arg); break;
    case kPhSelSum: k_sel_sum_b<<<g, kSelGridThreads, 0, s>>>(cl, off, ncl); break;
    case kPhSelFinal: k_sel_final_b<<<g, kSelThreads, 0, s>>>(cl, off, ncl); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dwg
