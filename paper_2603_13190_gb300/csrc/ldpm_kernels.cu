// ldpm_kernels.cu -- sm_103a kernels of the LDPM explicit central-difference step.
//
// One step (paper Sec. 3, central difference with lumped mass) is two launches.  Between steps the
// state is kept drifted: q_{n+1} and v_{n+1/2} (and f_n); kick_kernel / unkick_kernel convert from /
// to the whole-step state q_n, v_n at the API boundary.
//   facet_kernel / facet_warp_kernel / facet_edge_kernel
//                  per facet: rigid-body jump and strain (Sec. 2, Eq. (1)), per-tetrahedron
//                  volumetric strain (App. A.2 e_V), the Appendix A law, force A P t; then per
//                  tetrahedron vertex the fixed-order sum of its 6 facets' forces and moments
//                  (the tetrahedron's share of Eq. (2a)-(2b)).  The warp variant (one 8-tetrahedron
//                  tile per warp) runs the FP32 pass, the edge variant (5 tetrahedra per warp, an edge per
//                  lane) the FP64 step, the block variant the other FP64 passes and larger tiles;
//   gather_kernel  per particle: fixed-order sum of its (tetrahedron, vertex) shares, then the second
//                  half kick of this step, the energy increments, and the first half kick and drift
//                  of the next step.
// No tensor cores (no dense contraction), no float atomics.  The passes are bound by memory latency
// and instruction issue (the FP64 ones by the FP64 pipe) well before HBM bandwidth.
//
// Times of "n steps of .. facets" in the comments of these files are pairs: the same calls before and after
// that one change, in turn in one process.  The remaining code and the calls around the steps (models in
// flight, state read-outs) differ from comment to comment, so the two numbers of a pair compare with each
// other only.  Times marked ncu are single launches with cold caches.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "ldpm_device.cuh"
#include "ldpm_internal.h"

namespace ldpm {
namespace {

// ------------------------------------------------------------------------------------------------
// Facet pass.  A block owns TETS consecutive tetrahedra (12 * TETS facets, one thread each).
//   phase A  4 threads per tetrahedron gather the vertex records (mixed mode: the 96-byte FP32
//            mirror, two-float differences; FP64 mode: the 128-byte FP64 record) and write the
//            differences to vertex 0 of the tetrahedron to shared memory, then the tetrahedron's
//            volumetric strain;
//   phase B  one thread per facet: kinematics, law, force, and its contributions to its two
//            vertices (force and moment about each);
//   phase C  12 threads per tetrahedron: thread s sums components 2(s%3), 2(s%3)+1 of vertex s/3
//            over the vertex's 6 facets in a fixed order (its 3 edges ascending, each edge's two
//            facets in slot order).
// Shared-memory rows are 16-byte aligned and accessed with 128/64-bit vectors (the pass is bound by
// L1/shared-memory wavefronts before HBM).  The facet's geometry and history are loaded into
// registers before phase A so their HBM latency overlaps the gathers.
// ------------------------------------------------------------------------------------------------
constexpr int kRow = 16;  // vertex row: dx(3) du(3) dv(3) theta(3) omega(3) pad
constexpr int kCon = 12;  // facet row: contribution to vertex a (6), to vertex b (6)
// Row strides in elements: with 16-byte accesses, 8 consecutive rows must start in distinct 4-bank
// groups (stride = 4 mod 8 banks for floats is 20 or 12 words; doubles use 36 and 28 words).
template <class R>
struct Stride {
    static constexpr int row = sizeof(R) == 4 ? 20 : 18;
    static constexpr int con = sizeof(R) == 4 ? 12 : 14;
};

// Loads of data that the persistent step kernel writes during its own launch (particle records,
// history, vertex shares, the step counter).  With PERSIST they are explicit weak global loads
// (ld.global.ca): never the read-only non-coherent path a compiler may pick for const __restrict__
// pointers, which is valid only for data that no thread writes during the launch.  Values written
// by other blocks become visible through the grid barrier's fences.
template <bool PERSIST, class T>
__device__ __forceinline__ T ld_live(const T *p)
{
    if constexpr (PERSIST)
        return __ldca(p);
    else
        return *p;
}
template <bool PERSIST>
__device__ __forceinline__ double4a ld_live(const double4a *p)
{
    if constexpr (PERSIST) {
        const double2 a = __ldca(reinterpret_cast<const double2 *>(p));
        const double2 b = __ldca(reinterpret_cast<const double2 *>(p) + 1);
        return double4a{a.x, a.y, b.x, b.y};
    } else {
        return *p;
    }
}

// Staging of one tetrahedron vertex (lane4 = 4 * tetrahedron + vertex within the tile; all 32 lanes
// of the warp take part, the shuffles stay within each tetrahedron's 4 lanes): the particle record,
// differences to the tetrahedron's vertex 0 into shared row sv[lane4], and e_V of the tetrahedron.
template <class R, int MODE, bool PERSIST = false>
__device__ __forceinline__ void stage_vertex(const DeviceModel &m, const void *__restrict__ vsrc, int64_t tet0,
                                             int lane4, R (*sv)[Stride<R>::row], R *seV, int *sok)
{
    constexpr int E = 16 / (int)sizeof(R);
    const LawConst<R> *__restrict__ lawc = static_cast<const LawConst<R> *>(m.law);
    (void)lawc;
    const int jt = lane4 >> 2, vi = lane4 & 3;
    const int64_t tt = tet0 + jt;
    int p = -1;
    if (tt < m.T) p = reinterpret_cast<const int *>(m.tet)[4 * tt + vi];
    const int base = (threadIdx.x & 31) & ~3;
    R o[kRow];
    if constexpr (sizeof(R) == 4) {
        // mirror: x_hi 0..2, x_lo 3..5, u_hi 6..8, u_lo 9..11, theta 12..14, v 15..17, omega 18..20.
        // (a_hi - b_hi) + (a_lo - b_lo) carries FP32 relative accuracy of the difference itself.
        const float *src = static_cast<const float *>(vsrc);
        float rec[24];
        if (p >= 0) {
            const float4 *r4 = reinterpret_cast<const float4 *>(src + kMirror * (int64_t)p);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const float4 w = ld_live<PERSIST>(r4 + k);
                rec[4 * k] = w.x;
                rec[4 * k + 1] = w.y;
                rec[4 * k + 2] = w.z;
                rec[4 * k + 3] = w.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 24; ++k) rec[k] = 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float x0h = __shfl_sync(0xffffffffu, rec[k], base);
            const float x0l = __shfl_sync(0xffffffffu, rec[3 + k], base);
            const float u0h = __shfl_sync(0xffffffffu, rec[6 + k], base);
            const float u0l = __shfl_sync(0xffffffffu, rec[9 + k], base);
            const float v0 = __shfl_sync(0xffffffffu, rec[15 + k], base);
            o[k] = (rec[k] - x0h) + (rec[3 + k] - x0l);
            o[3 + k] = (rec[6 + k] - u0h) + (rec[9 + k] - u0l);
            o[6 + k] = rec[15 + k] - v0;
            o[9 + k] = rec[12 + k];
            o[12 + k] = rec[18 + k];
        }
    } else {
        // FP64 record: x 0..2, u 3..5, theta 6..8, v 9..11, omega 12..14
        const double *src = static_cast<const double *>(vsrc);
        double rec[16];
        if (p >= 0) {
            const double2 *r2 = reinterpret_cast<const double2 *>(src + 16 * (int64_t)p);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const double2 w = ld_live<PERSIST>(r2 + k);
                rec[2 * k] = w.x;
                rec[2 * k + 1] = w.y;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) rec[k] = 0.0;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double x0 = __shfl_sync(0xffffffffu, rec[k], base);
            const double u0 = __shfl_sync(0xffffffffu, rec[3 + k], base);
            const double v0 = __shfl_sync(0xffffffffu, rec[9 + k], base);
            o[k] = rec[k] - x0;
            o[3 + k] = rec[3 + k] - u0;
            o[6 + k] = rec[9 + k] - v0;
            o[9 + k] = rec[6 + k];
            o[12 + k] = rec[12 + k];
        }
    }
    if (MODE == FACET_METRIC) {  // whole-step state: u_n = u_{n+1} - dt v_{n+1/2}, same for theta
        const R dtm = lawc[m.tile_spec ? m.tile_spec[tet0 / 32] : 0].dt;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[3 + k] -= dtm * o[6 + k];
            o[9 + k] -= dtm * o[12 + k];
        }
    }
    o[15] = R(0);
#pragma unroll
    for (int k = 0; k < kRow; k += E) VecT<R>::put(&sv[lane4][k], &o[k]);
    // e_V = (1/3) div u of the linear tetrahedron.  With D = [dx1 dx2 dx3], grad N_i (i = 1..3)
    // are the rows of D^-1 = [dx2 x dx3; dx3 x dx1; dx1 x dx2] / det D, and vertex 0 carries no
    // displacement difference.  Lane i >= 1 forms its own term du_i . (dx_i1 x dx_i2).
    const V3<R> dxs = {o[0], o[1], o[2]};
    const V3<R> dus = {o[3], o[4], o[5]};
    const int i1 = vi == 3 ? 1 : vi + 1;
    const int i2 = i1 == 3 ? 1 : i1 + 1;
    V3<R> a1, a2;
    a1.x = __shfl_sync(0xffffffffu, dxs.x, base + i1);
    a1.y = __shfl_sync(0xffffffffu, dxs.y, base + i1);
    a1.z = __shfl_sync(0xffffffffu, dxs.z, base + i1);
    a2.x = __shfl_sync(0xffffffffu, dxs.x, base + i2);
    a2.y = __shfl_sync(0xffffffffu, dxs.y, base + i2);
    a2.z = __shfl_sync(0xffffffffu, dxs.z, base + i2);
    const V3<R> cr = cross(a1, a2);
    R term = vi == 0 ? R(0) : dot(dus, cr);
    R det = vi == 0 ? R(0) : dot(dxs, cr);
    term += __shfl_xor_sync(0xffffffffu, term, 1);
    term += __shfl_xor_sync(0xffffffffu, term, 2);
    det = __shfl_sync(0xffffffffu, det, base + 1);
    if (vi == 0) {
        seV[jt] = (p >= 0 && det != R(0)) ? term / (R(3) * det) : R(0);
        sok[jt] = p >= 0;
    }
}

// One facet (tetrahedron j of the tile, slot 0..11, global facet f): kinematics, law, history, force,
// and its contributions to its two vertices in cs[12] (zeros when the facet is not live).
// S1: one specimen in mixed mode, law constants taken from m.law1 (the kernel parameters) instead of
// the global array; see facet_warp_kernel.
// ra, rb: the staged rows of the facet's vertices a and b; eV: e_V of its tetrahedron.
template <class R, int MODE, bool PF, bool S1 = false, bool STREAM = false>
__device__ __forceinline__ void facet_one(const DeviceModel &m, int64_t tet0, int64_t f, bool live, const R4<R> &g,
                                          const R4<R> &h, const R4<R> &pp, const R *ra, const R *rb, R eV, R cs[12],
                                          const LawConst<R> *lbatch = nullptr)
{
    using T4 = R4<R>;
    constexpr int E = 16 / (int)sizeof(R);
    T4 *__restrict__ hout = static_cast<T4 *>(m.hist_out ? m.hist_out : m.hist);  // the new history
    T4 *__restrict__ fout = static_cast<T4 *>(m.fout);
    const LawConst<R> *__restrict__ lawc = static_cast<const LawConst<R> *>(m.law);
    (void)pp;
    if (!live) {
#pragma unroll
    for (int k = 0; k < 12; ++k) cs[k] = R(0);
    } else {
    R A[kRow], B[kRow];
#pragma unroll
    for (int k = 0; k < kRow; k += E) {
        VecT<R>::get(&A[k], ra + k);
        VecT<R>::get(&B[k], rb + k);
    }
    const V3<R> d = {B[0] - A[0], B[1] - A[1], B[2] - A[2]};
    const R inv_l = rsqrt_(dot(d, d));
    const R l = dot(d, d) * inv_l;
    const V3<R> n = inv_l * d;
    V3<R> mt, lt;
    tangent_frame(n, mt, lt);
    const V3<R> ca = {g.x, g.y, g.z};
    const V3<R> cb = ca - d;
    R tN, tM, tL, emax;
    const LawConst<R> *lsrc;
    if (lbatch) {  // the batch kernel's parameters
        lsrc = lbatch;
    } else if constexpr (S1 && sizeof(R) == 4) {
        lsrc = reinterpret_cast<const LawConst<R> *>(&m.law1);
    } else {
        const int sp = m.tile_spec ? m.tile_spec[tet0 / 32] : 0;  // specimens are padded to 32 tetrahedra
        lsrc = lawc + sp;
    }
    LawConst<R> cpf;
    if constexpr (PF) cpf = facet_params(*lsrc, pp.x, pp.y, pp.z);
    const LawConst<R> &c = PF ? cpf : *lsrc;
    if (MODE == FACET_FROM_HIST) {
        tN = h.x;
        tM = h.y;
        tL = h.z;
    } else {
        const V3<R> thA = {A[9], A[10], A[11]}, thB = {B[9], B[10], B[11]};
        const V3<R> du = {B[3] - A[3], B[4] - A[4], B[5] - A[5]};
        const V3<R> jump = du + cross(thB, cb) - cross(thA, ca);
        const V3<R> e3 = {dot(n, jump) * inv_l, dot(mt, jump) * inv_l, dot(lt, jump) * inv_l};
        if (MODE == FACET_ELASTIC) {
            tN = c.E0 * e3.x;
            tM = c.alpha * c.E0 * e3.y;
            tL = c.alpha * c.E0 * e3.z;
        } else if (MODE == FACET_METRIC) {
            // crack opening from the inelastic part of the jump: w_N = l <e_N - t_N / E0>,
            // w_T = l (e_T - t_T / (alpha E0)) (u here is already u_n)
            R wn = e3.x - h.x / c.E0;
            wn = wn > R(0) ? wn : R(0);
            const R aE = c.alpha * c.E0;
            const R wm = e3.y - h.y / aE, wl = e3.z - h.z / aE;
            T4 o4;
            o4.x = l * sqrt(wn * wn + wm * wm + wl * wl);
            o4.y = eV;
            o4.z = R(0);
            o4.w = R(0);
            fout[f] = o4;
            tN = tM = tL = R(0);
        } else {
            const V3<R> omA = {A[12], A[13], A[14]}, omB = {B[12], B[13], B[14]};
            const V3<R> dv = {B[6] - A[6], B[7] - A[7], B[8] - A[8]};
            const V3<R> djump = dv + cross(omB, cb) - cross(omA, ca);
            const R sdt = c.dt * inv_l;
            const V3<R> de3 = {dot(n, djump) * sdt, dot(mt, djump) * sdt, dot(lt, djump) * sdt};
            tN = h.x;
            tM = h.y;
            tL = h.z;
            emax = h.w;
            facet_law(c, l, e3, de3, eV, tN, tM, tL, emax);
            T4 hn;
            hn.x = tN;
            hn.y = tM;
            hn.z = tL;
            hn.w = emax;
            if constexpr (STREAM)
                __stcs(hout + f, hn);
            else
                hout[f] = hn;
        }
    }
    const R Ar = g.w;
    const V3<R> F = {Ar * (tN * n.x + tM * mt.x + tL * lt.x), Ar * (tN * n.y + tM * mt.y + tL * lt.y),
                     Ar * (tN * n.z + tM * mt.z + tL * lt.z)};
    if (MODE == FACET_FROM_HIST) {  // per-facet force, kept only for ldpm_facet_forces
        T4 Fo;
        Fo.x = F.x;
        Fo.y = F.y;
        Fo.z = F.z;
        Fo.w = R(0);
        fout[f] = Fo;
    }
    // vertex a receives +F and the moment c_a x F about itself; vertex b -F and c_b x (-F)
    const V3<R> Ma = cross(ca, F);
    const V3<R> Mb = cross(cb, F);
    cs[0] = F.x;
    cs[1] = F.y;
    cs[2] = F.z;
    cs[3] = Ma.x;
    cs[4] = Ma.y;
    cs[5] = Ma.z;
    cs[6] = -F.x;
    cs[7] = -F.y;
    cs[8] = -F.z;
    cs[9] = -Mb.x;
    cs[10] = -Mb.y;
    cs[11] = -Mb.z;
    }
}

// Per tetrahedron vertex v = slot / 3, components 2 q, 2 q + 1 (q = slot % 3): the fixed-order sum over
// its 3 edges (ascending), each edge's two facets in slot order.
template <class R>
__device__ __forceinline__ void vertex_sum(const DeviceModel &m, int64_t tet0, int j, int slot,
                                           const R (*scon)[Stride<R>::con])
{
    using V2 = typename VecT<R>::v2;
    R *__restrict__ tvc = static_cast<R *>(m.tvc);
    const int v = slot / 3;
    const int q = slot - 3 * v;
    const int edges = (int)((0x542531430210ull >> (12 * v)) & 0xFFF);
    const int sides = (0xEC8 >> (3 * v)) & 0x7;  // v0: 000, v1: 001, v2: 011, v3: 111
    R s0 = R(0), s1 = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int e2 = (edges >> (4 * k)) & 0xF;
        const int col = (((sides >> k) & 1) ? 6 : 0) + 2 * q;
        const V2 w0 = *reinterpret_cast<const V2 *>(&scon[12 * j + 2 * e2][col]);
        const V2 w1 = *reinterpret_cast<const V2 *>(&scon[12 * j + 2 * e2 + 1][col]);
        s0 += w0.x;
        s1 += w0.y;
        s0 += w1.x;
        s1 += w1.y;
    }
    *reinterpret_cast<V2 *>(tvc + (tet0 + j) * 24 + 6 * v + 2 * q) = V2{s0, s1};
}

// One tile of TETS tetrahedra run by a block of 12 TETS threads (one facet each): phases A-C above.
// PF: the facet's own E0, alpha, sigma_t (m.pf) replace the material's in the law.
template <class R, int MODE, int TETS, bool PF>
__device__ __forceinline__ void facet_block_tile(const DeviceModel &m, const void *__restrict__ vsrc, int64_t tet0,
                                                 R (*sv)[Stride<R>::row], R (*scon)[Stride<R>::con], R *seV,
                                                 int *sok)
{
    using T4 = R4<R>;
    constexpr int E = 16 / (int)sizeof(R);  // elements per 16-byte shared-memory vector
    const T4 *__restrict__ geo = static_cast<const T4 *>(m.geo);
    const T4 *__restrict__ hist = static_cast<const T4 *>(m.hist);
    const int tid = threadIdx.x;

    // ---- prefetch this thread's facet data
    const int j = tid / 12;
    const int slot = tid - 12 * j;
    const int64_t f = tet0 * 12 + tid;
    const bool valid = tet0 + j < m.T;
    T4 g{}, h{}, pp{};
    if (valid) {
        g = geo[f];
        if (MODE != FACET_ELASTIC) h = hist[f];
        if (PF) pp = static_cast<const T4 *>(m.pf)[f];
    }

    // ---- phase A: vertex records -> shared memory, e_V per tetrahedron
    if (tid < 4 * TETS) stage_vertex<R, MODE>(m, vsrc, tet0, tid, sv, seV, sok);
    __syncthreads();

    // ---- phase B: one facet
    const bool live = valid && sok[j];
    R cs[12];
    const int e = slot >> 1, va = (0x211000 >> (4 * e)) & 0xF, vb = (0x332321 >> (4 * e)) & 0xF;
    facet_one<R, MODE, PF>(m, tet0, f, live, g, h, pp, sv[4 * j + va], sv[4 * j + vb], seV[j], cs);
#pragma unroll
    for (int k = 0; k < kCon; k += E) VecT<R>::put(&scon[tid][k], &cs[k]);
    __syncthreads();

    // ---- phase C
    if (live && MODE != FACET_METRIC) vertex_sum<R>(m, tet0, j, slot, scon);
}

template <class R, int MODE, int TETS, bool PF>
__global__ void __launch_bounds__(12 * TETS) facet_kernel(DeviceModel m, const void *__restrict__ vsrc)
{
    __shared__ alignas(16) R sv[TETS * 4][Stride<R>::row];
    __shared__ alignas(16) R scon[12 * TETS][Stride<R>::con];
    __shared__ R seV[TETS];
    __shared__ int sok[TETS];
    const int64_t tet0 = (int64_t)blockIdx.x * TETS;
    if (MODE == FACET_STEP && blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
    facet_block_tile<R, MODE, TETS, PF>(m, vsrc, tet0, sv, scon, seV, sok);
}

// Warp-tile variant of facet_kernel: every warp owns a tile of 8 tetrahedra and runs phases A-C on it
// alone (lane = vertex in phase A, three facets per lane in phase B, three vertex sums per lane in
// phase C), synchronising only within the warp, so each warp's record gathers are in flight
// independently of the other warps.  Same arithmetic and summation order as facet_kernel<.., 8, ..>.
// The facets' contributions are stored vertex-major: plane s (0..5) holds, for every vertex of the
// tile, the contribution of the s-th facet in that vertex's fixed summation order (its 3 edges
// ascending, each edge's two facets in slot order), 6 values per vertex.  The sums of a tile's 192
// share values then read each plane in 16-byte vectors, contiguous for the lanes and free of bank
// conflicts.  Planes are kPlane words apart: 192 plus 20, so that vectors stay aligned and the facets'
// stores into different planes fall on different banks (72 wavefronts per tile, as few as any stride).
// With one specimen (S1) the law constants are read from the kernel's own parameters (m is a
// __grid_constant__, so taking its address makes no copy): there they are operands of the
// instructions that use them, where the global array costs a load per use and facet (measured on
// GB300 in the loaded state of 1.82M facets: 43.1 us against 45.2 us).
constexpr int kTileTets = 8;
constexpr int kPlane = 6 * 4 * kTileTets + 20;
// Where facet fi (0..95) of a tile finds its rows and its places in the planes, in elements.  Edge e = slot
// / 2 joins local vertices va < vb; it is the ka-th edge of va and the kb-th of vb (ascending), so the
// facet is entry 2 ka + slot % 2 of va's order, 2 kb + slot % 2 of vb's.  The five numbers come from a
// table (one 8-byte load from L1 where computing them took about 25 integer instructions per facet: 20
// steps of 2.0M facets 1081 -> 1051 us, same results bit for bit).
struct FacetSlot {
    int tet, row_a, row_b, pl_a, pl_b;
};
struct SlotTable {
    uint2 v[12 * kTileTets];
    constexpr SlotTable() : v{}
    {
        for (int fi = 0; fi < 12 * kTileTets; ++fi) {
            const int j = fi / 12, slot = fi - 12 * j, e = slot >> 1, sw = slot & 1;
            const int va = (0x211000 >> (4 * e)) & 0xF, vb = (0x332321 >> (4 * e)) & 0xF;
            const int ka = (0x221210 >> (4 * e)) & 0xF, kb = (0x211000 >> (4 * e)) & 0xF;
            const unsigned pa = (2 * ka + sw) * kPlane + 6 * (4 * j + va), pb = (2 * kb + sw) * kPlane + 6 * (4 * j + vb);
            v[fi].x = pa | (pb << 12) | ((unsigned)j << 24);
            v[fi].y = (unsigned)(4 * j + va) | ((unsigned)(4 * j + vb) << 8);
        }
    }
};
__device__ const SlotTable kSlotOf{};
template <class R>
__device__ __forceinline__ FacetSlot facet_slot(int fi)
{
    const uint2 w = __ldg(&kSlotOf.v[fi]);
    return {(int)(w.x >> 24), (int)(w.y & 0xffu) * Stride<R>::row, (int)(w.y >> 8) * Stride<R>::row,
            (int)(w.x & 0xfffu), (int)((w.x >> 12) & 0xfffu)};
}
// One 8-tetrahedron tile of the facet pass, run by one warp on its own shared rows: phases A-C below.
// PERSIST: called from the persistent step kernel (live data through ld_live).
template <class R, int MODE, bool PF, bool S1, bool PERSIST, bool STREAM = false>
__device__ __forceinline__ void facet_tile(const DeviceModel &m, const void *__restrict__ vsrc, int64_t tet0,
                                           int lane, R (*sv)[Stride<R>::row], R *spl, R *seV, int *sok,
                                           const LawConst<R> *lbatch = nullptr)
{
    using T4 = R4<R>;
    using V2 = typename VecT<R>::v2;
    const T4 *__restrict__ geo = static_cast<const T4 *>(m.geo);
    const T4 *hist = static_cast<const T4 *>(m.hist);
    // the tile is whole: T is a multiple of 8.  The lane's three facets, prefetched
    const int32_t f0 = (int32_t)tet0 * 12 + lane;  // 12 T < 2^31
    T4 g[3] = {}, h[3] = {}, pp[3] = {};
    FacetSlot fs[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        fs[i] = facet_slot<R>(lane + 32 * i);
        if constexpr (STREAM) {
            g[i] = __ldcs(geo + f0 + 32 * i);
            h[i] = __ldcs(hist + f0 + 32 * i);
        } else {
            g[i] = geo[f0 + 32 * i];
            if (MODE != FACET_ELASTIC) h[i] = ld_live<PERSIST>(hist + f0 + 32 * i);
        }
        if (PF) pp[i] = static_cast<const T4 *>(m.pf)[f0 + 32 * i];
    }
    // ---- phase A
    stage_vertex<R, MODE, PERSIST>(m, vsrc, tet0, lane, sv, seV, sok);
    __syncwarp();
    // ---- phase B
    const R *rows = &sv[0][0];
    // bit j: tetrahedron j is not padding
    const unsigned okm = __ballot_sync(0xffffffffu, lane < kTileTets && sok[lane & (kTileTets - 1)] != 0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int j = fs[i].tet;
        R cs[12];
        facet_one<R, MODE, PF, S1, STREAM>(m, tet0, f0 + 32 * i, (okm >> j) & 1u, g[i], h[i], pp[i], rows + fs[i].row_a,
                                   rows + fs[i].row_b, seV[j], cs, lbatch);
        if (MODE != FACET_METRIC) {
            R *da = spl + fs[i].pl_a, *db = spl + fs[i].pl_b;
#pragma unroll
            for (int c = 0; c < 6; c += 2) {
                *reinterpret_cast<V2 *>(da + c) = V2{cs[c], cs[c + 1]};
                *reinterpret_cast<V2 *>(db + c) = V2{cs[6 + c], cs[6 + c + 1]};
            }
        }
    }
    __syncwarp();
    // ---- phase C: the tile's 192 share values, four per lane and round, summed over the 6 planes (10
    // steps of 11.4M facets 2537 -> 2500 us against three rounds of two values)
    if (MODE != FACET_METRIC) {
        using V4 = R4<R>;
        V4 *__restrict__ tvc = reinterpret_cast<V4 *>(static_cast<R *>(m.tvc)) + (int32_t)tet0 * 6 + lane;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int t = lane + 32 * i;
            if ((i == 0 || lane < 16) && ((okm >> ((t * 43) >> 8)) & 1u)) {  // t / 6
                const V4 *src = reinterpret_cast<const V4 *>(spl) + t;
                V4 s = src[0];
                s.x = R(0) + s.x;
                s.y = R(0) + s.y;
                s.z = R(0) + s.z;
                s.w = R(0) + s.w;
#pragma unroll
                for (int sp = 1; sp < 6; ++sp) {
                    const V4 x = src[sp * (kPlane / 4)];
                    s.x += x.x;
                    s.y += x.y;
                    s.z += x.z;
                    s.w += x.w;
                }
                tvc[32 * i] = s;
            }
        }
    }
    __syncwarp();  // the warp's shared rows may be reused for another tile
}

// Mixed mode: capped at 80 registers (12 blocks of 2 warps per SM); without the cap the multi-specimen
// instantiation took 93 registers and ran 8 % slower on the 97.7M-facet batch (GB300, side by side).
template <class R, int MODE, int WPB, bool PF, bool S1, bool STREAM = false>
__global__ void __launch_bounds__(32 * WPB, sizeof(R) == 4 ? 12 : 1)
    facet_warp_kernel(const __grid_constant__ DeviceModel m, const void *__restrict__ vsrc)
{
    constexpr int TETS = kTileTets;
    __shared__ alignas(16) R sv_[WPB][TETS * 4][Stride<R>::row];
    __shared__ alignas(16) R spl_[WPB][6 * kPlane];
    __shared__ R seV_[WPB][TETS];
    __shared__ int sok_[WPB][TETS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tet0 = ((int64_t)blockIdx.x * WPB + w) * TETS;
    if (MODE == FACET_STEP && blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
    if (tet0 >= m.T) return;  // whole warp (T is a multiple of the tile)
    facet_tile<R, MODE, PF, S1, false, STREAM>(m, vsrc, tet0, lane, sv_[w], spl_[w], seV_[w], sok_[w]);
}

// The same for a batch of specimens, their law constants in the kernel parameters: a block of WPB
// 8-tetrahedron tiles (16 tetrahedra) lies within one specimen, found from the block index alone by
// a search over the specimens' first tetrahedra (all in the parameters), so the constants are read
// at a block-uniform index.
template <int MODE, int WPB, bool PF>
__global__ void __launch_bounds__(32 * WPB, 12)
    facet_warp_batch_kernel(const __grid_constant__ DeviceModel m, const void *__restrict__ vsrc,
                            const __grid_constant__ BatchLaw bl)
{
    static_assert(WPB * kTileTets <= 32 && 32 % (WPB * kTileTets) == 0, "a block within one 32-tetrahedron unit");
    constexpr int TETS = kTileTets;
    __shared__ alignas(16) float sv_[WPB][TETS * 4][Stride<float>::row];
    __shared__ alignas(16) float spl_[WPB][6 * kPlane];
    __shared__ float seV_[WPB][TETS];
    __shared__ int sok_[WPB][TETS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tet0 = ((int64_t)blockIdx.x * WPB + w) * TETS;
    const int32_t tb = (int32_t)blockIdx.x * (WPB * TETS);
    int lo = 0, hi = bl.n;  // bl.t0[lo] <= tb < bl.t0[hi]
#pragma unroll
    for (int it = 0; it < 7; ++it) {  // 2^7 > kParamSpecimens
        const int mid = (lo + hi) >> 1;
        if (hi - lo > 1) {
            if (bl.t0[mid] <= tb)
                lo = mid;
            else
                hi = mid;
        }
    }
    if (MODE == FACET_STEP && blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
    if (tet0 >= m.T) return;  // whole warp (T is a multiple of the tile)
    facet_tile<float, MODE, PF, false, false>(m, vsrc, tet0, lane, sv_[w], spl_[w], seV_[w], sok_[w], &bl.law[lo]);
}

// ------------------------------------------------------------------------------------------------
// Edge-tile facet pass of the FP64 step.  It is bound by the FP64 pipe (one warp instruction per ~64
// cycles and sub-partition), so it is built to need few FP64 instructions; integer, FP32 and
// shared-memory work is nearly free beside them.
//   - A warp owns 5 tetrahedra and a lane one edge with its two facets (30 of 32 lanes): with
//     d = x_b - x_a, [[u]] = (du - theta_b x d) + (theta_b - theta_a) x c, one cross product per edge
//     and one per facet (c: the facet's arm from a) instead of two per facet; the moments about b are
//     d x S - M_a with the two facets' S and M_a summed first.
//   - The frame, the lengths and grad e_V depend on the reference positions alone and come from memory
//     (m.frame, m.grad: 64 + 6 bytes per facet and step, 5 % of the pass at HBM rate).
//   - Comparisons and the law's filters run on the other pipes (compression_trial64, fracture_floor32).
//     The facets that may have reached a boundary are collected in shared memory, branch by branch, and
//     evaluated by full warps (a tenth of them spread over a warp's 60 facets would otherwise hold all
//     lanes twice).
// Phases: records to shared memory with cp.async; one edge per lane; contributions vertex-major in three
// planes (plane k: the k-th edge of each vertex), summed over the vertex's edges in ascending order.
// Against the block kernel (one facet per thread, frames rebuilt, the whole law evaluated everywhere), per
// launch on GB300 (ncu): 594 -> 225 us on 676k facets in tension past the peak, 540 -> 270 us on 1.15M
// facets in compression; the FP64 pipe is 86 % busy in both.
// ------------------------------------------------------------------------------------------------
constexpr int kERow = 18;       // doubles per staged vertex record (16, padded against bank conflicts)
constexpr int kEPlane = 122;    // doubles per contribution plane (20 vertices x 6 values, padded)
constexpr int kEItem = 7;       // doubles per collected facet
constexpr int kEWords = 12 * kEdgeTets * kEItem;  // doubles per warp; rows (360) and planes (366) lie in them
static_assert(4 * kEdgeTets * kERow <= kEWords && 3 * kEPlane <= kEWords, "rows and planes fit");
constexpr int kEdgeWarps = 2;   // warps (tiles) per block

// Tetrahedra [tet0, tet0 + 5) by one warp on its own shared words sw (a tile may straddle two specimens:
// the law constants are read per lane).
template <bool PF, bool PERSIST>
__device__ __forceinline__ void facet_edge_tile(const DeviceModel &m, const double *__restrict__ vsrc, int32_t tet0,
                                                int lane, double *sw)
{
    const int j = lane / 6, e = lane - 6 * j, jj = j < kEdgeTets ? j : 0;
    const int32_t tt = tet0 + j;
    const bool in = lane < 6 * kEdgeTets && tt < m.T;
    const double4a *__restrict__ geo = static_cast<const double4a *>(m.geo);
    const double4a *hist = static_cast<const double4a *>(m.hist);
    // ---- records to shared memory, this lane's facets to registers
    int vid = -1;
    if (lane < 4 * kEdgeTets && tet0 + (lane >> 2) < m.T)
        vid = __ldg(reinterpret_cast<const int *>(m.tet) + 4 * (int64_t)tet0 + lane);
#pragma unroll
    for (int i = 0; i < 5; ++i) {  // 16-byte pieces 1..7 of each record (piece 0 is position only)
        const int c = lane + 32 * i;
        const int v = c / 7, part = 1 + c - 7 * v;
        const int id = __shfl_sync(0xffffffffu, vid, v & 31);
        if (c < 28 * kEdgeTets)
            cp_async16<PERSIST>(sw + kERow * v + 2 * part, vsrc + (id >= 0 ? 16 * (int64_t)id + 2 * part : 0), id >= 0);
    }
    const bool live = __shfl_sync(0xffffffffu, vid, 4 * jj) >= 0 && in;
    const int64_t f = 12 * (int64_t)tt + 2 * e;
    double4a h[2] = {};
    V3<double> P0{}, P1{}, P2{}, d{}, gr{};
    double lA[2] = {}, ht = 0.0;
    if (live) {
        const double2 *fr = reinterpret_cast<const double2 *>(m.frame) + 8 * (6 * (int64_t)tt + e);
        const double2 a0 = __ldg(fr), a1 = __ldg(fr + 1), a2 = __ldg(fr + 2), a3 = __ldg(fr + 3), a4 = __ldg(fr + 4),
                      a5 = __ldg(fr + 5), a6 = __ldg(fr + 6), a7 = __ldg(fr + 7);
        P0 = {a0.x, a0.y, a1.x};
        P1 = {a1.y, a2.x, a2.y};
        P2 = {a3.x, a3.y, a4.x};
        d = {a4.y, a5.x, a5.y};
        lA[0] = a6.x;
        lA[1] = a6.y;
        ht = a7.y;
        if (e < 3) {
            const double *g3 = m.grad + 3 * (3 * (int64_t)tt + e);
            gr = {__ldg(g3), __ldg(g3 + 1), __ldg(g3 + 2)};
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) h[i] = ld_live<PERSIST>(hist + f + i);
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    // ---- one edge: local vertices va < vb
    const int va = (0x211000 >> (4 * e)) & 0xF, vb = (0x332321 >> (4 * e)) & 0xF;
    V3<double> wq, wv, dth, dom;
    double eV;
    {
        // record: x 0..2, u 3..5, theta 6..8, v 9..11, omega 12..14
        const double *A = sw + kERow * (4 * jj + va), *B = sw + kERow * (4 * jj + vb);
        const V3<double> du = {B[3] - A[3], B[4] - A[4], B[5] - A[5]};
        const V3<double> thB = {B[6], B[7], B[8]}, omB = {B[12], B[13], B[14]};
        dth = {thB.x - A[6], thB.y - A[7], thB.z - A[8]};
        dom = {omB.x - A[12], omB.y - A[13], omB.z - A[14]};
        wv = add_cross(V3<double>{B[9] - A[9], B[10] - A[10], B[11] - A[11]}, d, omB);
        wq = add_cross(du, d, thB);
        // e_V: the edges 0-1, 0-2, 0-3 hold its three terms
        const double term = fma(gr.x, du.x, fma(gr.y, du.y, gr.z * du.z));
        const int base = 6 * jj;
        const double t0 = __shfl_sync(0xffffffffu, term, base), t1 = __shfl_sync(0xffffffffu, term, base + 1),
                     t2 = __shfl_sync(0xffffffffu, term, base + 2);
        eV = t0 + t1 + t2;
    }
    __syncwarp();  // the rows are read: shared memory may be reused
    const LawConst<double> &c = static_cast<const LawConst<double> *>(m.law)[in && m.tile_spec ? m.tile_spec[tt / 32] : 0];
    V3<double> e3[2], t[2];  // strain; new traction (fracture: scalar effective traction in x until the end)
    double emax[2], inv_e[2], aT2[2];
    bool frac[2] = {false, false};
    bool need[2] = {false, false};
    auto par = [&](int i) -> FacetPar64 {
        if constexpr (PF) {
            const double4a pp = static_cast<const double4a *>(m.pf)[f + i];
            return {pp.x, pp.y, pp.w, pp.z};
        } else {
            return {c.E0, c.alpha, c.inv_alpha, c.sigma_t};
        }
    };
    if (live) {
        const double dt = c.dt;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const double4a g = geo[f + i];
            const V3<double> arm = {g.x, g.y, g.z};
            const FacetPar64 fp = par(i);
            const V3<double> J = add_cross(wq, dth, arm);
            const V3<double> es = {fma(P0.x, J.x, fma(P0.y, J.y, P0.z * J.z)), fma(P1.x, J.x, fma(P1.y, J.y, P1.z * J.z)),
                                   fma(P2.x, J.x, fma(P2.y, J.y, P2.z * J.z))};
            e3[i] = es;
            emax[i] = h[i].w;
            if (c.elastic) {
                const double aE = fp.alpha * fp.E0;
                t[i] = {fp.E0 * es.x, aE * es.y, aE * es.z};
                continue;
            }
            const V3<double> Jv = add_cross(wv, dom, arm);
            const V3<double> de = {dt * fma(P0.x, Jv.x, fma(P0.y, Jv.y, P0.z * Jv.z)),
                                   dt * fma(P1.x, Jv.x, fma(P1.y, Jv.y, P1.z * Jv.z)),
                                   dt * fma(P2.x, Jv.x, fma(P2.y, Jv.y, P2.z * Jv.z))};
            const double tN = h[i].x, tM = h[i].y, tL = h[i].z;
            if (order_bits(es.x) <= 0) {
                t[i] = {tN, tM, tL};
                need[i] = compression_trial64(c, fp, de, t[i]);
                continue;
            }
            // fracture (App. A.1), as facet_law; e = e^2 / e from the reciprocal root
            const double a2 = fp.alpha * fma(es.y, es.y, es.z * es.z);
            const double e2 = fma(es.x, es.x, a2);
            if (order_bits(e2) < order_bits(1e-300)) {  // e < c.tiny_strain = 1e-150: t = E e
                const double aE = fp.alpha * fp.E0, eff = sqrt(e2);
                t[i] = {fp.E0 * es.x, aE * es.y, aE * es.z};
                emax[i] = greater_than(emax[i], eff) ? emax[i] : eff;
                continue;
            }
            frac[i] = true;
            const double ie = rsqrt(e2), eff = e2 * ie;
            const double em = greater_than(emax[i], eff) ? emax[i] : eff;
            const V3<double> ep = es - de;
            const double e_old = sqrt(fma(ep.x, ep.x, fp.alpha * fma(ep.y, ep.y, ep.z * ep.z)));
            const double num = fma(de.x, es.x + ep.x, fp.alpha * fma(de.y, es.y + ep.y, de.z * (es.z + ep.z)));
            double d_eff = num / (eff + e_old);
            const double t_old = sqrt(fma(tN, tN, fma(tM, tM, tL * tL) * fp.inv_alpha));
            if (c.k_t > 0.0 && t_old <= 0.0 && d_eff > 0.0) {
                // reloading from zero traction: it stays zero up to e_tr = k_t (e_max - sigma_bt / E0)
                const double e_tr = c.k_t * (em - fracture_boundary64(c, fp, es.x, a2, ie, em, ht) / fp.E0);
                if (e_tr > e_old) d_eff = eff > e_tr ? eff - e_tr : 0.0;
            }
            double tr = fma(fp.E0, d_eff, t_old);
            tr = negative(tr) ? 0.0 : tr;
            need[i] = !fracture_inside32(c, fp, tr, es.x, a2, ie, em, ht);
            t[i].x = tr;
            emax[i] = em;
            inv_e[i] = ie;
            aT2[i] = a2;
        }
    }
    // ---- the facets that may have reached a boundary, collected per branch: item k goes to lane k % 32
    const int sp = m.tile_spec && in ? m.tile_spec[tt / 32] : 0;
#pragma unroll
    for (int br = 0; br < 2; ++br) {  // 0: fracture, 1: compression and friction
        const bool n0 = need[0] && frac[0] == (br == 0), n1 = need[1] && frac[1] == (br == 0);
        const unsigned b0 = __ballot_sync(0xffffffffu, n0), b1 = __ballot_sync(0xffffffffu, n1);
        const int items = __popc(b0) + __popc(b1);
        if (!items) continue;
        const unsigned below = (1u << lane) - 1u;
        double *w0 = sw + kEItem * __popc(b0 & below), *w1 = sw + kEItem * (__popc(b0) + __popc(b1 & below));
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (i == 0 ? n0 : n1) {
                double *w = i == 0 ? w0 : w1;
                w[0] = t[i].x;
                w[1] = e3[i].x;
                w[2] = br == 0 ? aT2[i] : t[i].y;
                w[3] = br == 0 ? inv_e[i] : t[i].z;
                w[4] = br == 0 ? emax[i] : eV;
                if (br == 0) w[5] = ht;
                w[6] = __longlong_as_double((f + i) | ((long long)sp << 40));
            }
        __syncwarp();
        for (int k = lane; k < items; k += 32) {
            double *w = sw + kEItem * k;
            const long long id = __double_as_longlong(w[6]);
            const LawConst<double> &ck = static_cast<const LawConst<double> *>(m.law)[id >> 40];
            FacetPar64 fp = {ck.E0, ck.alpha, ck.inv_alpha, ck.sigma_t};
            if constexpr (PF) {
                const double4a pp = static_cast<const double4a *>(m.pf)[id & 0xffffffffffll];
                fp = {pp.x, pp.y, pp.w, pp.z};
            }
            if (br == 0) {
                const double sb = fracture_boundary64(ck, fp, w[1], w[2], w[3], w[4], w[5]);
                if (greater_than(w[0], sb)) w[0] = sb;
            } else {
                V3<double> tr = {w[0], w[2], w[3]};
                compression_return64(ck, fp, w[1], w[4], tr);
                w[0] = tr.x;
                w[2] = tr.y;
                w[3] = tr.z;
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (i == 0 ? n0 : n1) {
                const double *w = i == 0 ? w0 : w1;
                t[i].x = w[0];
                if (br == 1) {
                    t[i].y = w[2];
                    t[i].z = w[3];
                }
            }
        __syncwarp();
    }
    if (live) {
        double4a *__restrict__ hout = static_cast<double4a *>(m.hist_out ? m.hist_out : m.hist);
        V3<double> S{}, MA{};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (frac[i]) {
                const double r = t[i].x * inv_e[i], ar = par(i).alpha * r;
                t[i] = {r * e3[i].x, ar * e3[i].y, ar * e3[i].z};
            }
            double4a hn;
            hn.x = t[i].x;
            hn.y = t[i].y;
            hn.z = t[i].z;
            hn.w = emax[i];
            hout[f + i] = hn;
            const double4a g = geo[f + i];
            const V3<double> a = lA[i] * t[i];
            const V3<double> F = {fma(a.x, P0.x, fma(a.y, P1.x, a.z * P2.x)), fma(a.x, P0.y, fma(a.y, P1.y, a.z * P2.y)),
                                  fma(a.x, P0.z, fma(a.y, P1.z, a.z * P2.z))};
            S = S + F;
            MA = add_cross(MA, V3<double>{g.x, g.y, g.z}, F);
        }
        // end a receives (S, MA), end b (-S, d x S - MA); e is the ka-th edge of va, the kb-th of vb
        const int ka = (0x221210 >> (4 * e)) & 0xF, kb = (0x211000 >> (4 * e)) & 0xF;
        const V3<double> MB = add_cross(V3<double>{-MA.x, -MA.y, -MA.z}, d, S);
        double2 *da = reinterpret_cast<double2 *>(sw + ka * kEPlane + 6 * (4 * j + va));
        double2 *db = reinterpret_cast<double2 *>(sw + kb * kEPlane + 6 * (4 * j + vb));
        da[0] = double2{S.x, S.y};
        da[1] = double2{S.z, MA.x};
        da[2] = double2{MA.y, MA.z};
        db[0] = double2{-S.x, -S.y};
        db[1] = double2{-S.z, MB.x};
        db[2] = double2{MB.y, MB.z};
    }
    const unsigned lv = __ballot_sync(0xffffffffu, live);
    __syncwarp();
    // ---- pair q of the tile's 120 share values over the vertex's three edges
    double2 *__restrict__ out = reinterpret_cast<double2 *>(static_cast<double *>(m.tvc) + 24 * (int64_t)tet0);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int q = lane + 30 * i;
        if (lane < 30 && ((lv >> (6 * (q / 12))) & 1u)) {
            const double2 *s2 = reinterpret_cast<const double2 *>(sw) + q;
            const double2 x = s2[0], y = s2[kEPlane / 2], z = s2[kEPlane];
            out[q] = double2{(x.x + y.x) + z.x, (x.y + y.y) + z.y};
        }
    }
    if (PERSIST) __syncwarp();  // the shared words are reused for the next tile
}

template <bool PF>
__global__ void __launch_bounds__(32 * kEdgeWarps)
    facet_edge_kernel(const __grid_constant__ DeviceModel m, const double *__restrict__ vsrc)
{
    __shared__ alignas(16) double sw[kEdgeWarps][kEWords];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tet0 = ((int64_t)blockIdx.x * kEdgeWarps + w) * kEdgeTets;
    if (blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
    if (tet0 >= m.T) return;  // the whole warp
    facet_edge_tile<PF, false>(m, vsrc, (int32_t)tet0, lane, sw[w]);
}

// m.frame and m.grad (see ldpm_internal.h) from the reference positions; one thread per edge.
__global__ void __launch_bounds__(128) frame_kernel(DeviceModel m)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 6 * (int64_t)m.T) return;
    const int64_t tt = k / 6;
    const int e = (int)(k - 6 * tt);
    double *fr = m.frame + 16 * k;
    const int *tv = reinterpret_cast<const int *>(m.tet) + 4 * tt;
    if (tv[0] < 0) {
        for (int q = 0; q < 16; ++q) fr[q] = 0.0;
        if (e < 3)
            for (int q = 0; q < 3; ++q) m.grad[3 * (3 * tt + e) + q] = 0.0;
        return;
    }
    V3<double> x[4];
    for (int v = 0; v < 4; ++v) {
        const double *p = m.pstate + 16 * (int64_t)tv[v];
        x[v] = {p[0], p[1], p[2]};
    }
    const int va = (0x211000 >> (4 * e)) & 0xF, vb = (0x332321 >> (4 * e)) & 0xF;
    const V3<double> d = x[vb] - x[va];
    const double l2 = dot(d, d), l = sqrt(l2), il = 1.0 / l;
    const V3<double> n = il * d;
    V3<double> mt, lt;
    tangent_frame(n, mt, lt);
    const double lim = static_cast<const LawConst<double> *>(m.law)[m.tile_spec ? m.tile_spec[tt / 32] : 0].l_t;
    const double4a *geo = static_cast<const double4a *>(m.geo) + 2 * k;
    const double rec[16] = {il * n.x, il * n.y, il * n.z, il * mt.x, il * mt.y, il * mt.z, il * lt.x, il * lt.y,
                            il * lt.z, d.x, d.y, d.z, l * geo[0].w, l * geo[1].w, l, 2.0 * l / (lim - l)};
    for (int q = 0; q < 16; ++q) fr[q] = rec[q];
    if (e < 3) {
        const V3<double> dx[3] = {x[1] - x[0], x[2] - x[0], x[3] - x[0]};
        const double det = dot(dx[0], cross(dx[1], dx[2]));
        const V3<double> g = cross(dx[(e + 1) % 3], dx[(e + 2) % 3]);
        const double s = det != 0.0 ? 1.0 / (3.0 * det) : 0.0;
        double *o = m.grad + 3 * (3 * tt + e);
        o[0] = s * g.x;
        o[1] = s * g.y;
        o[2] = s * g.z;
    }
}

// ------------------------------------------------------------------------------------------------
// Particle pass.  A group of LPP lanes owns one particle: it sums the particle's (tetrahedron,
// vertex) contributions in CSR order (Eq. (2a)-(2b)), reduces across the group by halving exchanges,
// after which six lanes of the group hold components 0..5 and update one DOF each.  With LPP = 8 a
// warp updates 4 particles per instruction.
// The particle's own records (mass, constraint, q, v, f_n) do not depend on the contributions and are
// loaded before the sum, so their latency overlaps the CSR gather.
// FP64 mode: everything is FP64.  Mixed mode: the shares are FP32 (each the sum of a tetrahedron's 6
// FP32 facet terms at one vertex); the particle sums of the shares are float-float (48 mantissa bits;
// components paired in packed FP32 instructions), converted to FP64 once; the velocity and
// displacement updates are FP64; the energy increments (trapezoid products with v_{n+1/2} and their
// 6-DOF sums) are float-float, scaled by dt/2 and added into the FP64 accumulators with one FP64 FMA
// each.  The GB300 FP64 pipe issues one warp instruction per ~64 cycles per sub-partition, so the
// compensated sums run on the FP32 pipe; FP32 <-> FP64 conversions are integer operations.
// ------------------------------------------------------------------------------------------------
// One group of LPP lanes, particle p (all 32 lanes of the warp take part in its shuffles).
template <class R, int MODE, int LPP, bool PERSIST, bool STREAM = false>
__device__ __forceinline__ void gather_group(const DeviceModel &m, int64_t p, int lane, double *__restrict__ out6)
{
    static_assert(LPP == 8 || LPP == 16 || LPP == 32, "lanes per particle");
    constexpr bool kMixed = sizeof(R) == 4;
    const int32_t *__restrict__ ent = static_cast<const int32_t *>(m.ent);
    const R *tvc = static_cast<const R *>(m.tvc);
    const int sub = lane & (LPP - 1);
    const bool valid = p < m.N;
    // after the group's reduction, lanes 0..5 (mixed: pair_halving_sum6) or 0, 1, 2, 4, 5, 6 (FP64:
    // halving_sum6) of the group hold the sums of DOFs 0..5; the other lanes mirror DOF 0 and store
    // nothing
    const int slot6 = sub >= 8 ? -1 : kMixed ? (sub < 6 ? sub : -1) : halving_slot6(sub);
    const bool act = valid && slot6 >= 0;
    const int d = slot6 >= 0 ? slot6 : 0;
    const int64_t pc_ = valid ? p : 0;
    int r0 = 0, r1 = 0;
    if (valid) {
        r0 = m.row[p];
        r1 = m.row[p + 1];
    }
    // ---- the particle's own records (step mode), issued ahead of the gather
    double *ps = m.pstate + 16 * pc_;
    double *pd = m.pdyn + 8 * pc_;
    const double *pc = m.pconst + 8 * pc_;
    const bool has_fext = m.f_ext != nullptr;
    double im = 0.0, vh = 0.0, q0 = 0.0, fa_old = 0.0, fe = 0.0;
    int mask = 0, sp = 0;
    if (MODE != GATHER_ASSEMBLE) {
        im = pc[d];
        mask = (int)(((uint64_t)__double_as_longlong(pc[6]) >> (8 * d)) & 0xffu);
        sp = (int)__double_as_longlong(pc[7]);
        vh = ps[9 + d];
        q0 = ps[3 + d];
        if (has_fext) fe = m.f_ext[6 * pc_ + d];
    }
    // Each CSR entry is one (tetrahedron, vertex) slot: 6 values, force (3) and moment about the
    // particle (3).  Lane `sub` sums entries sub, sub + LPP, sub + 2 LPP, ... of the particle's row in
    // that order: the first kSlotTab from the slot table (all of them in flight at once, addressed by
    // the particle index alone), the rest of a longer row through row/ent.
    constexpr int KT = (kSlotTab + LPP - 1) / LPP;  // table positions per lane
    const int32_t *__restrict__ tab = m.stab + (int64_t)pc_ * kSlotTab;
    auto slot_id = [&](int k) -> int {
        const int j = sub + LPP * k;
        return (valid && j < kSlotTab) ? __ldg(tab + j) : -1;
    };
    const int j_over = sub + LPP * ((kSlotTab - sub + LPP - 1) / LPP);  // this lane's first entry past the table
    double fa_new;
    ff fa_ff{};  // mixed: the same sum as a float-float
    if constexpr (kMixed) {
        // components (0, 1), (2, 3), (4, 5) as packed float-float pairs
        ff2 a[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c] = ff2{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
        {
            int id[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) id[k] = slot_id(k);
            // the shares in batches of KB entries in flight (all ids are loaded above): 48 registers,
            // 20 blocks of 64 threads per SM
            constexpr int KB = 2;
#pragma unroll
            for (int k0 = 0; k0 < KT; k0 += KB) {
                float2 w[KB][3];
#pragma unroll
                for (int k = k0; k < k0 + KB && k < KT; ++k)
                    if (id[k] >= 0) {
                        const float2 *src = reinterpret_cast<const float2 *>(tvc + 6 * (int64_t)id[k]);
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            w[k - k0][c] = STREAM ? __ldcs(src + c) : ld_live<PERSIST>(src + c);
                    }
#pragma unroll
                for (int k = k0; k < k0 + KB && k < KT; ++k)
                    if (id[k] >= 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) ff2_acc(a[c], w[k - k0][c]);
                    }
            }
        }
        for (int j = j_over; j < r1 - r0; j += LPP) {  // rows longer than the table
            const float2 *src = reinterpret_cast<const float2 *>(tvc + 6 * (int64_t)ent[r0 + j]);
#pragma unroll
            for (int c = 0; c < 3; ++c) ff2_acc(a[c], ld_live<PERSIST>(src + c));
        }
        // lanes beyond the first 8 of a group fold into them
#pragma unroll
        for (int off = LPP / 2; off >= 8; off >>= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) a[c] = ff2_add(a[c], ff2_shfl_xor(a[c], off));
        if (MODE != GATHER_ASSEMBLE) fa_old = pd[d];  // f_n: needed only by the energy increments
        fa_ff = ff_norm(pair_halving_sum6(a, lane));
        fa_new = ff_to_double(fa_ff);
    } else {
        double a[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) a[k] = 0.0;
        {
            int id[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) id[k] = slot_id(k);
            double2 w[KT][3];
#pragma unroll
            for (int k = 0; k < KT; ++k)
                if (id[k] >= 0) {
                    const double2 *src = reinterpret_cast<const double2 *>(tvc + 6 * (int64_t)id[k]);
                    w[k][0] = ld_live<PERSIST>(src);
                    w[k][1] = ld_live<PERSIST>(src + 1);
                    w[k][2] = ld_live<PERSIST>(src + 2);
                }
#pragma unroll
            for (int k = 0; k < KT; ++k)
                if (id[k] >= 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        a[2 * c] += w[k][c].x;
                        a[2 * c + 1] += w[k][c].y;
                    }
                }
        }
        for (int j = j_over; j < r1 - r0; j += LPP) {  // rows longer than the table
            const double2 *src = reinterpret_cast<const double2 *>(tvc + 6 * (int64_t)ent[r0 + j]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 w = ld_live<PERSIST>(src + c);
                a[2 * c] += w.x;
                a[2 * c + 1] += w.y;
            }
        }
#pragma unroll
        for (int off = LPP / 2; off >= 8; off >>= 1)
#pragma unroll
            for (int k = 0; k < 6; ++k) a[k] += __shfl_xor_sync(0xffffffffu, a[k], off);
        if (MODE != GATHER_ASSEMBLE) fa_old = pd[d];
        halving_sum6(a, lane);
        fa_new = a[0];
    }
    if (MODE == GATHER_ASSEMBLE) {
        if (act) out6[6 * p + d] = fa_new;
        return;
    }
    // ---- velocity-form central difference for DOF d (state on entry: q_{n+1}, v_{n+1/2}, f_n)
    const SpecDyn &S = m.spec[sp];
    const double dt = S.dt, hdt = S.half_dt;
    // energy terms need the external work only where a lane is constrained or loaded
    const bool need_we = __any_sync(0xffffffffu, act && (mask != 0 || has_fext));
    // prescribed velocity vb ramp(t): the constraint's accelerations at t_n and t_{n+1} are
    // vb (ramp(t +- dt/2) differences) / dt, so their sum telescopes to vb (r(t1+dt/2) - r(t0-dt/2)) / dt
    double g_bc = 0.0, v_bc = 0.0;
    if (mask > 1) {
        const int64_t n1 = ld_live<PERSIST>(reinterpret_cast<const long long *>(m.step));
        const double t1 = (double)n1 * dt;
        const double r_next = ramp(t1 + hdt, S.inv_ramp);
        g_bc = m.bc_vm[6 * pc_ + d] * (r_next - ramp(t1 - dt - hdt, S.inv_ramp)) * S.inv_dt;
        v_bc = m.bc_vel[6 * pc_ + d] * r_next;
    }
    double v_next, dWi_acc, dWe_acc;
    if (mask == 0) {
        const double fa = has_fext ? fe + fa_new : fa_new;
        if constexpr (kMixed) {
            v_next = fma(fa, dt * im, vh);  // v_{n+3/2} = v_{n+1/2} + dt a_{n+1}
        } else {
            const double dv = fa * (hdt * im);  // dt/2 a_{n+1}
            v_next = (vh + dv) + dv;
        }
    } else {
        v_next = mask == 1 ? 0.0 : v_bc;
    }
    // energy increments over [t_n, t_{n+1}] (trapezoid): dq = dt v_{n+1/2},
    //   dW_int = -(f_n + f_{n+1}) dq / 2 on every DOF, dW_ext = g dq / 2 with g the sum of the
    //   external forces (2 f_ext on loaded DOFs, the supports' reactions on constrained ones)
    if constexpr (kMixed) {
        // float-float products with v_{n+1/2}, summed over the six DOFs as one packed pair
        // (internal, external); the common factor dt/2 is applied in FP64 when accumulating
        const ff fsum = ff_add(ff_from_double(fa_old), fa_ff);
        const ff vhf = ff_from_double(vh);
        ff g = {0.0f, 0.0f};
        if (mask == 0) {
            if (has_fext) {
                const ff f1 = ff_from_double(fe);
                g = ff{2.0f * f1.hi, 2.0f * f1.lo};
            }
        } else {
            g = mask == 1 ? ff_neg(fsum) : ff_add(ff_from_double(g_bc), ff_neg(fsum));
        }
        const ff zero = {0.0f, 0.0f};
        ff2 e = ff2_pack(act ? ff_neg(ff_mul(fsum, vhf)) : zero, (need_we && act) ? ff_mul(g, vhf) : zero);
        // the six DOF contributions into every lane of the group (lanes 6, 7 hold zeros)
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) e = ff2_add(e, ff2_shfl_xor(e, off));
        dWi_acc = f2d_bits(e.hi.x) + f2d_bits(e.lo.x);
        dWe_acc = need_we ? f2d_bits(e.hi.y) + f2d_bits(e.lo.y) : 0.0;
    } else {
        double g_sum = 0.0;
        if (mask == 0) {
            if (has_fext) g_sum = 2.0 * fe;
        } else if (mask == 1) {
            g_sum = -(fa_old + fa_new);
        } else {
            g_sum = g_bc - (fa_old + fa_new);
        }
        const double hdq = hdt * vh;
        double dWi = act ? -(fa_old + fa_new) * hdq : 0.0;
        double dWe = (need_we && act) ? g_sum * hdq : 0.0;
        // sum the six DOF contributions into lane 0 of the group (lanes 3, 7 hold zeros)
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) dWi += __shfl_xor_sync(0xffffffffu, dWi, off);
        if (need_we) {
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) dWe += __shfl_xor_sync(0xffffffffu, dWe, off);
        }
        dWi_acc = dWi;
        dWe_acc = dWe;
    }
    // store the drifted state of the next step: v_{n+3/2} and q_{n+2} = q_{n+1} + dt v_{n+3/2}
    const double q = q0 + dt * v_next;
    if (act) {
        pd[d] = fa_new;
        ps[3 + d] = q;
        ps[9 + d] = v_next;
        if (m.pm32) write_mirror(m.pm32 + kMirror * pc_, d, q, v_next);
        if (!finite_bits(v_next) || !finite_bits(q)) *(volatile int32_t *)m.flag = 1;
        if (sub == 0) {
            if constexpr (kMixed) {
                pd[6] = fma(hdt, dWi_acc, pd[6]);
                if (need_we) pd[7] = fma(hdt, dWe_acc, pd[7]);
            } else {
                pd[6] += dWi_acc;
                if (need_we) pd[7] += dWe_acc;
            }
        }
    }
}

// The step's pass takes the particles in descending order: the facet pass ends with the last tetrahedra, whose
// shares are still in L2, and the next facet pass starts with the records written last (up to 1 % of a step).
template <class R, int MODE, int LPP, bool STREAM = false>
__global__ void __launch_bounds__(64, sizeof(R) == 4 ? 20 : 1) gather_kernel(DeviceModel m, double *__restrict__ out6)
{
    const int lane = threadIdx.x & 31;
    const int64_t blk = MODE == GATHER_STEP_MID ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int64_t p = ((blk * blockDim.x + threadIdx.x) >> 5) * (32 / LPP) + lane / LPP;
    gather_group<R, MODE, LPP, false, STREAM>(m, p, lane, out6);
}

// ------------------------------------------------------------------------------------------------
// Persistent step kernel: one cooperative launch runs `nsteps` whole steps.  Each step is the facet
// pass (warps take 8-tetrahedron tiles in a grid-stride loop), a grid barrier, the particle pass (warps
// take groups of 4 particles), and a second grid barrier; the arithmetic and summation orders are
// those of facet_warp_kernel and gather_kernel<.., 8>, so results equal the launch-pair path bit for
// bit.  The cooperative launch guarantees that all blocks are resident, so every barrier completes
// unless a block fails to arrive; each wait is nevertheless bounded (PersistCtl::wait_ns of
// %globaltimer and kMaxPolls polls), after which the block sets the status word and returns, and
// every other block stops at its next wait.
// ------------------------------------------------------------------------------------------------
constexpr uint32_t kMaxPolls = 1u << 24;

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Strong relaxed load at GPU scope: served by L2, and, unlike an acquire, it does not invalidate the
// SM's L1 at every poll (which would cost the blocks still working on that SM their cached lines).
__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier `target / gridDim.x` of the launch: all blocks' writes before it are visible to all blocks
// after it.  After the block's __syncthreads, thread 0 arrives with a release reduction on the
// arrival counter (it orders the block's earlier writes before the arrival; with `arrive` false, the
// fault-injection hook, it does not arrive) and polls the count with relaxed loads, spinning for 256
// polls and then sleeping 64 ns between polls, until it reaches `target`; an acquire fence after the
// last poll then orders the other blocks' writes before the block's later reads (a relaxed read
// followed by a fence is an acquire in the PTX memory model).  Returns false in every thread of the
// block if the wait gave up: its own limit was reached (the status word is set), or another block had
// set the status.
__device__ __forceinline__ bool grid_barrier(const PersistCtl &c, unsigned target, bool arrive)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        if (arrive) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c.arrive) : "memory");
        const uint64_t t0 = global_ns();
        for (uint32_t it = 0;; ++it) {
            if (ld_relaxed_gpu(c.arrive) >= target) break;
            if (*(volatile const int32_t *)c.status != 0) {
                ok = 0;
                break;
            }
            if (it >= kMaxPolls || global_ns() - t0 > c.wait_ns) {
                atomicCAS(c.status, 0, kStatusTimeout);
                ok = 0;
                break;
            }
            if (it > 256) __nanosleep(64);
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <class R, bool PF, bool S1, int WPB>
__global__ void __launch_bounds__(32 * WPB)
    step_persistent_kernel(const __grid_constant__ DeviceModel m, const void *__restrict__ vsrc, int64_t nsteps,
                           PersistCtl ctl)
{
    constexpr int TETS = kTileTets;
    __shared__ alignas(16) R sv_[WPB][TETS * 4][Stride<R>::row];
    __shared__ alignas(16) R spl_[WPB][6 * kPlane];
    __shared__ R seV_[WPB][TETS];
    __shared__ int sok_[WPB][TETS];
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = *(volatile const int32_t *)ctl.status;
    __syncthreads();
    if (s_stop != 0) return;  // an earlier launch gave up: no work (the whole block)
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * WPB + w, nw = (int64_t)gridDim.x * WPB;
    const int64_t tiles = m.T / TETS;             // T is a multiple of the tile
    const int64_t groups = ((int64_t)m.N + 3) / 4;  // 4 particles of 8 lanes per warp
    unsigned target = 0;
    for (int64_t n = 0; n < nsteps; ++n) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
        for (int64_t t = gw; t < tiles; t += nw)
            facet_tile<R, FACET_STEP, PF, S1, true>(m, vsrc, t * TETS, lane, sv_[w], spl_[w], seV_[w], sok_[w]);
        target += gridDim.x;
        if (!grid_barrier(ctl, target, !(n == 0 && (int)blockIdx.x == ctl.skip_block))) return;
        for (int64_t g = gw; g < groups; g += nw) gather_group<R, GATHER_STEP_MID, 8, true>(m, 4 * g + lane / 8, lane, nullptr);
        target += gridDim.x;
        if (!grid_barrier(ctl, target, true)) return;
    }
}

// FP64 variant: the facet phase takes the edge tiles of facet_edge_kernel.
template <bool PF, int WPB>
__global__ void __launch_bounds__(32 * WPB)
    step_persistent_edge_kernel(const __grid_constant__ DeviceModel m, const double *__restrict__ vsrc, int64_t nsteps,
                                PersistCtl ctl)
{
    __shared__ alignas(16) double sw[WPB][kEWords];
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = *(volatile const int32_t *)ctl.status;
    __syncthreads();
    if (s_stop != 0) return;  // an earlier launch gave up: no work (the whole block)
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * WPB + w, nw = (int64_t)gridDim.x * WPB;
    const int64_t tiles = ((int64_t)m.T + kEdgeTets - 1) / kEdgeTets;
    const int64_t groups = ((int64_t)m.N + 3) / 4;
    unsigned target = 0;
    for (int64_t n = 0; n < nsteps; ++n) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *m.step += 1;
        for (int64_t t = gw; t < tiles; t += nw)
            facet_edge_tile<PF, true>(m, vsrc, (int32_t)(t * kEdgeTets), lane, sw[w]);
        target += gridDim.x;
        if (!grid_barrier(ctl, target, !(n == 0 && (int)blockIdx.x == ctl.skip_block))) return;
        for (int64_t g = gw; g < groups; g += nw)
            gather_group<double, GATHER_STEP_MID, 8, true>(m, 4 * g + lane / 8, lane, nullptr);
        target += gridDim.x;
        if (!grid_barrier(ctl, target, true)) return;
    }
}

template <class R, bool PF, bool S1>
constexpr int persist_wpb()
{
    return sizeof(R) == 4 ? 4 : 2;  // static shared memory stays below 48 KB per block
}

template <class R, bool PF, bool S1>
const void *persist_fn()
{
    if constexpr (sizeof(R) == 4)
        return reinterpret_cast<const void *>(&step_persistent_kernel<R, PF, S1, persist_wpb<R, PF, S1>()>);
    else
        return reinterpret_cast<const void *>(&step_persistent_edge_kernel<PF, persist_wpb<R, PF, S1>()>);
}

// First half kick and drift of a stepping call: v_{n+1/2} = v_n + dt/2 a_n, q_{n+1} = q_n + dt v_{n+1/2}.
__global__ void __launch_bounds__(256) kick_kernel(DeviceModel m)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * (int64_t)m.N) return;
    const int64_t p = i / 6;
    const int d = (int)(i - 6 * p);
    double *ps = m.pstate + 16 * p;
    const double *pc = m.pconst + 8 * p;
    const int mask = (int)(((uint64_t)__double_as_longlong(pc[6]) >> (8 * d)) & 0xffu);
    const int sp = (int)__double_as_longlong(pc[7]);
    const double dt = m.spec[sp].dt;
    double vh;
    if (mask == 0) {
        const double fe = m.f_ext ? m.f_ext[6 * p + d] : 0.0;
        vh = ps[9 + d] + 0.5 * dt * (fe + m.pdyn[8 * p + d]) * pc[d];
    } else if (mask == 1) {
        vh = 0.0;
    } else {
        const double t = (double)(*m.step) * dt;
        vh = m.bc_vel[6 * p + d] * ramp(t + 0.5 * dt, m.spec[sp].inv_ramp);
    }
    const double q = ps[3 + d] + dt * vh;
    ps[9 + d] = vh;
    ps[3 + d] = q;
    if (m.pm32) write_mirror(m.pm32 + kMirror * p, d, q, vh);
}

// Whole-step values (q_n, v_n) of DOF d of internal particle p from the drifted state (q_{n+1},
// v_{n+1/2}) the library keeps between calls: the inverse of kick_kernel under the same boundary
// conditions.
__device__ __forceinline__ void unkick_dof(const DeviceModel &m, int64_t p, int d, double &qn, double &vn)
{
    const double *ps = m.pstate + 16 * p;
    const double *pc = m.pconst + 8 * p;
    const int mask = (int)(((uint64_t)__double_as_longlong(pc[6]) >> (8 * d)) & 0xffu);
    const SpecDyn &S = m.spec[(int)__double_as_longlong(pc[7])];
    const double vh = ps[9 + d];
    if (mask == 0) {
        const double fe = m.f_ext ? m.f_ext[6 * p + d] : 0.0;
        vn = vh - S.half_dt * (fe + m.pdyn[8 * p + d]) * pc[d];
    } else if (mask == 1) {
        vn = 0.0;
    } else {
        vn = m.bc_vel[6 * p + d] * ramp((double)(*m.step) * S.dt, S.inv_ramp);
    }
    qn = ps[3 + d] - S.dt * vh;
}

// Whole-step state into out12 [N][12] (q then v, internal order), or with out12 null into pstate (and
// the mirror) in place.
__global__ void __launch_bounds__(256) unkick_kernel(DeviceModel m, double *__restrict__ out12)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * (int64_t)m.N) return;
    const int64_t p = i / 6;
    const int d = (int)(i - 6 * p);
    double qn, vn;
    unkick_dof(m, p, d, qn, vn);
    if (out12) {
        out12[12 * p + d] = qn;
        out12[12 * p + 6 + d] = vn;
    } else {
        double *ps = m.pstate + 16 * p;
        ps[3 + d] = qn;
        ps[9 + d] = vn;
        if (m.pm32) write_mirror(m.pm32 + kMirror * p, d, qn, vn);
    }
}

// Whole-step state in the caller's particle order: caller particle k is internal particle pmap[k];
// q, v [n][6] (either may be null).
__global__ void __launch_bounds__(256) state_to_user_kernel(DeviceModel m, const int32_t *__restrict__ pmap, int64_t n,
                                                            double *__restrict__ q, double *__restrict__ v)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * n) return;
    const int64_t k = i / 6;
    const int d = (int)(i - 6 * k);
    double qn, vn;
    unkick_dof(m, pmap[k], d, qn, vn);
    if (q) q[i] = qn;
    if (v) v[i] = vn;
}

// FP32 mirror of every particle from the FP64 records.
__global__ void __launch_bounds__(256) mirror_kernel(DeviceModel m)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= m.N) return;
    const double *ps = m.pstate + 16 * p;
    float *pm = m.pm32 + kMirror * p;
    for (int k = 0; k < 3; ++k) d2f_split(ps[k], pm[k], pm[3 + k]);
    for (int d = 0; d < 6; ++d) write_mirror(pm, d, ps[3 + d], ps[9 + d]);
    for (int k = 21; k < kMirror; ++k) pm[k] = 0.0f;
}

// Perturbation of the displacements and rotations of free DOFs (dq [N][6], internal order).  In the
// drifted state q_{n+1} = q_n + dt v_{n+1/2}, adding dq to q_n adds it to q_{n+1}; velocities, forces
// and history are unchanged, so the next strain increment is measured from the perturbed state.
__global__ void __launch_bounds__(256) perturb_kernel(DeviceModel m, const double *__restrict__ dq)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * (int64_t)m.N) return;
    const int64_t p = i / 6;
    const int d = (int)(i - 6 * p);
    const int mask = (int)(((uint64_t)__double_as_longlong(m.pconst[8 * p + 6]) >> (8 * d)) & 0xffu);
    if (mask != 0) return;
    double *ps = m.pstate + 16 * p;
    const double q = ps[3 + d] + dq[i];
    ps[3 + d] = q;
    if (m.pm32) write_mirror(m.pm32 + kMirror * p, d, q, ps[9 + d]);
}

// 1 / x, x > 0, to an ulp or two: FP32 seed and two Newton steps, 4 FP64 instructions where the division takes
// about 9.  Where x or 1 / x is not a normal number (inverse masses below 2^-1022 or from 2^1022): the division.
__device__ __forceinline__ double recip64(double x)
{
    // seed from the mantissa alone (in [1, 2)), so that no x leaves FP32's range
    const long long b = __double_as_longlong(x);
    if ((unsigned)(b >> 52) - 1u >= 2044u) return 1.0 / x;
    const double mant = __longlong_as_double((b & 0xfffffffffffffll) | 0x3ff0000000000000ll);
    const double y0 = f2d_bits(__frcp_rn(d2f_trunc(mant)));
    const double y1 = fma(y0, fma(-mant, y0, 1.0), y0);
    const double y2 = fma(y1, fma(-mant, y1, 1.0), y1);  // in (0.5, 1]: exponent 1022 or 1023
    const int sh = 1023 - (int)((b >> 52) & 0x7ff);
    return __longlong_as_double(__double_as_longlong(y2) + ((long long)sh << 52));
}

// Energy sums of particles [p0, p1): thread = (particle, DOF), 8 lanes per particle (lanes 0..5 the DOFs,
// 6 and 7 the accumulators W_int and W_ext), up to kEnergyBlocks blocks striding over the particles, so
// that a specimen of a few thousand particles fills the chip (one particle per thread, a chain of six
// divisions each, took 15 us in 15 blocks on 3.7k particles; a step with a read-back there, the two
// copies of the error words included, went from 65 to 39 us).  Each block writes its
// 16 sums in a fixed order; the block that finishes last (ticket from an atomic counter that wraps back
// to 0) adds the partials in block order, and writes them with the handle's non-finite flag and barrier
// status to out18, which is pinned host memory: the caller waits for the stream and reads them there.
// No thread waits on another block.
constexpr int kEnergyBlocks = 304;
__global__ void __launch_bounds__(256) energy_kernel(DeviceModel m, int32_t p0, int32_t p1, double *partial,
                                                     unsigned *ticket, const int32_t *status, double *out18)
{
    __shared__ double red[8][8][3];  // warp, lane class, (kinetic, fixed reaction, prescribed reaction)
    __shared__ bool last;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, d = lane & 7;
    double kin = 0.0, rf = 0.0, rp = 0.0;  // for d = 6, 7 `kin` sums the accumulator
    for (int64_t p = (int64_t)p0 + (int64_t)blockIdx.x * 32 + (tid >> 3); p < p1; p += 32 * (int64_t)gridDim.x) {
        const double *pd = m.pdyn + 8 * p;
        const double fd = pd[d];
        if (d >= 6) {
            kin += fd;
            continue;
        }
        const double *pc = m.pconst + 8 * p;
        const double im = pc[d];
        const int mk = (int)(((uint64_t)__double_as_longlong(pc[6]) >> (8 * d)) & 0xffu);
        const SpecDyn &S = m.spec[(int)__double_as_longlong(pc[7])];
        // whole-step velocity v_n from the stored v_{n+1/2} (inverse half kick)
        double v = 0.0;
        if (mk == 0) {
            v = m.pstate[16 * p + 9 + d] - S.half_dt * (m.f_ext ? m.f_ext[6 * p + d] + fd : fd) * im;
        } else if (mk == 1) {
            rf -= fd;
        } else {
            const double t = (double)(*m.step) * S.dt;
            v = m.bc_vel[6 * p + d] * ramp(t, S.inv_ramp);
            const double ra = ramp(t + S.half_dt, S.inv_ramp) - ramp(t - S.half_dt, S.inv_ramp);
            rp += m.bc_vm[6 * p + d] * ra * S.inv_dt - fd;
        }
        if (mk != 1) kin += v * v * recip64(im);
    }
#pragma unroll
    for (int off = 16; off >= 8; off >>= 1) {
        kin += __shfl_xor_sync(0xffffffffu, kin, off);
        rf += __shfl_xor_sync(0xffffffffu, rf, off);
        rp += __shfl_xor_sync(0xffffffffu, rp, off);
    }
    if (lane < 8) {
        red[w][lane][0] = kin;
        red[w][lane][1] = rf;
        red[w][lane][2] = rp;
    }
    __syncthreads();
    // out: W_int, W_ext, W_kin, pad, fixed reactions (6), prescribed reactions (6)
    if (tid < 16) {
        double b = 0.0;
        for (int k = 0; k < 8; ++k) {
            if (tid < 2) b += red[k][6 + tid][0];
            if (tid == 2)
                for (int q = 0; q < 6; ++q) b += 0.5 * red[k][q][0];
            if (tid >= 4) b += red[k][(tid - 4) % 6][tid < 10 ? 1 : 2];
        }
        partial[16 * (int64_t)blockIdx.x + tid] = b;
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __shared__ double fin[16][16];
    const unsigned per = (gridDim.x + 15) / 16;  // partials of one of 16 consecutive runs of blocks
    double s = 0.0;
    for (unsigned k = (tid >> 4) * per; k < gridDim.x && k < ((tid >> 4) + 1) * per; ++k)
        s += __ldcg(partial + 16 * (int64_t)k + (tid & 15));
    fin[tid >> 4][tid & 15] = s;
    __syncthreads();
    if (tid < 16) {
        double r = 0.0;
#pragma unroll
        for (int k = 0; k < 16; ++k) r += fin[k][tid];
        out18[tid] = r;
    } else if (tid == 16) {
        out18[16] = (double)*m.flag;
    } else if (tid == 17) {
        out18[17] = (double)*status;
    }
}

// History <-> caller format (t_N, global tangential traction, e_max), in the internal facet order.
// The frame is rebuilt from the particle positions exactly as the facet pass forms it.
template <class R>
__device__ __forceinline__ bool facet_frame_of(const DeviceModel &m, int64_t f, V3<R> &n, V3<R> &mt, V3<R> &lt)
{
    const int64_t tt = f / 12;
    const int e = (int)(f - 12 * tt) >> 1;
    const int va = (0x211000 >> (4 * e)) & 0xF;
    const int vb = (0x332321 >> (4 * e)) & 0xF;
    const int *tv = reinterpret_cast<const int *>(m.tet) + 4 * tt;
    const int p0 = tv[0], pa = tv[va], pb = tv[vb];
    if (p0 < 0) return false;
    V3<R> dxa, dxb;
    if constexpr (sizeof(R) == 4) {
        const float *x0 = m.pm32 + kMirror * (int64_t)p0, *xa = m.pm32 + kMirror * (int64_t)pa,
                    *xb = m.pm32 + kMirror * (int64_t)pb;
        dxa = {(xa[0] - x0[0]) + (xa[3] - x0[3]), (xa[1] - x0[1]) + (xa[4] - x0[4]),
               (xa[2] - x0[2]) + (xa[5] - x0[5])};
        dxb = {(xb[0] - x0[0]) + (xb[3] - x0[3]), (xb[1] - x0[1]) + (xb[4] - x0[4]),
               (xb[2] - x0[2]) + (xb[5] - x0[5])};
    } else {
        const double *x0 = m.pstate + 16 * (int64_t)p0, *xa = m.pstate + 16 * (int64_t)pa,
                     *xb = m.pstate + 16 * (int64_t)pb;
        dxa = {R(xa[0] - x0[0]), R(xa[1] - x0[1]), R(xa[2] - x0[2])};
        dxb = {R(xb[0] - x0[0]), R(xb[1] - x0[1]), R(xb[2] - x0[2])};
    }
    const V3<R> d = dxb - dxa;
    const R inv_l = rsqrt_(dot(d, d));
    n = inv_l * d;
    tangent_frame(n, mt, lt);
    return true;
}

// History of n facets in the caller's order: umap[k] = 2 f + s for internal facet f, s = 1 where the
// caller's facet runs from the internal vertex b to a (the tangential traction vector flips sign).
// The FP64 pipe (conversions included) bound this read-out: mixed mode now forms the products of two
// floats exactly with integer instructions and spends one FP64 addition per component (the same bits as
// FP64 arithmetic gives), FP64 mode takes the stored frames.  The 5 values per facet go through shared
// memory so that a block writes one contiguous range.  11.4M facets, mixed: 401 -> 180 us; 1.15M
// facets, FP64: 99 -> 27 us (ncu).
constexpr int kHistBlock = 128;
template <class R>
__global__ void __launch_bounds__(kHistBlock)
    hist_to_user_kernel(DeviceModel m, const int32_t *__restrict__ umap, int64_t nf, double *__restrict__ out5)
{
    __shared__ double s5[5 * kHistBlock];
    const int64_t k0 = (int64_t)blockIdx.x * kHistBlock, k = k0 + threadIdx.x;
    if (k < nf) {
        const int32_t code = umap[k];
        const int64_t f = code >> 1;
        const R4<R> h = static_cast<const R4<R> *>(m.hist)[f];
        double o[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        if constexpr (sizeof(R) == 4) {
            V3<float> n, mt, lt;
            if (facet_frame_of<float>(m, f, n, mt, lt)) {
                o[0] = f2d_bits(h.x);
                o[1] = mul_exact(h.y, mt.x) + mul_exact(h.z, lt.x);
                o[2] = mul_exact(h.y, mt.y) + mul_exact(h.z, lt.y);
                o[3] = mul_exact(h.y, mt.z) + mul_exact(h.z, lt.z);
                o[4] = f2d_bits(h.w);
            }
        } else {
            const int64_t ed = f >> 1;  // the facet's edge: m / l at 3..5, t / l at 6..8, l at 14 of its frame
            const double *fr = m.frame + 16 * ed;
            if (fr[14] > 0.0) {
                const double a = h.y * fr[14], b = h.z * fr[14];
                o[0] = h.x;
                o[1] = fma(a, fr[3], b * fr[6]);
                o[2] = fma(a, fr[4], b * fr[7]);
                o[3] = fma(a, fr[5], b * fr[8]);
                o[4] = h.w;
            }
        }
        const long long flip = (long long)(code & 1) << 63;
#pragma unroll
        for (int c = 0; c < 5; ++c)
            s5[5 * threadIdx.x + c] =
                c >= 1 && c <= 3 ? __longlong_as_double(__double_as_longlong(o[c]) ^ flip) : o[c];
    }
    __syncthreads();
    const int64_t n5 = 5 * (nf - k0 < kHistBlock ? nf - k0 : (int64_t)kHistBlock);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const int i = threadIdx.x + c * kHistBlock;
        if (i < n5) out5[5 * k0 + i] = s5[i];
    }
}

template <class R>
__global__ void hist_from_user_kernel(DeviceModel m, const double *__restrict__ in5)
{
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= 12 * (int64_t)m.T) return;
    V3<R> n, mt, lt;
    R4<R> h;
    h.x = h.y = h.z = h.w = R(0);
    if (facet_frame_of<R>(m, f, n, mt, lt)) {
        const double *u = in5 + 5 * f;
        h.x = R(u[0]);
        h.y = R(u[1] * double(mt.x) + u[2] * double(mt.y) + u[3] * double(mt.z));
        h.z = R(u[1] * double(lt.x) + u[2] * double(lt.y) + u[3] * double(lt.z));
        h.w = R(u[4]);
    }
    static_cast<R4<R> *>(m.hist)[f] = h;
}

// Whether the mixed step reads geometry, history and (in the particle pass) the shares, and writes the history,
// with the streaming hint.  They pass through once per step; where the model's arrays (about 75 bytes per
// facet, 126 MB of L2) are around the size of L2 the hint leaves L2 to what both passes share (records, slot
// tables).  Where they are several times L2, or other models' steps run in between, nothing survives a pass
// anyway and marking the shares first for eviction only sends them to memory.  10 steps in tension, without
// and with the hint, us (compression alike):
//   facets           0.84M       2.0M      2.6M      3.5M       4.8M       6.0M       7.5M       9.4M      11.3M
//   one alone     279, 278  548, 524  711, 666  910, 855 1182, 1118 1451, 1393 1784, 1745 2204, 2172 2609, 2582
//   three in turn 197, 190  448, 438  599, 589  802, 805 1075, 1096 1346, 1383 1689, 1742 2112, 2191 2537, 2621
// The line is where the two uses balance: at 4M facets the hint takes 5 % off a model stepped alone and adds
// 1 % where three take turns; past it, it gives less and costs more.  A batch of 6.1M facets loses (2175,
// 2230); smaller batches were not measured and go without.
bool stream_hints(const DeviceModel &m) { return 12 * (int64_t)m.T <= 4000000; }

template <class R, int MODE, bool PF>
cudaError_t launch_facet_pf(const DeviceModel &m, const void *pst, cudaStream_t s, const BatchLaw *bl)
{
    const int tpb = m.tets_per_block;
    const unsigned blocks = (unsigned)((m.T + tpb - 1) / tpb);
    if (blocks == 0) return cudaSuccess;
    // FP32 facet pass with 8-tetrahedron tiles: one tile per warp, 2 warps per block (measured on GB300:
    // 43.6 us against 47.4 us for the 96-thread block kernel on 1.82M facets).
    if constexpr (sizeof(R) == 4) {
        if (tpb == kTileTets) {
            constexpr int WPB = 2;
            const int64_t tiles = (m.T + kTileTets - 1) / kTileTets;
            const unsigned nb = (unsigned)((tiles + WPB - 1) / WPB);
            if constexpr (MODE == FACET_STEP) {
                if (m.n_spec == 1 && stream_hints(m)) {
                    facet_warp_kernel<R, MODE, WPB, PF, true, true><<<nb, 32 * WPB, 0, s>>>(m, pst);
                    return cudaGetLastError();
                }
            }
            if (m.n_spec == 1)
                facet_warp_kernel<R, MODE, WPB, PF, true><<<nb, 32 * WPB, 0, s>>>(m, pst);
            else if (bl && bl->n == m.n_spec)
                facet_warp_batch_kernel<MODE, WPB, PF><<<nb, 32 * WPB, 0, s>>>(m, pst, *bl);
            else
                facet_warp_kernel<R, MODE, WPB, PF, false><<<nb, 32 * WPB, 0, s>>>(m, pst);
            return cudaGetLastError();
        }
    }
    if constexpr (sizeof(R) == 8 && MODE == FACET_STEP) {
        // the FP64 step: edge tiles whatever the launch shape, so that it has one arithmetic (the block kernel
        // forms its sums in another order, and takes twice the time: facet_edge_tile)
        const int64_t tiles = ((int64_t)m.T + kEdgeTets - 1) / kEdgeTets;
        facet_edge_kernel<PF><<<(unsigned)((tiles + kEdgeWarps - 1) / kEdgeWarps), 32 * kEdgeWarps, 0, s>>>(
            m, static_cast<const double *>(pst));
    } else {
        switch (tpb) {
        case 16:
            facet_kernel<R, MODE, 16, PF><<<blocks, 192, 0, s>>>(m, pst);
            break;
        case 32:
            facet_kernel<R, MODE, 32, PF><<<blocks, 384, 0, s>>>(m, pst);
            break;
        default:
            if constexpr (sizeof(R) == 8) facet_kernel<R, MODE, 8, PF><<<blocks, 96, 0, s>>>(m, pst);
            break;
        }
    }
    return cudaGetLastError();
}

// Per-facet parameters matter only where the law or E0 / alpha enter: the step and the metrics.
template <class R, int MODE>
cudaError_t launch_facet_tpb(const DeviceModel &m, const void *pst, cudaStream_t s, const BatchLaw *bl)
{
    if constexpr (MODE == FACET_STEP || MODE == FACET_METRIC)
        if (m.pf) return launch_facet_pf<R, MODE, true>(m, pst, s, bl);
    return launch_facet_pf<R, MODE, false>(m, pst, s, bl);
}

// Persistent launch of `nsteps` steps (cooperative; grid = resident blocks per SM x SMs).  Returns
// cudaErrorCooperativeLaunchTooLarge (or another launch error) if the grid cannot be co-resident.
template <class R>
cudaError_t launch_persistent_r(const DeviceModel &m, int64_t nsteps, const PersistCtl &ctl, int *grid_out,
                                cudaStream_t s)
{
    const void *fn = (sizeof(R) == 4 && m.n_spec == 1) ? (m.pf ? persist_fn<R, true, true>() : persist_fn<R, false, true>())
                                                        : (m.pf ? persist_fn<R, true, false>() : persist_fn<R, false, false>());
    const int threads = 32 * persist_wpb<R, false, false>();
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    // as many blocks as the device holds at once, but no more than the work needs: every block takes
    // part in every barrier, so idle blocks on a small specimen would only slow the barriers down
    // (a tile takes a warp, as do 4 particles)
    const int wpb = threads / 32;
    constexpr int tets = sizeof(R) == 4 ? kTileTets : kEdgeTets;
    const int64_t tiles = ((int64_t)m.T + tets - 1) / tets, groups = ((int64_t)m.N + 3) / 4;
    const int64_t need = (std::max(tiles, groups) + wpb - 1) / wpb;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * sms, need));
    if (grid_out) *grid_out = (int)grid;
    if (nsteps <= 0) return cudaSuccess;
    const void *vsrc = sizeof(R) == 4 ? static_cast<const void *>(m.pm32) : static_cast<const void *>(m.pstate);
    DeviceModel mm = m;
    int64_t ns = nsteps;
    PersistCtl c = ctl;
    void *args[] = {&mm, &vsrc, &ns, &c};
    e = cudaMemsetAsync(ctl.arrive, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, 0, s);
}

}  // namespace

cudaError_t launch_unkick(const DeviceModel &m, double *out12, cudaStream_t s)
{
    const int64_t n = 6 * (int64_t)m.N;
    if (n == 0) return cudaSuccess;
    unkick_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(m, out12);
    return cudaGetLastError();
}

cudaError_t launch_state_to_user(const DeviceModel &m, const int32_t *pmap, int64_t n, double *q, double *v,
                                 cudaStream_t s)
{
    if (n <= 0 || (!q && !v)) return cudaSuccess;
    state_to_user_kernel<<<(unsigned)((6 * n + 255) / 256), 256, 0, s>>>(m, pmap, n, q, v);
    return cudaGetLastError();
}

cudaError_t launch_kick(const DeviceModel &m, cudaStream_t s)
{
    const int64_t n = 6 * (int64_t)m.N;
    if (n == 0) return cudaSuccess;
    kick_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(m);
    return cudaGetLastError();
}

template <class R>
cudaError_t launch_facet(const DeviceModel &m, int mode, const void *src_override, cudaStream_t s,
                         const BatchLaw *bl)
{
    const void *pst = src_override ? src_override
                                   : (sizeof(R) == 4 ? static_cast<const void *>(m.pm32)
                                                     : static_cast<const void *>(m.pstate));
    switch (mode) {
    case FACET_FROM_HIST:
        return launch_facet_tpb<R, FACET_FROM_HIST>(m, pst, s, bl);
    case FACET_ELASTIC:
        return launch_facet_tpb<R, FACET_ELASTIC>(m, pst, s, bl);
    case FACET_METRIC:
        return launch_facet_tpb<R, FACET_METRIC>(m, pst, s, bl);
    default:
        return launch_facet_tpb<R, FACET_STEP>(m, pst, s, bl);
    }
}

template <class R, int LPP>
cudaError_t launch_gather_lpp(const DeviceModel &m, int mode, double *out6, cudaStream_t s)
{
    const int64_t warps = ((int64_t)m.N + (32 / LPP) - 1) / (32 / LPP);
    // blocks of 2 warps, up to 20 per SM at 48 registers (mixed mode; measured on GB300 against 12, 16
    // and 18 per SM with more shares in flight, and against 8-warp blocks)
    const unsigned blocks = (unsigned)((warps * 32 + 63) / 64);
    switch (mode) {
    case GATHER_ASSEMBLE:
        gather_kernel<R, GATHER_ASSEMBLE, LPP><<<blocks, 64, 0, s>>>(m, out6);
        break;
    default:
        if constexpr (sizeof(R) == 4 && LPP == 8) {
            if (m.n_spec == 1 && stream_hints(m)) {
                gather_kernel<R, GATHER_STEP_MID, LPP, true><<<blocks, 64, 0, s>>>(m, out6);
                break;
            }
        }
        gather_kernel<R, GATHER_STEP_MID, LPP><<<blocks, 64, 0, s>>>(m, out6);
        break;
    }
    return cudaGetLastError();
}

template <class R>
cudaError_t launch_gather(const DeviceModel &m, int mode, double *out6, cudaStream_t s)
{
    if (m.N == 0) return cudaSuccess;
    switch (m.gather_lanes) {
    case 32:
        return launch_gather_lpp<R, 32>(m, mode, out6, s);
    case 16:
        return launch_gather_lpp<R, 16>(m, mode, out6, s);
    default:
        return launch_gather_lpp<R, 8>(m, mode, out6, s);
    }
}

cudaError_t launch_frames(const DeviceModel &m, cudaStream_t s)
{
    const int64_t n = 6 * (int64_t)m.T;
    if (!m.frame || n == 0) return cudaSuccess;
    frame_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(m);
    return cudaGetLastError();
}

cudaError_t launch_mirror(const DeviceModel &m, cudaStream_t s)
{
    if (!m.pm32 || m.N == 0) return cudaSuccess;
    mirror_kernel<<<(unsigned)((m.N + 255) / 256), 256, 0, s>>>(m);
    return cudaGetLastError();
}

cudaError_t launch_perturb(const DeviceModel &m, const double *dq, cudaStream_t s)
{
    const int64_t n = 6 * (int64_t)m.N;
    if (n == 0) return cudaSuccess;
    perturb_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(m, dq);
    return cudaGetLastError();
}

cudaError_t launch_energy(const DeviceModel &m, int32_t p0, int32_t p1, double *partial, unsigned *ticket,
                          const int32_t *status, double *out18, cudaStream_t s)
{
    // an empty range still reports the flags
    const int nb = std::min(kEnergyBlocks, std::max(1, (p1 - p0 + 31) / 32));
    energy_kernel<<<nb, 256, 0, s>>>(m, p0, p1, partial, ticket, status, out18);
    return cudaGetLastError();
}

template <class R>
cudaError_t launch_hist_to_user(const DeviceModel &m, const int32_t *umap, int64_t n, double *out5, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    hist_to_user_kernel<R><<<(unsigned)((n + kHistBlock - 1) / kHistBlock), kHistBlock, 0, s>>>(m, umap, n, out5);
    return cudaGetLastError();
}

template <class R>
cudaError_t launch_hist_from_user(const DeviceModel &m, const double *in5, cudaStream_t s)
{
    const int64_t n = 12 * (int64_t)m.T;
    if (n == 0) return cudaSuccess;
    hist_from_user_kernel<R><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(m, in5);
    return cudaGetLastError();
}

template <class R>
cudaError_t launch_persistent(const DeviceModel &m, int64_t nsteps, const PersistCtl &ctl, int *grid_out,
                              cudaStream_t s)
{
    return launch_persistent_r<R>(m, nsteps, ctl, grid_out, s);
}

template cudaError_t launch_persistent<float>(const DeviceModel &, int64_t, const PersistCtl &, int *, cudaStream_t);
template cudaError_t launch_persistent<double>(const DeviceModel &, int64_t, const PersistCtl &, int *, cudaStream_t);
template cudaError_t launch_facet<float>(const DeviceModel &, int, const void *, cudaStream_t, const BatchLaw *);
template cudaError_t launch_facet<double>(const DeviceModel &, int, const void *, cudaStream_t, const BatchLaw *);
template cudaError_t launch_gather<float>(const DeviceModel &, int, double *, cudaStream_t);
template cudaError_t launch_gather<double>(const DeviceModel &, int, double *, cudaStream_t);
template cudaError_t launch_hist_to_user<float>(const DeviceModel &, const int32_t *, int64_t, double *, cudaStream_t);
template cudaError_t launch_hist_to_user<double>(const DeviceModel &, const int32_t *, int64_t, double *, cudaStream_t);
template cudaError_t launch_hist_from_user<float>(const DeviceModel &, const double *, cudaStream_t);
template cudaError_t launch_hist_from_user<double>(const DeviceModel &, const double *, cudaStream_t);

}  // namespace ldpm
