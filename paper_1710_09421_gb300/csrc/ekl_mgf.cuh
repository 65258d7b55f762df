// Lattice-level smoothing of the split multigrid solve (ekl_mgs.cuh) with two
// half sweeps per launch: a V-cycle's eight lattice passes become four.
//
// Every red-black update reads only the other colour, so a smoothing pass is
// determined by the colour-0 values it starts from; between launches only
// those are kept, in a compact array with one float per x-pair (half a
// vector's bytes).  Each launch takes them to the next ones:
//   PRE    c0 = r / deg          -> c1 -> c0            (pre-smoothing, first half)
//   RESTR  c0                    -> c1 -> residual, summed over 2x2x2 cells to level 1
//   PRO    c0 + correction       -> c1 -> c0            (post-smoothing, first half)
//   POST   c0                    -> c1 -> c0, and z = both colours in full
// The updates, the residual and the restriction's order of additions are
// those of the one-half-sweep passes (ekl_mg.cuh), so z and level 1's
// right-hand side are the same bit for bit.
//
// A block walks the planes of a z-chunk of a tile of whole x-rows (or of
// x-segments on wide lattices) with a halo of two rows, two planes and, on
// segments, 2 V nodes.  A thread owns 2 V consecutive nodes of one row, V of
// each colour.  At step q it takes colour 0 of plane q, updates colour 1 of
// plane q - 1 and colour 0 (or the residual) of plane q - 2.  The z neighbours
// of an update are the thread's own values of the planes before and after, in
// registers; the y neighbours and one x neighbour come from shared memory,
// written a step earlier, so one block barrier per plane is enough.  The next
// plane's loads are issued a step ahead.  The loop is unrolled over three
// planes, so the register rings rotate by name.
//
// What bounds it: the chain of a plane step (0.9 us: a plane's loads, the two
// dependent updates and the barrier) at 15 to 16 warps an SM, so it serves
// lattices larger than L2, where the one-half-sweep passes are bound by their
// traffic.  Counters on 128x128x256 (10 warps an SM): issue slots 30 to 34 % busy,
// DRAM 18 to 23 % of its peak; warps wait for loads (1.8 to 3.2 cycles per
// instruction issued) and at the barrier (1.3 to 2.2).  256x256x512, us per launch: PRE 66, RESTR 108, PRO 79, POST 86 and
// the r.z partials 47, in place of three half sweeps of 88, the restriction of
// 101, and half sweeps of 127, 88, 88 and 106.  Two half sweeps per launch on
// 64x64x128 (13 us each), a whole pass per launch in tiles with a halo of four
// (13 us each) and planes staged three ahead with cp.async (109 us instead of 90)
// were slower.
#pragma once
#include "ekl_mg.cuh"

namespace ekl {

constexpr int MGF_THREADS = 512;   // 128 registers a thread
enum { MGF_PRE = 0, MGF_RESTR = 1, MGF_PRO = 2, MGF_POST = 3 };

// whether a solve over this many nodes does not stay in L2 (126 MB): 37 bytes a
// node, r, z, p, p', q, the link byte, and phi and b of 8
inline bool mgf_beyond_l2(long long nodes) { return (size_t)nodes * 37 > (size_t)126 << 20; }

struct MgfGeom {
    int nx, ny, nz, per[3];
    int tx, own_y, own_z;          // nodes, rows and planes of a tile (rows and planes even)
    int ntx, nty, ntz;             // tiles
    int lpr, rows;                 // threads per row (with halo threads on segments), rows with halo
};

__host__ __device__ inline int mgf_threads(const MgfGeom &G) { return (G.lpr * G.rows + 31) / 32 * 32; }

// dynamic shared memory: colour-0 planes (three: the residual looks two
// planes back), colour-1 planes (two) and the odd rows' x-pair residuals (two)
template <int MODE> __host__ __device__ inline size_t mgf_smem(const MgfGeom &G, int V)
{
    const size_t plane = (size_t)G.lpr * V * G.rows;
    return (MODE == MGF_RESTR ? 3 + 2 + 2 : 2 + 2) * plane * sizeof(float);
}

template <int V> struct MgfVec { float v[V]; };
template <int V> __device__ __forceinline__ MgfVec<V> mgf_zero()
{
    MgfVec<V> r;
#pragma unroll
    for (int i = 0; i < V; i++) r.v[i] = 0.f;
    return r;
}
template <int V> __device__ __forceinline__ MgfVec<V> mgf_lds(const float *p)
{
    MgfVec<V> r;
    if constexpr (V == 4) {
        const float4 t = *(const float4 *)p;
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else {
        const float2 t = *(const float2 *)p;
        r.v[0] = t.x; r.v[1] = t.y;
    }
    return r;
}
template <int V> __device__ __forceinline__ void mgf_sts(float *p, const MgfVec<V> &a)
{
    if constexpr (V == 4) *(float4 *)p = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
    else *(float2 *)p = make_float2(a.v[0], a.v[1]);
}
template <int V> __device__ __forceinline__ MgfVec<V> mgf_ldg(const float *p)
{
    MgfVec<V> r;
    if constexpr (V == 4) {
        const float4 t = __ldcg((const float4 *)p);
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else {
        const float2 t = __ldcg((const float2 *)p);
        r.v[0] = t.x; r.v[1] = t.y;
    }
    return r;
}
template <int V> __device__ __forceinline__ void mgf_stg(float *p, const MgfVec<V> &a)
{
    if constexpr (V == 4) __stcg((float4 *)p, make_float4(a.v[0], a.v[1], a.v[2], a.v[3]));
    else __stcg((float2 *)p, make_float2(a.v[0], a.v[1]));
}

// the link bytes of V nodes of one colour, a byte each
constexpr unsigned MGF_WALLS = 0x80808080u;
__device__ __forceinline__ unsigned mgf_byte(unsigned lk, int i) { return (lk >> (8 * i)) & 0xffu; }
// nodes that take no value: walls and nodes without an open face
__device__ __forceinline__ bool mgf_dead(unsigned b) { return (b & MG_LINK_SOLID) || (b & 0x7Eu) == 0x7Eu; }

// a + b on two floats at once (one instruction, each half rounded to nearest)
__device__ __forceinline__ float2 mgf_add2(float2 a, float2 b)
{
    float2 r;
    asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n"
        " mov.b64 {%0, %1}, z;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
template <int V> __device__ __forceinline__ void mgf_addv(MgfVec<V> &a, const MgfVec<V> &b)
{
#pragma unroll
    for (int i = 0; i < V; i += 2) {
        const float2 t = mgf_add2(make_float2(a.v[i], a.v[i + 1]), make_float2(b.v[i], b.v[i + 1]));
        a.v[i] = t.x;
        a.v[i + 1] = t.y;
    }
}

// Neighbours of V nodes whose x-parity in the row is s (0: the even nodes):
// `own` holds the other colour of the same row, `edge` its one value outside
// the thread's nodes; closed faces and walls contribute zeros.  acc is added
// to in face order.
template <int V>
__device__ __forceinline__ void mgf_gather(MgfVec<V> &acc, const MgfVec<V> &own, float edge, bool s,
                                           const MgfVec<V> &ym, const MgfVec<V> &yp, const MgfVec<V> &zm,
                                           const MgfVec<V> &zp)
{
    // the row's other-colour values from the first node's left neighbour on
    float w[V + 1];
    w[0] = s ? own.v[0] : edge;
#pragma unroll
    for (int i = 1; i < V; i++) w[i] = s ? own.v[i] : own.v[i - 1];
    w[V] = s ? edge : own.v[V - 1];
#pragma unroll
    for (int i = 0; i < V; i++) {
        acc.v[i] += w[i];
        acc.v[i] += w[i + 1];
    }
    mgf_addv(acc, ym);
    mgf_addv(acc, yp);
    mgf_addv(acc, zm);
    mgf_addv(acc, zp);
}
// Inverse degree (0 on dead nodes) and degree of a node by its link byte, in
// shared memory: beside walls a warp then takes one load per node, where the
// bit counts, selects and conversions took some 20 instructions and half of
// a step on lattices with a membrane.
struct MgfLut {
    float inv[256], deg[256];
};
__device__ __forceinline__ void mgf_lut_fill(MgfLut &t)
{
    for (int b = threadIdx.x; b < 256; b += blockDim.x) {
        const int d = __popc(mg_open((unsigned)b));
        t.inv[b] = mgf_dead((unsigned)b) ? 0.f : mg_inv_deg(d);
        t.deg[b] = (float)d;
    }
    __syncthreads();
}
// (r + sum) / deg, zero on dead nodes
template <int V> __device__ __forceinline__ void mgf_scale(MgfVec<V> &a, unsigned lk, const MgfLut &t)
{
    if (lk == 0) {
#pragma unroll
        for (int i = 0; i < V; i++) a.v[i] *= 1.f / 6.f;
    } else {
#pragma unroll
        for (int i = 0; i < V; i++) a.v[i] *= t.inv[mgf_byte(lk, i)];
    }
}

struct MgfArgs {
    const float *r;
    const uint8_t *link;
    const float *cin;   // compact colour-0 values read (RESTR, PRO, POST)
    float *cout;        // compact colour-0 values written (PRE, PRO)
    float *z;           // POST: the full vector
    const float *e1;    // PRO: level-1 correction
    float *f1, *e1out;  // RESTR: level-1 right-hand side, and its first smoothing values
    const float4 *sig1;
    int cnx, cny, cnz;  // level-1 extents
};

template <int MODE, int V, bool FIRST>
__device__ __forceinline__ void mgf_body(const MgfGeom &G, const MgfArgs &A, int tile)
{
    extern __shared__ __align__(16) float mgf_sm[];
    __shared__ MgfLut lut;
    mgf_lut_fill(lut);
    const float deg6 = lut.deg[0];  // six open faces
    const int pitch = G.lpr * V, plane = pitch * G.rows;
    constexpr int N0 = MODE == MGF_RESTR ? 3 : 2;
    float *s0 = mgf_sm, *s1 = s0 + N0 * plane, *sr = s1 + 2 * plane;
    const int bx = tile % G.ntx, u = tile / G.ntx, by = u % G.nty, bz = u / G.nty;
    const int i = threadIdx.x % G.lpr, j = threadIdx.x / G.lpr;
    const bool thr = j < G.rows;  // (the block may have a few threads more)
    // this thread's nodes: x .. x + 2 V - 1 of row y
    const bool seg = G.ntx > 1;
    int x = bx * G.tx + 2 * V * (seg ? i - 1 : i), y = by * G.own_y + j - 2;
    bool live = thr;
    const bool own_x = seg ? i > 0 && i < G.lpr - 1 && x < G.nx : true;
    if (x < 0 || x >= G.nx) {
        live = live && G.per[0];
        x += x < 0 ? G.nx : -G.nx;
    }
    const bool own_y = j >= 2 && j < G.own_y + 2 && y < G.ny;
    if (y < 0 || y >= G.ny) {
        // beyond a closed side, or past the last tile's rows
        live = live && G.per[1] && y < 2 * G.ny && y >= -G.ny;
        y += y < 0 ? G.ny : -G.ny;
    }
    live = live && x >= 0 && x < G.nx && y >= 0 && y < G.ny;
    const bool mine = live && own_x && own_y;
    const int za = bz * G.own_z, zb = min(za + G.own_z, G.nz);
    // shared-memory offsets of this thread's values and of its neighbours'
    const int jj = thr ? j : 0, o = jj * pitch + i * V;
    const int om = (jj > 0 ? jj - 1 : jj) * pitch + i * V, op = (jj < G.rows - 1 ? jj + 1 : jj) * pitch + i * V;
    const int row = jj * pitch;
    const bool wrap = !seg && G.per[0];
    // index (in a plane) of the value left of the thread's first and right of its last, -1: none
    const int ol = i > 0 ? o - 1 : wrap ? row + pitch - 1 : -1;
    const int orr = i < G.lpr - 1 ? o + V : wrap ? row : -1;
    const int nxy = G.nx * G.ny, hrow = (G.nx >> 1) * y, hxy = (G.nx >> 1) * G.ny;

    // raw values of the next plane and its index in the lattice
    float4 fr[V / 2];     // r of the 2 V nodes
    uint2 fl;             // their link bytes (V = 2: .x)
    MgfVec<V> fc, fe;     // compact colour 0, level-1 correction
    const int n0 = x + G.nx * y, h0 = (x >> 1) + hrow;
    int zq = za - 2;      // plane of the next fetch
    if (zq < 0 && G.per[2]) zq += G.nz;
    auto fetch = [&](bool any) {
#pragma unroll
        for (int k = 0; k < V / 2; k++) fr[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        fl = make_uint2(MGF_WALLS, MGF_WALLS);
        fc = mgf_zero<V>();
        fe = mgf_zero<V>();
        if (any && live && zq >= 0 && zq < G.nz) {
            const int n = n0 + nxy * zq, h = h0 + hxy * zq;
#pragma unroll
            for (int k = 0; k < V / 2; k++) fr[k] = __ldcg((const float4 *)(A.r + n) + k);
            if constexpr (V == 4) fl = __ldg((const uint2 *)(A.link + n));
            else fl.x = __ldg((const unsigned *)(A.link + n));
            if constexpr (MODE != MGF_PRE) fc = mgf_ldg<V>(A.cin + h);
            if constexpr (MODE == MGF_PRO) fe = mgf_ldg<V>(A.e1 + (x >> 1) + A.cnx * ((y >> 1) + A.cny * (zq >> 1)));
        }
        zq++;
        if (zq == G.nz && G.per[2]) zq = 0;
    };

    // what a thread keeps of a plane: both colours, r and the link bytes
    struct Plane {
        MgfVec<V> c0, c1, r0, r1;
        unsigned l0, l1;
    };
    Plane R[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        R[k].c0 = R[k].c1 = R[k].r0 = R[k].r1 = mgf_zero<V>();
        R[k].l0 = R[k].l1 = MGF_WALLS;
    }
    MgfVec<V> c0d = mgf_zero<V>();  // RESTR: colour 0 of plane q - 3
    MgfVec<V> c1d = mgf_zero<V>();  // colour 1 of plane q - 3
    MgfVec<V> rs = mgf_zero<V>(), low = mgf_zero<V>();  // RESTR: x-pair residuals of the last plane; lower plane's sums
    (void)c0d; (void)rs; (void)low;
    fetch(true);
    int k0 = 0;  // buffer of plane q among the N0 colour-0 planes
    // the residual's sums are completed a step after their plane
    const int qend = zb + (MODE == MGF_RESTR ? 2 + (zb & 1) : 1);
    // one step; a, b, c hold the planes q, q - 1 and q - 2
    auto step = [&](int q, Plane &a, Plane &b, Plane &c) {
        // colour 0 of the row's plane q sits on x-parity sp
        const bool sp = (y + q) & 1;
        // the neighbours of both updates, written a step ago or earlier: all
        // shared loads first
        const int kb = k0 == 0 ? N0 - 1 : k0 - 1;            // plane q - 1
        const int oe = sp ? orr : ol;
        const float *pb = s0 + kb * plane, *p1 = s1 + (q & 1) * plane;
        const MgfVec<V> ym0 = mgf_lds<V>(pb + om), yp0 = mgf_lds<V>(pb + op);
        const float edge = oe < 0 ? 0.f : pb[oe];
        const MgfVec<V> ym = mgf_lds<V>(p1 + om), yp = mgf_lds<V>(p1 + op);
        const float edge1 = oe < 0 ? 0.f : p1[oe];
        {
            MgfVec<V> ev, od;  // even and odd nodes
#pragma unroll
            for (int t = 0; t < V / 2; t++) {
                ev.v[2 * t] = fr[t].x;
                od.v[2 * t] = fr[t].y;
                ev.v[2 * t + 1] = fr[t].z;
                od.v[2 * t + 1] = fr[t].w;
            }
            unsigned le, lo;
            if constexpr (V == 4) {
                le = __byte_perm(fl.x, fl.y, 0x6420);
                lo = __byte_perm(fl.x, fl.y, 0x7531);
            } else {
                le = __byte_perm(fl.x, 0u, 0x4420);
                lo = __byte_perm(fl.x, 0u, 0x4431);
            }
#pragma unroll
            for (int t = 0; t < V; t++) {
                a.r0.v[t] = sp ? od.v[t] : ev.v[t];
                a.r1.v[t] = sp ? ev.v[t] : od.v[t];
            }
            a.l0 = sp ? lo : le;
            a.l1 = sp ? le : lo;
        }
        if constexpr (MODE == MGF_PRE) {
            a.c0 = a.r0;
            mgf_scale(a.c0, a.l0, lut);
        } else if constexpr (MODE == MGF_PRO) {
            a.c0 = fc;
            mgf_addv(a.c0, fe);
            if (a.l0 != 0) {
#pragma unroll
                for (int t = 0; t < V; t++)
                    if (mgf_dead(mgf_byte(a.l0, t))) a.c0.v[t] = 0.f;
            }
        } else {
            a.c0 = fc;
        }
        if (thr) mgf_sts<V>(s0 + k0 * plane + o, a.c0);
        fetch(q <= zb);
        // colour 1 of plane q - 1, whose x-parity is sp there
        b.c1 = b.r1;
        mgf_gather(b.c1, b.c0, edge, sp, ym0, yp0, c.c0, a.c0);
        mgf_scale(b.c1, b.l1, lut);
        if (thr) mgf_sts<V>(s1 + ((q - 1) & 1) * plane + o, b.c1);
        // plane q - 2: colour 0 sits on x-parity sp
        const int pz = q - 2;
        if constexpr (MODE != MGF_RESTR) {
            MgfVec<V> cn = c.r0;
            mgf_gather(cn, c.c1, edge1, sp, ym, yp, c1d, b.c1);
            mgf_scale(cn, c.l0, lut);
            if (mine && pz >= za && pz < zb) {
                if constexpr (MODE == MGF_POST) {
                    float4 *dst = (float4 *)(A.z + n0 + nxy * pz);
                    MgfVec<V> ev, od;
#pragma unroll
                    for (int t = 0; t < V; t++) {
                        ev.v[t] = sp ? c.c1.v[t] : cn.v[t];
                        od.v[t] = sp ? cn.v[t] : c.c1.v[t];
                    }
#pragma unroll
                    for (int t = 0; t < V; t += 2)
                        __stcg(dst + t / 2, make_float4(ev.v[t], od.v[t], ev.v[t + 1], od.v[t + 1]));
                } else {
                    mgf_stg<V>(A.cout + h0 + hxy * pz, cn);
                }
            }
        } else {
            // sums of the plane before: even rows add their own x-pairs and
            // the next row's, then the two planes of a cell
            const int pl = q - 3;
            if (mine && (j & 1) == 0 && pl >= za && pl < zb + (zb & 1)) {
                MgfVec<V> sum = rs;
                mgf_addv(sum, mgf_lds<V>(sr + (pl & 1) * plane + op));
                if (pl & 1) {
                    const int Y = y >> 1, Z = pl >> 1, I = (x >> 1) + A.cnx * (Y + A.cny * Z);
                    mgf_addv(sum, low);  // (a sum of two: its order does not matter)
                    mgf_stg<V>(A.f1 + I, sum);
                    if (FIRST) {
#pragma unroll
                        for (int t = 0; t < V; t++)
                            if (!(((x >> 1) + t + Y + Z) & 1)) __stcg(A.e1out + I + t, sum.v[t] * __ldg(&A.sig1[I + t].w));
                    }
                } else {
                    low = sum;
                }
            }
            // residuals of plane q - 2: colour 0 against colour 1 and back
            const float *p0 = s0 + (kb == 0 ? N0 - 1 : kb - 1) * plane;
            const int oe0 = sp ? ol : orr;
            const float edge0 = oe0 < 0 ? 0.f : p0[oe0];
            MgfVec<V> a0, a1;
            const bool bulk = (c.l0 | c.l1) == 0;
#pragma unroll
            for (int t = 0; t < V; t++) {
                // (a degree that the compiler does not know, as in the other
                // passes, so that it rounds the product alike)
                const float d0 = bulk ? deg6 : lut.deg[mgf_byte(c.l0, t)], d1 = bulk ? deg6 : lut.deg[mgf_byte(c.l1, t)];
                a0.v[t] = c.r0.v[t] - d0 * c.c0.v[t];
                a1.v[t] = c.r1.v[t] - d1 * c.c1.v[t];
            }
            mgf_gather(a0, c.c1, edge1, sp, ym, yp, c1d, b.c1);
            mgf_gather(a1, c.c0, edge0, !sp, mgf_lds<V>(p0 + om), mgf_lds<V>(p0 + op), c0d, b.c0);
            if ((c.l0 | c.l1) != 0) {
#pragma unroll
                for (int t = 0; t < V; t++) {
                    if (mgf_dead(mgf_byte(c.l0, t))) a0.v[t] = 0.f;
                    if (mgf_dead(mgf_byte(c.l1, t))) a1.v[t] = 0.f;
                }
            }
            rs = a0;
            mgf_addv(rs, a1);  // (the x-pair's sum)
            if (thr) mgf_sts<V>(sr + (pz & 1) * plane + o, rs);
            c0d = c.c0;
        }
        c1d = c.c1;
        k0 = k0 == N0 - 1 ? 0 : k0 + 1;
        __syncthreads();
    };
    for (int q = za - 2; q <= qend; q += 3) {
        step(q, R[0], R[2], R[1]);
        if (q + 1 > qend) break;
        step(q + 1, R[1], R[0], R[2]);
        if (q + 2 > qend) break;
        step(q + 2, R[2], R[1], R[0]);
    }
}

template <int MODE, int V, bool FIRST>
__global__ void __launch_bounds__(MGF_THREADS, 1) mgf_kernel(MgfGeom G, MgfArgs A)
{
    cudaGridDependencySynchronize();
    mgf_body<MODE, V, FIRST>(G, A, blockIdx.x);
}

// one block of a launch over all replicas of a batch
struct MgfBlock {
    int rep, tile;
};

// Partials of r.z after the last smoothing launch, with the thread-to-node
// map and the order of additions of the reducing half sweep it stands in for
// (fine_half<true, .>), so that the CG scalars do not depend on which
// form smoothed: 9 bytes a node more than a reduction inside the launch.
template <typename L>
__device__ __forceinline__ float mgf_dot(const Grid3 &g, const L *__restrict__ link, const float *r, const float *z,
                                         int t0, int nt)
{
    constexpr int U = 4;
    const int hx = g.nx >> 1, np = hx * g.ny * g.nz;
    float rz = 0.f;
    for (int h0 = t0; h0 < np; h0 += U * nt) {
        float2 rv[U], zv[U];
        unsigned mk[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int h = h0 + u * nt;
            mk[u] = MGF_WALLS;
            rv[u] = zv[u] = make_float2(0.f, 0.f);
            if (h >= np) continue;
            rv[u] = __ldcg((const float2 *)r + h);
            zv[u] = __ldcg((const float2 *)z + h);
            mk[u] = __ldg((const unsigned short *)link + h);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int h = h0 + u * nt, row = h / hx, zz = row / g.ny, y = row - zz * g.ny;
            const bool odd = (y + zz) & 1;  // colour 0 is the odd node of the pair
            const unsigned b0 = odd ? mk[u] >> 8 : mk[u] & 0xffu, b1 = odd ? mk[u] & 0xffu : mk[u] >> 8;
            const float r0 = odd ? rv[u].y : rv[u].x, z0 = odd ? zv[u].y : zv[u].x;
            const float r1 = odd ? rv[u].x : rv[u].y, z1 = odd ? zv[u].x : zv[u].y;
            if (!mgf_dead(b0 & 0xffu)) rz += r0 * z0;
            if (!mgf_dead(b1 & 0xffu)) rz += r1 * z1;
        }
    }
    return rz;
}

// Tiles of a lattice: x-rows whole or in segments, the rows and planes of a
// tile (even numbers) and with them the number of blocks, by the least
// estimated time: the waves of resident blocks times the planes a block
// walks (its own and four of halo) and its start-up (about 2000 cycles), a
// step costing the larger of its dependent chain (about 600 cycles) and about
// 105 cycles per resident warp, 120 where rows do not fill whole warps (the
// warps then hold rows of both parities).  False when the rows cannot be
// read in aligned pieces.  share: lattices like this one in the launch; vmax 2:
// pieces of four nodes even where eight would fit.
inline bool mgf_pick(MgfGeom &G, int &V, int nx, int ny, int nz, const int per[3], int num_sms, int share = 1,
                     int vmax = 4)
{
    V = nx % 8 == 0 && vmax == 4 ? 4 : nx % 4 == 0 ? 2 : 0;
    if (V == 0) return false;
    double best = 1e300;
    for (int tx : {nx, 32, 64, 128, 256}) {
        if (tx > nx || tx % (2 * V) || (tx == nx && nx > 1024)) continue;
        const int lpr = tx / (2 * V) + (tx < nx ? 2 : 0), ntx = (nx + tx - 1) / tx;
        for (int oy = 2; lpr * (oy + 4) <= MGF_THREADS; oy += 2) {
            const int rows = oy + 4, nty = (ny + oy - 1) / oy, thr = (lpr * rows + 31) / 32 * 32;
            const size_t smem = 7 * (size_t)lpr * V * rows * sizeof(float) + sizeof(MgfLut) + 1024;
            int bps = (int)((227 * 1024) / smem);
            if (bps > MGF_THREADS / thr) bps = MGF_THREADS / thr;
            if (bps < 1) continue;
            for (int oz = 2; oz <= ((nz + 1) & ~1); oz += 2) {
                const int ntz = (nz + oz - 1) / oz;
                const long long blocks = (long long)ntx * nty * ntz * share;
                const long long waves = (blocks + (long long)num_sms * bps - 1) / ((long long)num_sms * bps);
                const int res = (int)((blocks + num_sms * waves - 1) / (num_sms * waves));  // blocks on an SM at a time
                const double step = (lpr % 32 ? 120.0 : 105.0) * (thr / 32) * (res < bps ? res : bps);
                const double cost = (double)waves * ((oz + 4) * (step > 600.0 ? step : 600.0) + 2000.0);
                if (cost < best) {
                    best = cost;
                    G = MgfGeom{nx, ny, nz, {per[0], per[1], per[2]}, tx, oy, oz, ntx, nty, ntz, lpr, rows};
                }
                if (oy >= ny && oz >= nz) break;
            }
            if (oy >= ny) break;
        }
    }
    return best < 1e300;
}

}  // namespace ekl
