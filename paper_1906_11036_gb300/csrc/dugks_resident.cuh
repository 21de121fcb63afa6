// dugks_resident.cuh -- many DUGKS steps of one D2Q9 grid in one launch, the
// state resident in shared memory (arXiv:1906.11036, Section 2, the step
// summary at the end of the section).
//
// The grid is cut into at most one tile per SM.  A CTA keeps ftilde of its
// tile in shared memory from the first step of a call to the last; per step
// it only exchanges P = fbar^+ (Eq. 2.21) of the tile's rim with the eight
// neighbouring tiles.  What bounds the row-marching step (step_vp,
// fused_step) on such grids is its serial chain: a warp passes 18 rows one
// after another while most SMs hold no warp at all (64^2 in FP64: 12 warps,
// 150 us per step).  Here every SM works on a few cells, so the chain is one
// cell and two faces long, and the launch, the read and the write of the
// state are paid once per call instead of once per step.
//
// Per step:
//   1. each thread forms P, ftilde^+ (Eq. 2.23) and the moments of P of its
//      cells (rim cells first), publishes rim cells, and writes the mirrored
//      ghosts of cells next to a Dirichlet wall;
//   2. the threads of the rim's outer neighbours poll their cells;
//   3. faces: a warp takes 32 consecutive faces of one line and marches with
//      them along the face plane (res_march); neighbouring lanes hold the two
//      faces of a cell, so a cell's flux difference needs one shuffle per
//      crossing pair and no flux array.  The y-faces update
//      ftilde^+ in place; the x-faces leave their flux differences in an
//      array of their own (both directions run at once), which step 1 of the
//      next step adds; where that array does not fit (seq) they update in
//      place after the y-faces.
//
// Exchange: a rim cell's nine values (eight moving P and phi) travel as
// 16-byte words that carry their own step number (three per cell in FP32, six
// in FP64), written and read by single 128-bit accesses, so no fence and no
// separate flag is needed and a message costs one trip through L2.  Two
// buffers alternate between steps: a tile overwrites a word two steps later,
// after it has received the words that its readers published once they had
// read it.  The step number comes from a counter of the CTA in device memory,
// so a launch replayed from a CUDA graph does not meet its own old words.
// All CTAs of a launch must run at once: the launch is cooperative.  Every
// wait is bounded; one that expires sets the error word, which ends every tile
// that waits after that.  Tiles out of its reach may still finish and store
// their cells: the state is then invalid, the step counters differ, and later
// launches return at once.
//
// In FP32 the arithmetic is that of sv_rows operation by operation: a grid
// gives the same bits whether it runs here, in step_vp or in a batch.
#pragma once
#include <type_traits>

#include "dugks_step_vp.cuh"

namespace dugks {

// a pair of FP64 values with the interface of F2
struct D2 {
    double2 v;
};
__device__ __forceinline__ D2 operator+(D2 a, D2 b) { return D2{make_double2(a.v.x + b.v.x, a.v.y + b.v.y)}; }
__device__ __forceinline__ D2 operator-(D2 a, D2 b) { return D2{make_double2(a.v.x - b.v.x, a.v.y - b.v.y)}; }
__device__ __forceinline__ D2 operator*(D2 a, D2 b) { return D2{make_double2(a.v.x * b.v.x, a.v.y * b.v.y)}; }
__device__ __forceinline__ D2 fma2(D2 a, D2 b, D2 c) {
    return D2{make_double2(fma(a.v.x, b.v.x, c.v.x), fma(a.v.y, b.v.y, c.v.y))};
}
__device__ __forceinline__ F2 pk(float a, float b) { return f2(a, b); }
__device__ __forceinline__ D2 pk(double a, double b) { return D2{make_double2(a, b)}; }
template <typename T>
using Pair = typename std::conditional<sizeof(T) == 4, F2, D2>::type;
template <typename T>
using Vec2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
template <typename P>
__device__ __forceinline__ P shfl_next(P x) {
    return pk(__shfl_down_sync(0xffffffffu, x.v.x, 1), __shfl_down_sync(0xffffffffu, x.v.y, 1));
}

template <typename T, int NC>
struct ResConsts {
    Vec2<T> hbp[4][NC];  // per pair: b_bp (feq_PA, feq_PB) in powers of phi
    Vec2<T> hf[4][NC];   // per pair: b_f (feq_PA, feq_PB)
    Vec2<T> fq[4][NC];   // per pair: (feq_PA, feq_PB) (ghosts)
    T a_bp, b_bp, a_f, third, hc;
    T bcv[4];
};

template <typename T>
struct ResArgs {
    const T* fin;            // state [9][ny][pitch] read at the start
    T* fout;                 // state written at the end (may be fin: a CTA touches its own cells only)
    T* rec;                  // if set, the states after steps 1 .. nsteps - 1, rstride elements apart
    long long rstride;
    long long pitch, plane;
    int nx, ny, xper, yper;
    const FaceM<T>*fx, *fy;  // faces -1 .. n+1 at index f + 1
    const CellM<T>*cx, *cy;  // cells -1 .. n at index j + 1
    int ntx, nty, txm, tym;  // tiles per axis and the largest tile
    int nsteps, seq, march;
    uint4* xch;              // [2][tiles][res_slots][words]: published cells
    unsigned* epoch;         // [tiles]: steps done so far
    int* err;
    unsigned long long wait_ns;  // limit of a wait for a neighbour's cell
};

constexpr int kResSrcChunk = 32;  // steps per launch with source terms (their time factors are launch arguments)

template <typename T>
struct ResSrc {
    int nterms, first;
    int dpow[8];
    T db[8];
    T kP_g[Q], kP_f[Q], kU_g[Q], kU_f[Q];  // as in SrcArgs
    const T* field;  // S_k of cell (j, k): field[q * fplane + k * fpitch + j]
    long long fplane, fpitch;
    T* hist;         // phi^{n-1}, read at the start and phi^n written at the end
    long long hpitch;
    T en[kResSrcChunk][8], ep[kResSrcChunk][8];  // exp(rate t_n), exp(rate t_{n-1}) of each step
};

// words of 16 bytes per published cell: nine values and a step number in each word
template <typename T>
constexpr int kResWords = sizeof(T) == 4 ? 3 : 6;

// shared-memory layout, the same on the host and the device
template <typename T>
struct ResLayout {
    int EX, NE, UX, NU;  // row pitches (odd, so that walking along y is free of bank conflicts) and sizes
    size_t oP, oM, oU, oZ, oD, oFx, oFy, oCx, oCy, oI, oS, oH, bytes;
    __host__ __device__ ResLayout(int txm, int tym, int seq, int nsrc) {
        EX = (txm + 2) | 1;
        NE = EX * (tym + 2);
        UX = txm | 1;
        NU = UX * tym;
        size_t o = 0;
        auto take = [&](size_t n) {
            const size_t at = o;
            o += (n + 15) / 16 * 16;
            return at;
        };
        oP = take(size_t(4) * NE * 2 * sizeof(T));       // P pairs
        oU = take(size_t(4) * NU * 2 * sizeof(T));       // ftilde^+ pairs, updated to ftilde
        oD = take(seq ? 0 : size_t(3) * NU * 2 * sizeof(T));  // x-flux differences of pairs 0, 2, 3
        oM = take(size_t(3) * NE * sizeof(T));           // phi, Mx, My of P
        oZ = take(size_t(NU) * sizeof(T));               // rest ftilde
        oFx = take(size_t(11) * (txm + 1) * sizeof(T));   // face weights per x-face / y-face of the tile
        oFy = take(size_t(11) * (tym + 1) * sizeof(T));
        oCx = take(size_t(2) * (txm + 2) * sizeof(T));   // ig and r per column / row, halo included
        oCy = take(size_t(2) * (tym + 2) * sizeof(T));
        oI = take(size_t(txm) * tym * 4);                // the cells in processing order
        oS = take(size_t(nsrc) * NU * sizeof(T));        // source fields
        oH = take(nsrc ? size_t(NU) * sizeof(T) : 0);    // phi^{n-1}
        bytes = o;
    }
};

// first column (row) of tile b when n columns are cut into nt nearly equal tiles
__host__ __device__ inline int res_cut(int b, int n, int nt) { return int((long long)b * n / nt); }

// published cells of a tile: its rim, then the ghosts of its corner cells (two per wall side),
// which the tiles beside it need for the slopes of their halo cells
__host__ __device__ inline int res_slots(int txm, int tym) { return 2 * (txm + tym) + 8; }

__device__ __forceinline__ void st_word(uint4* p, unsigned a, unsigned b, unsigned c, unsigned d) {
    const unsigned long long lo = a | ((unsigned long long)b << 32), hi = c | ((unsigned long long)d << 32);
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}
__device__ __forceinline__ uint4 ld_word(const uint4* p) {
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_uint4(unsigned(lo), unsigned(lo >> 32), unsigned(hi), unsigned(hi >> 32));
}

// nine values of a rim cell -> its words
__device__ __forceinline__ void res_publish(uint4* p, const F2 (&P)[4], float phi, unsigned tag) {
    auto u = [](float x) { return __float_as_uint(x); };
    st_word(p, u(P[0].v.x), u(P[0].v.y), u(P[1].v.x), tag);
    st_word(p + 1, u(P[1].v.y), u(P[2].v.x), u(P[2].v.y), tag);
    st_word(p + 2, u(P[3].v.x), u(P[3].v.y), u(phi), tag);
}
__device__ __forceinline__ void res_publish(uint4* p, const D2 (&P)[4], double phi, unsigned tag) {
    const double v[9] = {P[0].v.x, P[0].v.y, P[1].v.x, P[1].v.y, P[2].v.x, P[2].v.y, P[3].v.x, P[3].v.y, phi};
    unsigned w[18];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        w[2 * i] = unsigned(__double2loint(v[i]));
        w[2 * i + 1] = unsigned(__double2hiint(v[i]));
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) st_word(p + i, w[3 * i], w[3 * i + 1], w[3 * i + 2], tag);
}
__device__ __forceinline__ bool res_receive(const uint4* p, F2 (&P)[4], float& phi, unsigned tag) {
    const uint4 a = ld_word(p), b = ld_word(p + 1), c = ld_word(p + 2);
    if (a.w != tag || b.w != tag || c.w != tag) return false;
    auto g = [](unsigned x) { return __uint_as_float(x); };
    P[0] = f2(g(a.x), g(a.y));
    P[1] = f2(g(a.z), g(b.x));
    P[2] = f2(g(b.y), g(b.z));
    P[3] = f2(g(c.x), g(c.y));
    phi = g(c.z);
    return true;
}
__device__ __forceinline__ bool res_receive(const uint4* p, D2 (&P)[4], double& phi, unsigned tag) {
    unsigned w[18];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const uint4 a = ld_word(p + i);
        ok = ok && a.w == tag;
        w[3 * i] = a.x;
        w[3 * i + 1] = a.y;
        w[3 * i + 2] = a.z;
    }
    if (!ok) return false;
    double v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = __hiloint2double(int(w[2 * i + 1]), int(w[2 * i]));
#pragma unroll
    for (int q = 0; q < 4; ++q) P[q] = pk(v[2 * q], v[2 * q + 1]);
    phi = v[8];
    return true;
}

template <typename T, int NC>
__device__ __forceinline__ Pair<T> res_poly(const Vec2<T> (&c)[NC], Pair<T> x) {
    Pair<T> s{c[NC - 1]};
#pragma unroll
    for (int m = NC - 2; m >= 0; --m) s = fma2(s, x, Pair<T>{c[m]});
    return s;
}

// Mx, My of P (as sv_moments)
template <typename PT, typename T>
__device__ __forceinline__ void res_moments(const PT (&P)[4], T& mx, T& my) {
    const T d0 = P[0].v.x - P[0].v.y, d1 = P[1].v.x - P[1].v.y, d2 = P[2].v.x - P[2].v.y, d3 = P[3].v.x - P[3].v.y;
    mx = (d0 + d2) - d3;
    my = (d1 + d2) + d3;
}

// weights of a face in shared memory: normal weights of the left and of the right cell for a pair
// that moves along the normal (4), 1 - w, w, hcd, hc tl, hc tr; in FP64 the first four and a second
// pair of tangential weights carry the factor a_f of Eq. 2.22 (one multiplication less per value)
// faces of a march unrolled: 2 (us per step: 512^2 FP32 6.25, 330x517 with walls 4.84, 400^2 4.64) against
// 1 (6.35, 4.88, 4.56)
constexpr int kResUnroll = 2;
template <typename T>
constexpr int kResFace = sizeof(T) == 4 ? 9 : 11;

// m faces one after another along their own plane, from the face whose left (lower) cell is at e0:
// the original f (Eq. 2.22) of the three pairs that cross each (x-faces: 0, 2, 3; y-faces: 1, 2, 3),
// handed to put(t, f).  sn: stride from the left to the right cell; st: stride along the march;
// lim: cells up to the end of the tile (positions beyond it are read again and not used); w: the
// face weights, the same along the march; ig: central-difference factors along it, two apart.
// A march keeps three positions of the two cells' slope pairs in registers, so a face costs 6 pair
// loads and 6 moments instead of 14 and 8: in FP32 the shared-memory pipe bounds the large tiles.
template <typename T, int NC, bool YF, typename Put>
__device__ __forceinline__ void res_march(const ResConsts<T, NC>& k, const Pair<T>* __restrict__ sP,
                                          const T* __restrict__ sM, const int NE, const int e0, const int sn,
                                          const int st, const T* __restrict__ w, const T* __restrict__ ig, const int m,
                                          const int lim, Put&& put) {
    using PT = Pair<T>;
    constexpr bool F32 = sizeof(T) == 4;
    const PT lp = pk(w[0], w[1]), rp = pk(w[2], w[3]);
    const T l0 = w[4], r0 = w[5], hcd = w[6], gl = w[7], gr = w[8];
    T fl = T(0), fr = T(0);
    if constexpr (!F32) {
        fl = w[9];
        fr = w[10];
    }
    // pair 3 = (6, 8): e = (-1, 1): its normal weights are swapped at x-faces, the sign of its
    // tangential component at y-faces (folded into the order of the difference)
    const PT lp3 = YF ? lp : pk(w[1], w[0]), rp3 = YF ? rp : pk(w[3], w[2]);
    const T* Mn = sM + (YF ? 2 : 1) * NE;  // normal moment
    const T* Mt = sM + (YF ? 1 : 2) * NE;  // tangential moment
    const PT *p0 = sP + (YF ? 1 : 0) * NE, *p2 = sP + 2 * NE, *p3 = sP + 3 * NE;
    // positions t - 1 and t of the march, left and right cell
    PT a2L = p2[e0 - st], a2R = p2[e0 - st + sn], a3L = p3[e0 - st], a3R = p3[e0 - st + sn];
    PT b2L = p2[e0], b2R = p2[e0 + sn], b3L = p3[e0], b3R = p3[e0 + sn];
    T amL = Mt[e0 - st], amR = Mt[e0 - st + sn], bmL = Mt[e0], bmR = Mt[e0 + sn];
    const int mw = __reduce_max_sync(0xffffffffu, min(m, lim));  // blocks at the end of the tile are shorter
#pragma unroll kResUnroll
    for (int t = 0; t < mw; ++t) {
        const int e = e0 + min(t, lim - 1) * st, en = e0 + min(t + 1, lim) * st;
        const PT c2L = p2[en], c2R = p2[en + sn], c3L = p3[en], c3R = p3[en + sn];
        const T cmL = Mt[en], cmR = Mt[en + sn];
        const T g = ig[2 * min(t, lim - 1)];
        const PT d3L = YF ? a3L - c3L : c3L - a3L, d3R = YF ? a3R - c3R : c3R - a3R;
        PT f[3];
        if constexpr (F32) {
            // phi_b from the moments of the two cells
            const T gmL = (cmL - amL) * g, gmR = (cmR - amR) * g;
            const T pb = fma(l0, sM[e], fma(hcd, Mn[e], -gl * gmL)) + fma(r0, sM[e + sn], fma(-hcd, Mn[e + sn], -gr * gmR));
            const PT pb2 = pk(pb, pb), af = pk(k.a_f, k.a_f), g2 = pk(g, g), tl = pk(-gl, gl), tr = pk(-gr, gr);
            const PT L0 = lp * p0[e];
            const PT L2 = fma2(tl, (c2L - a2L) * g2, lp * b2L), L3 = fma2(tl, d3L * g2, lp3 * b3L);
            PT v0, v2, v3;
            if constexpr (YF) {
                v0 = fma2(rp, p0[e + sn], L0);
                v2 = fma2(tr, (c2R - a2R) * g2, fma2(rp, b2R, L2));
                v3 = fma2(tr, d3R * g2, fma2(rp3, b3R, L3));
            } else {
                v0 = L0 + rp * p0[e + sn];
                v2 = L2 + fma2(tr, (c2R - a2R) * g2, rp * b2R);
                v3 = L3 + fma2(tr, d3R * g2, rp3 * b3R);
            }
            f[0] = fma2(af, v0, res_poly<T, NC>(k.hf[YF ? 1 : 0], pb2));
            f[1] = fma2(af, v2, res_poly<T, NC>(k.hf[2], pb2));
            f[2] = fma2(af, v3, res_poly<T, NC>(k.hf[3], pb2));
        } else {
            T pb = fma(l0, sM[e], r0 * sM[e + sn]);
            pb = fma(hcd, Mn[e] - Mn[e + sn], pb);
            pb = fma(-(gl * g), cmL - amL, pb);
            pb = fma(-(gr * g), cmR - amR, pb);
            const PT pb2 = pk(pb, pb);
            const T hl = fl * g, hr = fr * g;
            const PT tl = pk(-hl, hl), tr = pk(-hr, hr);
            f[0] = fma2(rp, p0[e + sn], fma2(lp, p0[e], res_poly<T, NC>(k.hf[YF ? 1 : 0], pb2)));
            f[1] = fma2(rp, b2R, fma2(lp, b2L, res_poly<T, NC>(k.hf[2], pb2)));
            f[1] = fma2(tr, c2R - a2R, fma2(tl, c2L - a2L, f[1]));
            f[2] = fma2(rp3, b3R, fma2(lp3, b3L, res_poly<T, NC>(k.hf[3], pb2)));
            f[2] = fma2(tr, d3R, fma2(tl, d3L, f[2]));
        }
        put(t, f);
        a2L = b2L; a2R = b2R; a3L = b3L; a3R = b3R;
        b2L = c2L; b2R = c2R; b3L = c3L; b3R = c3R;
        amL = bmL; amR = bmR;
        bmL = cmL; bmR = cmR;
    }
}

// Step 1 of one tile of at most 32 cells in FP64: warps 0 .. 3 take eight cells each (c: this lane's
// cell, bit 31 set where it has one), lane group q = lane / 8 the pair q; sums over the pairs go
// through shuffles.  The FP64 pipe of a quarter of an SM takes 64 clocks for an instruction of a warp
// whatever its active lanes, so one warp alone needs about 75 x 64 clocks for its cells while the
// other three quarters idle; split, each quarter runs about 28 (64^2: 5.9 -> 4.7 us per step).
// hq: the lane's pair of hbp; no source terms, no wall cells.
template <typename T, int NC, typename Slot>
__device__ __forceinline__ void res_cell_parts(const ResArgs<T>& a, const ResConsts<T, NC>& k, const Vec2<T>* hq, Pair<T>* sP,
                                               T* sM, Pair<T>* sU, T* sZ, const Pair<T>* sD, const T* sCx, unsigned c,
                                               int NE, int NU, int EX, int UX, int lane, int warp, int step, int x0, int y0,
                                               Slot&& slot, unsigned tag) {
    if constexpr (sizeof(T) == 8 && NC <= 4) {
        using PT = Pair<T>;
        if (warp >= 4) return;
        const int q = lane >> 3, lx = int(c & 0xfffu), ly = int(c >> 12 & 0xfffu);
        const int u = ly * UX + lx, e = (ly + 1) * EX + lx + 1;
        const bool live = c >> 31;
        auto over_pairs = [&](T x) {
            x += __shfl_xor_sync(0xffffffffu, x, 8);
            return x + __shfl_xor_sync(0xffffffffu, x, 16);
        };
        PT F = sU[q * NU + u];
        if (!a.seq) {  // the x-fluxes of the step before (pair 1 has none)
            const T r = sCx[2 * (lx + 1) + 1], rx = q == 1 ? T(0) : (q == 3 ? -r : r);
            F = fma2(pk(-rx, rx), sD[max(q - 1, 0) * NU + u], F);
        }
        const T Fz = sZ[u];
        if (a.rec && step > 0 && live) {
            T* dst = a.rec + (step - 1) * a.rstride + (long long)(y0 + ly) * a.pitch + x0 + lx;
            if (q == 0) dst[0] = Fz;
            const int pa = q == 0 ? PA(0) : q == 1 ? PA(1) : q == 2 ? PA(2) : PA(3);
            const int pb = q == 0 ? PB(0) : q == 1 ? PB(1) : q == 2 ? PB(2) : PB(3);
            dst[pa * a.plane] = F.v.x;
            dst[pb * a.plane] = F.v.y;
        }
        const T phi = Fz + over_pairs(F.v.x + F.v.y);
        PT h{hq[NC - 1]};
#pragma unroll
        for (int m = NC - 2; m >= 0; --m) h = fma2(h, pk(phi, phi), PT{hq[m]});
        const PT P = fma2(pk(k.a_bp, k.a_bp), F, h);
        if (live) sP[q * NE + e] = P;
        if (live && q == 0) sM[e] = phi;
        __syncwarp();
        // the words of the eight cells, six each, as 32-bit halves of the values just stored
        for (int i = lane; i < 48; i += 32) {
            const unsigned oc = __shfl_sync(i < 32 ? 0xffffffffu : 0x0000ffffu, c, i / 6);
            if (!(oc >> 31) || !(oc >> 24 & 1u)) continue;
            const int olx = int(oc & 0xfffu), oly = int(oc >> 12 & 0xfffu), oe = (oly + 1) * EX + olx + 1, w = i % 6;
            unsigned v[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const int half = 3 * w + m, d = half >> 1;  // value d: pair d / 2, component d % 2; 8: phi
                const unsigned* src = d < 8 ? reinterpret_cast<const unsigned*>(sP + (d >> 1) * NE + oe) + 2 * (d & 1)
                                            : reinterpret_cast<const unsigned*>(sM + oe);
                v[m] = src[half & 1];
            }
            st_word(slot(olx, oly) + w, v[0], v[1], v[2], tag);
        }
        const T Pz = fma(k.a_bp, Fz, fma(k.b_bp, phi, -over_pairs(h.v.x + h.v.y)));
        const T d = P.v.x - P.v.y;
        const T mx = over_pairs(q == 1 ? T(0) : (q == 3 ? -d : d)), my = over_pairs(q == 0 ? T(0) : d);
        if (live) {
            sU[q * NU + u] = fma2(pk(k.third, k.third), P - F, P);
            if (q == 0) {
                sM[NE + e] = mx;
                sM[2 * NE + e] = my;
                sZ[u] = fma(k.third, Pz - Fz, Pz);
            }
        }
    }
}

// threads per CTA at most.  FP32: 512 at 128 registers (us per step at 70x45, 400^2, 512^2: 1.83, 4.64, 6.25;
// 384 1.72, 4.44, 7.08; 640 at 96 registers 1.97, 5.43, 8.86; 768 at 80 2.34, 6.54, 11.4).  FP64: 256, eight
// warps keep its pipe busy.
template <typename T>
constexpr int kResThreads = sizeof(T) == 4 ? 512 : 256;

template <typename T, int NC, bool SRC>
__global__ void __launch_bounds__(kResThreads<T>, 1)
    resident_steps(const __grid_constant__ ResArgs<T> a, const __grid_constant__ ResConsts<T, NC> k,
                   const __grid_constant__ ResSrc<T> sa) {
    using PT = Pair<T>;
    constexpr int W = kResWords<T>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = NT >> 5;
    const int bx = blockIdx.x % a.ntx, by = blockIdx.x / a.ntx;
    const int x0 = res_cut(bx, a.nx, a.ntx), tx = res_cut(bx + 1, a.nx, a.ntx) - x0;
    const int y0 = res_cut(by, a.ny, a.nty), ty = res_cut(by + 1, a.ny, a.nty) - y0;
    const ResLayout<T> L(a.txm, a.tym, a.seq, SRC ? sa.nterms : 0);
    const int EX = L.EX, NE = L.NE, UX = L.UX, NU = L.NU;
    PT* sP = reinterpret_cast<PT*>(smem_raw + L.oP);
    PT* sU = reinterpret_cast<PT*>(smem_raw + L.oU);
    PT* sD = reinterpret_cast<PT*>(smem_raw + L.oD);
    T* sM = reinterpret_cast<T*>(smem_raw + L.oM);
    T* sZ = reinterpret_cast<T*>(smem_raw + L.oZ);
    T* sFx = reinterpret_cast<T*>(smem_raw + L.oFx);
    T* sFy = reinterpret_cast<T*>(smem_raw + L.oFy);
    T* sCx = reinterpret_cast<T*>(smem_raw + L.oCx);
    T* sCy = reinterpret_cast<T*>(smem_raw + L.oCy);
    unsigned* sI = reinterpret_cast<unsigned*>(smem_raw + L.oI);
    T* sS = reinterpret_cast<T*>(smem_raw + L.oS);
    T* sH = reinterpret_cast<T*>(smem_raw + L.oH);

    // a wait that expired in an earlier launch: the state is not advanced any further
    if (__syncthreads_or(tid == 0 && (*reinterpret_cast<volatile int*>(a.err) & 1))) return;
    const unsigned tag0 = *reinterpret_cast<volatile unsigned*>(a.epoch + blockIdx.x);

    // cells of the tile in the order they are processed: the rim first (its P is what the
    // neighbours wait for), then the interior
    const int ncell = tx * ty;
    const bool thin = tx <= 2 || ty <= 2;  // every cell is on the rim
    const int nrim = thin ? ncell : 2 * tx + 2 * (ty - 2);
    auto cell_of = [&](int i, int& lx, int& ly) {
        if (thin) {
            ly = i / tx;
            lx = i - ly * tx;
        } else if (i < 2 * tx) {
            ly = i < tx ? 0 : ty - 1;
            lx = i < tx ? i : i - tx;
        } else if (i < nrim) {
            const int r = i - 2 * tx;
            ly = 1 + (r >> 1);
            lx = (r & 1) ? tx - 1 : 0;
        } else {
            const int r = i - nrim, w = tx - 2, qq = r / w;
            ly = 1 + qq;
            lx = 1 + r - qq * w;
        }
    };
    // slot of a rim cell in its tile's published cells
    auto slot_of = [&](int lx, int ly, int tw, int th) {
        if (ly == 0) return lx;
        if (ly == th - 1) return a.txm + lx;
        return 2 * a.txm + (lx == 0 ? ly : a.tym + ly);
    };
    const int nslots = res_slots(a.txm, a.tym), gslot = nslots - 8;
    const size_t xbuf = size_t(a.ntx) * a.nty * nslots * W;  // words of one of the two buffers
    uint4* own = a.xch + size_t(blockIdx.x) * nslots * W;

    // this thread's halo cell (one outer neighbour of the rim), taken from the last threads on
    const int h = NT - 1 - tid;
    const uint4* hsrc = nullptr;
    int he = 0;
    if (h < 2 * (tx + 2) + 2 * ty) {
        int lx, ly;
        if (h < 2 * (tx + 2)) {
            ly = h < tx + 2 ? -1 : ty;
            lx = (h < tx + 2 ? h : h - (tx + 2)) - 1;
        } else {
            const int r = h - 2 * (tx + 2);
            ly = r < ty ? r : r - ty;
            lx = r < ty ? -1 : tx;
        }
        he = (ly + 1) * EX + lx + 1;
        int gx = x0 + lx, gy = y0 + ly;
        const bool wx = !a.xper && (gx < 0 || gx >= a.nx), wy = !a.yper && (gy < 0 || gy >= a.ny);
        // beyond a wall: the ghost of a cell of this tile is written by that cell, the one of a
        // neighbouring tile's corner cell is received, a corner ghost is never used
        const bool take = wx ? (!wy && (ly < 0 || ly >= ty)) : (!wy || lx < 0 || lx >= tx);
        if (take) {
            int ox = bx, oy = by;
            if (!wx && lx < 0) ox = bx == 0 ? a.ntx - 1 : bx - 1;
            if (!wx && lx >= tx) ox = bx == a.ntx - 1 ? 0 : bx + 1;
            if (!wy && ly < 0) oy = by == 0 ? a.nty - 1 : by - 1;
            if (!wy && ly >= ty) oy = by == a.nty - 1 ? 0 : by + 1;
            int s;
            if (wx) {
                s = gslot + 4 + (gx < 0 ? 0 : 2) + (ly < 0 ? 1 : 0);  // W, E: the ghost of its last / first row
            } else if (wy) {
                s = gslot + (gy < 0 ? 0 : 2) + (lx < 0 ? 1 : 0);  // S, N: the ghost of its last / first column
            } else {
                gx = gx < 0 ? gx + a.nx : (gx >= a.nx ? gx - a.nx : gx);
                gy = gy < 0 ? gy + a.ny : (gy >= a.ny ? gy - a.ny : gy);
                const int qx = res_cut(ox, a.nx, a.ntx), qy = res_cut(oy, a.ny, a.nty);
                s = slot_of(gx - qx, gy - qy, res_cut(ox + 1, a.nx, a.ntx) - qx, res_cut(oy + 1, a.ny, a.nty) - qy);
            }
            hsrc = a.xch + (size_t(oy * a.ntx + ox) * nslots + s) * W;
        }
    }

    // weights of the tile's faces and cells; everything else of the P planes starts at zero
    // (corner ghosts are never written and only met by zero weights)
    constexpr int FW = kResFace<T>;
    auto face_row = [&](T* d, const FaceM<T>& m) {
        const T u = T(1) - m.w, s = sizeof(T) == 4 ? T(1) : k.a_f;
        d[0] = s * (u + m.hcd);
        d[1] = s * (u - m.hcd);
        d[2] = s * (m.w - m.hcd);
        d[3] = s * (m.w + m.hcd);
        d[4] = u;
        d[5] = m.w;
        d[6] = m.hcd;
        d[7] = k.hc * m.tl;
        d[8] = k.hc * m.tr;
        if (FW > 9) {
            d[FW - 2] = s * d[7];
            d[FW - 1] = s * d[8];
        }
    };
    for (int i = tid; i <= tx; i += NT) face_row(sFx + FW * i, a.fx[x0 + i + 1]);
    for (int i = tid; i <= ty; i += NT) face_row(sFy + FW * i, a.fy[y0 + i + 1]);
    for (int i = tid; i < tx + 2; i += NT) {
        const CellM<T> m = a.cx[min(x0 + i, a.nx + 1)];  // column x0 - 1 + i
        sCx[2 * i] = m.ig;
        sCx[2 * i + 1] = m.r;
    }
    for (int i = tid; i < ty + 2; i += NT) {
        const CellM<T> m = a.cy[min(y0 + i, a.ny + 1)];
        sCy[2 * i] = m.ig;
        sCy[2 * i + 1] = m.r;
    }
    // column, row and flags of each cell: 1 << 24 on the rim, 1 << (25 + side) at a wall (W, E, S, N)
    for (int i = tid; i < ncell; i += NT) {
        int lx, ly;
        cell_of(i, lx, ly);
        unsigned c = unsigned(lx) | unsigned(ly) << 12;
        if (i < nrim) c |= 1u << 24;
        if (!a.xper) c |= (x0 + lx == 0 ? 1u << 25 : 0u) | (x0 + lx == a.nx - 1 ? 1u << 26 : 0u);
        if (!a.yper) c |= (y0 + ly == 0 ? 1u << 27 : 0u) | (y0 + ly == a.ny - 1 ? 1u << 28 : 0u);
        sI[i] = c;
    }
    for (int i = tid; i < 4 * NE; i += NT) sP[i] = pk(T(0), T(0));
    for (int i = tid; i < 3 * NE; i += NT) sM[i] = T(0);
    for (int i = tid; i < ncell; i += NT) {
        const int ly = i / tx, lx = i - ly * tx, u = ly * UX + lx;
        const T* src = a.fin + (long long)(y0 + ly) * a.pitch + x0 + lx;
#pragma unroll
        for (int q = 0; q < 4; ++q) sU[q * NU + u] = pk(src[PA(q) * a.plane], src[PB(q) * a.plane]);
        sZ[u] = src[0];
        if (!a.seq)
#pragma unroll
            for (int s = 0; s < 3; ++s) sD[s * NU + u] = pk(T(0), T(0));
        if (SRC) {
            for (int q = 0; q < sa.nterms; ++q)
                sS[q * NU + u] = sa.field[q * sa.fplane + (long long)(y0 + ly) * sa.fpitch + x0 + lx];
            sH[u] = sa.hist[(long long)(y0 + ly) * sa.hpitch + x0 + lx];
        }
    }
    __syncthreads();

    // ftilde of cell u (column lx): ftilde^+ with the y-fluxes, plus the x-fluxes not yet added
    auto state_of = [&](int u, int lx, PT (&F)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] = sU[q * NU + u];
        if (!a.seq) {
            const T rx = sCx[2 * (lx + 1) + 1];
            F[0] = fma2(pk(-rx, rx), sD[u], F[0]);
            F[2] = fma2(pk(-rx, rx), sD[NU + u], F[2]);
            F[3] = fma2(pk(rx, -rx), sD[2 * NU + u], F[3]);
        }
    };

    // marches: lines of tx + 1 (ty + 1) faces, one per block of `march` rows (columns)
    const int M = a.march;
    const int nxm = (tx + 1) * ((ty + M - 1) / M), nym = (ty + 1) * ((tx + M - 1) / M);
    const int gxn = (nxm - 2) / 31 + 1, gyn = (nym - 2) / 31 + 1;  // groups of 32 (each shares its last one)
    const unsigned mx_div = 0xffffffffu / unsigned(tx + 1) + 1u, my_div = 0xffffffffu / unsigned(ty + 1) + 1u;
    // a lane's march of group g (y-faces first): the tile's face line and the block along it
    struct March {
        int e0, f, r0, lim;
        bool live;
    };
    auto march_of = [&](int g) {
        const bool y = g < gyn;
        const int it0 = (y ? g : g - gyn) * 31 + lane, nm = y ? nym : nxm, line = y ? ty + 1 : tx + 1;
        const int it = min(it0, nm - 1), blk = int(__umulhi(unsigned(it), y ? my_div : mx_div));
        March m;
        m.f = it - blk * line;  // below row f / west of column f
        m.r0 = blk * M;
        m.e0 = y ? m.f * EX + m.r0 + 1 : (m.r0 + 1) * EX + m.f;
        m.lim = (y ? tx : ty) - m.r0;
        m.live = lane < 31 && it0 < nm && m.f < line - 1;
        return m;
    };
    // x-faces: flux differences into sD, or (seq) straight into the state
    auto x_group = [&](const March& m) {
        res_march<T, NC, false>(k, sP, sM, NE, m.e0, 1, EX, sFx + FW * m.f, sCy + 2 * (m.r0 + 1), M, m.lim,
                                [&](int t, const PT (&fl)[3]) {
            const PT d0 = shfl_next(fl[0]) - fl[0], d1 = shfl_next(fl[1]) - fl[1], d2 = shfl_next(fl[2]) - fl[2];
            if (m.live && t < m.lim) {
                const int u = (m.r0 + t) * UX + m.f;
                if (a.seq) {
                    const T rx = sCx[2 * (m.f + 1) + 1];
                    sU[u] = fma2(pk(-rx, rx), d0, sU[u]);
                    sU[2 * NU + u] = fma2(pk(-rx, rx), d1, sU[2 * NU + u]);
                    sU[3 * NU + u] = fma2(pk(rx, -rx), d2, sU[3 * NU + u]);
                } else {
                    sD[u] = d0;
                    sD[NU + u] = d1;
                    sD[2 * NU + u] = d2;
                }
            }
        });
    };
    auto y_group = [&](const March& m) {
        const T r = sCy[2 * (min(m.f, ty - 1) + 1) + 1];
        const PT rp = pk(r, -r), rn = pk(-r, r);
        res_march<T, NC, true>(k, sP, sM, NE, m.e0, EX, 1, sFy + FW * m.f, sCx + 2 * (m.r0 + 1), M, m.lim,
                               [&](int t, const PT (&fl)[3]) {
            const PT n0 = shfl_next(fl[0]), n1 = shfl_next(fl[1]), n2 = shfl_next(fl[2]);
            if (m.live && t < m.lim) {
                PT* U = sU + m.f * UX + m.r0 + t;
                U[NU] = fma2(rn, n0, fma2(rp, fl[0], U[NU]));
                U[2 * NU] = fma2(rn, n1, fma2(rp, fl[1], U[2 * NU]));
                U[3 * NU] = fma2(rn, n2, fma2(rp, fl[2], U[3 * NU]));
            }
        });
    };
    // most tiles give a warp one group and a thread one cell: these are worked out once
    const March m_first = march_of(min(warp, gyn + gxn - 1)), mx_first = march_of(gyn + min(warp, gxn - 1));
    const unsigned c_first = tid < ncell ? sI[tid] : 0u;
    // FP64 tiles of one warp's cells: four warps take eight cells each, a lane per pair
    constexpr bool kSplit = sizeof(T) == 8 && NC <= 4 && !SRC;
    const bool split = kSplit && ncell <= 32 && nwarps >= 4 && !__syncthreads_or(tid < ncell && (c_first >> 25));
    const int i_split = warp * 8 + (lane & 7);
    const unsigned c_split = split && warp < 4 && i_split < ncell ? sI[i_split] | 1u << 31 : 0u;
    Vec2<T> hq[kSplit ? NC : 1];
    if constexpr (kSplit)
#pragma unroll
        for (int m = 0; m < NC; ++m) hq[m] = k.hbp[lane >> 3][m];
    bool fail = false;
    for (int step = 0; step < a.nsteps; ++step) {
        const unsigned tag = tag0 + unsigned(step) + 1u;
        uint4* pub = own + (tag & 1u) * xbuf;
        if (split) {
            res_cell_parts<T, NC>(a, k, hq, sP, sM, sU, sZ, sD, sCx, c_split, NE, NU, EX, UX, lane, warp, step, x0, y0,
                                  [&](int lx, int ly) { return pub + slot_of(lx, ly, tx, ty) * W; }, tag);
        }
        unsigned c = c_first;
        for (int i = split ? ncell : tid; i < ncell; i += NT) {
            if (i != tid) c = sI[i];
            const int lx = int(c & 0xfffu), ly = int(c >> 12 & 0xfffu);
            const int u = ly * UX + lx, e = (ly + 1) * EX + lx + 1;
            PT F[4], P[4], U[4];
            state_of(u, lx, F);
            const T Fz = sZ[u];
            if (a.rec && step > 0) {
                T* dst = a.rec + (step - 1) * a.rstride + (long long)(y0 + ly) * a.pitch + x0 + lx;
                dst[0] = Fz;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    dst[PA(q) * a.plane] = F[q].v.x;
                    dst[PB(q) * a.plane] = F[q].v.y;
                }
            }
            // P (Eq. 2.21), ftilde^+ (Eq. 2.23), as sv_cell
            const PT s4 = (F[0] + F[1]) + (F[2] + F[3]);
            const T phi = Fz + (s4.v.x + s4.v.y);
            const PT x2 = pk(phi, phi), abp = pk(k.a_bp, k.a_bp), th = pk(k.third, k.third);
            PT hs = pk(T(0), T(0));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const PT hq = res_poly<T, NC>(k.hbp[q], x2);
                P[q] = fma2(abp, F[q], hq);
                hs = hs + hq;
            }
            T Pz = fma(k.a_bp, Fz, fma(k.b_bp, phi, -(hs.v.x + hs.v.y)));
            T m0 = phi, Uz;
            auto relaxed = [&]() {  // ftilde^+ (Eq. 2.23)
#pragma unroll
                for (int q = 0; q < 4; ++q) U[q] = fma2(th, P[q] - F[q], P[q]);
                Uz = fma(k.third, Pz - Fz, Pz);
            };
            // the neighbours' P leaves before ftilde^+ is formed: their waits end earlier (not with source
            // terms, which enter both, nor at high degree, where the longer lives of P and F spill)
            constexpr bool kEarly = !SRC && NC <= 4;
            if constexpr (!kEarly) relaxed();
            if constexpr (SRC) {  // the source terms (as add_source_vp), phi^{n-1} kept in shared memory
                const bool first = sa.first && step == 0;
                const PT X = pk(phi, first ? phi : sH[u]);
                sH[u] = phi;
                PT pw = pk(T(1), T(1)), Fs = pk(T(0), T(0));
                for (int q = 0; q < sa.nterms; ++q) {
                    for (int m = 0; m < sa.dpow[q]; ++m) pw = pw * X;
                    const T S = sS[q * NU + u];
                    Fs = fma2(pk(sa.en[step][q], sa.ep[step][q]) * pk(S, S), pw, Fs);
                }
                PT d = pk(T(0), T(0));
#pragma unroll
                for (int m = (NC < 9 ? NC - 2 : 7); m >= 0; --m) d = fma2(d, X, pk(sa.db[m], sa.db[m]));
                const PT G = d * Fs;
                const T Ft = fma(T(0.25), Fs.v.x - Fs.v.y, Fs.v.x), gt = fma(T(0.25), G.v.x - G.v.y, G.v.x);
                const T Fa = fma(T(0.5), Fs.v.x - Fs.v.y, Fs.v.x), ga = fma(T(0.5), G.v.x - G.v.y, G.v.x);
                const T p1 = sa.kP_f[1] * Ft, p2 = sa.kP_f[5] * Ft, u1 = sa.kU_f[1] * Fa, u2 = sa.kU_f[5] * Fa;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const T pq = q < 2 ? p1 : p2, uq = q < 2 ? u1 : u2;
                    P[q] = P[q] + fma2(pk(sa.kP_g[PA(q)], sa.kP_g[PB(q)]), pk(gt, gt), pk(pq, pq));
                    U[q] = U[q] + fma2(pk(sa.kU_g[PA(q)], sa.kU_g[PB(q)]), pk(ga, ga), pk(uq, uq));
                }
                Pz = fma(sa.kP_f[0], Ft, Pz);
                Uz = fma(sa.kU_f[0], Fa, Uz);
                const PT p4 = (P[0] + P[1]) + (P[2] + P[3]);
                m0 = Pz + (p4.v.x + p4.v.y);
            }
            if (c & 1u << 24) res_publish(pub + slot_of(lx, ly, tx, ty) * W, P, m0, tag);
            if constexpr (kEarly) relaxed();
            T mx, my;
            res_moments(P, mx, my);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                sP[q * NE + e] = P[q];
                sU[q * NU + u] = U[q];
            }
            sM[e] = m0;
            sM[NE + e] = mx;
            sM[2 * NE + e] = my;
            sZ[u] = Uz;
            // mirrored ghosts beyond Dirichlet walls (non-equilibrium extrapolation, as sv_ghost)
            if (c >> 25)
#pragma unroll 1
                for (int side = 0; side < 4; ++side) {
                    if (!(c >> (25 + side) & 1u)) continue;
                    const int eg = e + (side == 0 ? -1 : side == 1 ? 1 : side == 2 ? -EX : EX);
                    const T phig = T(2) * k.bcv[side] - phi;
                    const PT xg = pk(phig, phig);
                    PT Pg[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        Pg[q] = P[q] + (res_poly<T, NC>(k.fq[q], xg) - res_poly<T, NC>(k.fq[q], x2));
                    T gx, gy;
                    res_moments(Pg, gx, gy);
#pragma unroll
                    for (int q = 0; q < 4; ++q) sP[q * NE + eg] = Pg[q];
                    const T mg = SRC ? m0 + (phig - phi) : phig;
                    sM[eg] = mg;
                    sM[NE + eg] = gx;
                    sM[2 * NE + eg] = gy;
                    // the tiles beside need the ghosts of this tile's corner cells
                    const bool lo = side < 2 ? ly == 0 : lx == 0, hi = side < 2 ? ly == ty - 1 : lx == tx - 1;
                    uint4* gp = pub + (gslot + (side < 2 ? 4 + 2 * side : 2 * (side - 2))) * W;
                    if (lo) res_publish(gp, Pg, mg, tag);
                    if (hi) res_publish(gp + W, Pg, mg, tag);
                }
        }
        // the halo cell of this thread, once its owner has published it
        if (hsrc) {
            const uint4* p = hsrc + (tag & 1u) * xbuf;
            PT P[4];
            T phi;
            if (!res_receive(p, P, phi, tag)) {
                unsigned long long t0 = 0, t1;
                for (unsigned spin = 1;; ++spin) {
                    if (res_receive(p, P, phi, tag)) break;
                    if ((spin & 255u) == 0) {  // give up after wait_ns, or when another CTA has
                        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
                        if (t0 == 0) t0 = t1;
                        if (t1 - t0 > a.wait_ns || (*reinterpret_cast<volatile int*>(a.err) & 1)) {
                            fail = true;
                            break;
                        }
                    }
                }
            }
            if (!fail) {
                T mx, my;
                res_moments(P, mx, my);
#pragma unroll
                for (int q = 0; q < 4; ++q) sP[q * NE + he] = P[q];
                sM[he] = phi;
                sM[NE + he] = mx;
                sM[2 * NE + he] = my;
            }
        }
        if (__syncthreads_or(fail)) {
            fail = true;
            break;
        }
        // faces (seq: the x-faces wait for the y-faces)
        if (!a.seq) {
            March m = m_first;
            for (int g = warp; g < gyn + gxn;) {
                if (g < gyn) y_group(m);
                else x_group(m);
                if ((g += nwarps) < gyn + gxn) m = march_of(g);
            }
        } else {
            March m = m_first;
            for (int g = warp; g < gyn;) {
                y_group(m);
                if ((g += nwarps) < gyn) m = march_of(g);
            }
            __syncthreads();
            m = mx_first;
            for (int g = warp; g < gxn;) {
                x_group(m);
                if ((g += nwarps) < gxn) m = march_of(gyn + g);
            }
        }
        __syncthreads();
    }
    if (fail) {
        if (tid == 0) atomicOr(a.err, 1);
        return;
    }
    for (int i = tid; i < ncell; i += NT) {
        const int ly = i / tx, lx = i - ly * tx, u = ly * UX + lx;
        PT F[4];
        state_of(u, lx, F);
        T* dst = a.fout + (long long)(y0 + ly) * a.pitch + x0 + lx;
        dst[0] = sZ[u];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            dst[PA(q) * a.plane] = F[q].v.x;
            dst[PB(q) * a.plane] = F[q].v.y;
        }
        if (SRC) sa.hist[(long long)(y0 + ly) * sa.hpitch + x0 + lx] = sH[u];
    }
    if (tid == 0) a.epoch[blockIdx.x] = tag0 + unsigned(a.nsteps);
}

}  // namespace dugks
