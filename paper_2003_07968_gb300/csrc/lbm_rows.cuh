// lbm_rows.cuh -- kernels whose warps work on rows of 64 columns, each lane on
// two adjacent columns.
//
// A lane holds columns x and x + 1 in the lanes of a float2; the values of its
// neighbouring columns come from the neighbouring lanes by shuffles, so a row
// needs one 8-byte access per plane (one 4-byte access in FP16 storage) and
// no unaligned ones.  60 of the 64 columns are the warp's own; the two on
// each side are what the pulls (one column) of psi's ring (one column) reach.
// The arithmetic is that of lbm_device.cuh, operation for operation, so every
// result is bitwise that of the tile kernels.
#pragma once
#include "lbm_async.cuh"
#include "lbm_kernels.h"
#include "lbm_rows_plan.h"

namespace pplbm {
namespace {


// Pairs of horizontally adjacent stored values.
template <class S> struct PairIO;
template <>
struct PairIO<StoreF32> {
    using Raw = float2;
    static __device__ __forceinline__ Raw ld(const float* p) {
        Raw v;
        asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ float2 val(Raw r) { return r; }
    static __device__ __forceinline__ float2 left(Raw r) {
        return make_float2(__shfl_up_sync(0xffffffffu, r.y, 1), r.x);
    }
    static __device__ __forceinline__ float2 right(Raw r) {
        return make_float2(r.y, __shfl_down_sync(0xffffffffu, r.x, 1));
    }
    static __device__ __forceinline__ void st(float* p, float2 v) {
        *reinterpret_cast<float2*>(p) = v;
    }
};
template <>
struct PairIO<StoreF16> {
    using Raw = uint32_t;
    static __device__ __forceinline__ Raw ld(const __half* p) {
        Raw v;
        asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ float2 val(Raw r) {
        return __half22float2(*reinterpret_cast<const __half2*>(&r));
    }
    static __device__ __forceinline__ float2 left(Raw r) {
        return val(__byte_perm(__shfl_up_sync(0xffffffffu, r, 1), r, 0x5432));
    }
    static __device__ __forceinline__ float2 right(Raw r) {
        return val(__byte_perm(r, __shfl_down_sync(0xffffffffu, r, 1), 0x5432));
    }
    static __device__ __forceinline__ void st(__half* p, float2 v) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v.x, v.y);
    }
};

// A row of values around the thread's pair of columns: at x - 1, x and x + 1.
struct Row3 {
    float2 l, c, r;
};
template <class S>
__device__ __forceinline__ Row3 row3(typename PairIO<S>::Raw v) {
    Row3 o;
    o.l = PairIO<S>::left(v);
    o.c = PairIO<S>::val(v);
    o.r = PairIO<S>::right(v);
    return o;
}
__device__ __forceinline__ Row3 row3(float2 v) { return row3<StoreF32>(v); }

// The pulled state of row y from g (g[i]: plane i's row y - c_iy at the pair's
// own columns) and the rest plane's rows y - 1, y, y + 1.
template <class S>
__device__ __forceinline__ Site<float2> row_site(const typename PairIO<S>::Raw g[9],
                                                 const Row3& Rm, const Row3& Rc, const Row3& Rp) {
    using IO = PairIO<S>;
    float2 R[9], Gs[9];
    Gs[0] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const Row3& w = plane_cy(i) == 0 ? Rc : plane_cy(i) > 0 ? Rm : Rp;  // row y - c_iy
        R[i] = plane_cx(i) == 0 ? w.c : plane_cx(i) > 0 ? w.l : w.r;        // column x - c_ix
        if (i)
            Gs[i] = plane_cx(i) == 0  ? IO::val(g[i])
                    : plane_cx(i) > 0 ? IO::left(g[i])
                                      : IO::right(g[i]);
    }
    return make_site(R, Gs);
}

// Collision of a row from its pulled state and psi's rows y - 1, y, y + 1.
template <class S, bool MRT>
__device__ __forceinline__ void row_collide(const SiteConsts& C, const float* mrt_s,
                                            const Site<float2>& s, const Row3& P0, const Row3& P1,
                                            const Row3& P2, float2 v[9]) {
    float2 p[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const Row3& w = plane_cy(i) == 0 ? P1 : plane_cy(i) > 0 ? P2 : P0;  // row y + c_iy
        p[i] = plane_cx(i) == 0 ? w.c : plane_cx(i) > 0 ? w.r : w.l;        // column x + c_ix
    }
    collide<S, MRT>(C, mrt_s, s, p, v);
}

// Store a row's outputs: q is the pair's place in the row (plane 0), in0 and
// in1 say which of its two sites are the warp's; `edge` (uniform): the row or
// the strip touches the lattice's edge, so some sites have periodic images.
template <class S>
__device__ __forceinline__ void row_store(typename S::T* q, int64_t plane, int pitch, int x, int y,
                                          int nx, int ny, bool in0, bool in1, bool edge,
                                          const float2 v[9]) {
    using T = typename S::T;
    if (in1) {
#pragma unroll
        for (int i = 0; i < 9; ++i) PairIO<S>::st(q + i * plane, v[i]);
    } else if (in0) {
#pragma unroll
        for (int i = 0; i < 9; ++i) q[i * plane] = S::cv(v[i].x);
    }
    if (edge) {
        // the row itself (m = 0: images across x only) and its image rows
        for (int m = 0; m < 3; ++m) {
            if (m == 1 && y >= GW) continue;
            if (m == 2 && y < ny - GW) continue;
            T* r = q + (int64_t)(m == 0 ? 0 : m == 1 ? ny : -ny) * pitch;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                T* o = r + i * plane;
                const T u0 = S::cv(v[i].x), u1 = S::cv(v[i].y);
                if (m && in0) o[0] = u0;
                if (m && in1) o[1] = u1;
                if (in0 && x < GW) o[nx] = u0;
                if (in1 && x + 1 < GW) o[1 + nx] = u1;
                if (in0 && x >= nx - GW) o[-nx] = u0;
                if (in1 && x + 1 >= nx - GW) o[1 - nx] = u1;
            }
        }
    }
}

// A strip of columns: x0 .. xend - 1 are the warp's, lane l holds columns
// x0 - 2 + 2 l and the next.
struct Strip {
    int x, xl;  // the pair's first column; the same clamped into the row for loads
    bool in0, in1;
    unsigned live;  // lanes whose psi is needed (x0 - 1 .. xend)
};
__device__ __forceinline__ Strip strip_of(int x0, int xend, int pitch, int gx) {
    Strip s;
    s.x = x0 - 2 + 2 * (int)(threadIdx.x & 31);
    s.xl = min(s.x, pitch - gx - 2);
    s.in0 = s.x >= x0 && s.x < xend;
    s.in1 = s.x >= x0 && s.x + 1 < xend;
    s.live = (unsigned)(s.x >= x0 - 1 && s.x <= xend) |
             ((unsigned)(s.x + 1 >= x0 - 1 && s.x + 1 <= xend) << 1);
    return s;
}

// ---------------------------------------------------------------- one step a launch
// What a warp pulls for row y of its columns, from global memory (row: the
// pair's place in row y of plane 0).
template <class S>
__device__ __forceinline__ void load_g(typename PairIO<S>::Raw g[9], const typename S::T* row,
                                       int64_t plane, int pitch) {
#pragma unroll
    for (int i = 1; i < 9; ++i)
        g[i] = PairIO<S>::ld(row + i * plane - (int64_t)plane_cy(i) * pitch);
}

// entry of a row-item list: (lattice, x0, y0, rows | width << 24)
__device__ __forceinline__ int item_rows(int w) { return w & 0xffffff; }
__device__ __forceinline__ int item_width(int w) { return w >> 24; }

// k_rows: one step; every warp marches down the rows of an item of its own,
// with no shared memory and no barrier.  Row y's values are loaded one row
// ahead into registers; its pulled state and psi are computed, psi's row goes
// to the neighbouring lanes by shuffles, and row y - 1, whose state waited in
// registers, is collided and stored.  An item of h rows computes psi for
// h + 2 and reads h + 4; a tile kernel's 32 x 16 tile computes it for 18 x 34
// sites, fetches 20 x 40 and holds its warps at a barrier per tile.
//
// What bounds it: FP16 storage the FP32 pipe (its heavy half is busy 73 % of its
// cycles, 64 % of issue slots; paired instructions take two cycles), FP32
// storage beyond L2 DRAM.  Measured per step, tile kernel (32 x 16) -> this one,
// FP16: 4096^2 244 -> 190 us, 8192^2 937 -> 688 us (97.6 GLUPS); MRT 288 -> 230
// and 1112 -> 846 us.  FP32 storage has the batch instance only, for the last
// step of served requests with an odd number of steps (k_rows2 takes the others;
// on handles the tile kernel takes an odd step); it spills 76 bytes.
// Unrolling the row loop by 2 to save its register copies gained 4 % in FP16
// BGK and spilled in the others (MRT 10 % slower); 5 blocks an SM spill too.
template <class S, int EOSP, bool MRT, bool ONE>
__global__ void __launch_bounds__(32 * kRowWarps, 4)
    k_rows(StepArgs a, const __grid_constant__ LatDev lat0) {
    using T = typename S::T;
    using IO = PairIO<S>;
    using Raw = typename IO::Raw;
    __shared__ LatDev slat[ONE ? 1 : kRowWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    (void)lane;
    for (int t = blockIdx.x * kRowWarps + w; t < a.ntiles; t += gridDim.x * kRowWarps) {
        const int4 tl = __ldg(&a.tiles[t]);
        if (a.quota) {
            const int left = __ldg(&a.quota[tl.x]) - a.step;
            if (left <= 0 || (a.last_only && left > 1)) continue;
        }
        if (!ONE) {
            // the lattice's constants, in the warp's own copy
            __syncwarp();
            for (int k = lane; k < (int)(sizeof(LatDev) / 4); k += 32)
                reinterpret_cast<int*>(&slat[w])[k] = __ldg(reinterpret_cast<const int*>(a.lats + tl.x) + k);
            __syncwarp();
        }
        const LatDev& L = ONE ? lat0 : slat[w];
        const SiteConsts C = site_consts(L);
        const int nx = L.nx, ny = L.ny, pitch = L.pitch, gx = L.gx;
        const int64_t plane = L.plane;
        const int x0 = tl.y, y0 = tl.z, y1 = tl.z + item_rows(tl.w), xend = x0 + item_width(tl.w);
        const Strip sp = strip_of(x0, xend, pitch, gx);
        // row y0 - 1 of plane 0 (the first row whose psi is needed)
        const T* p = reinterpret_cast<const T*>(a.pop) + L.off_f[a.parity] +
                     (int64_t)(y0 - 1 + GY) * pitch + gx + sp.xl;
        T* q = reinterpret_cast<T*>(a.pop) + L.off_f[a.parity ^ 1] +
               (int64_t)(y0 - 2 + GY) * pitch + gx + sp.x;
        Row3 Rm = row3<S>(IO::ld(p - pitch)), Rc = row3<S>(IO::ld(p));
        Raw gn[9], rn;
        load_g<S>(gn, p, plane, pitch);
        rn = IO::ld(p + pitch);
        Site<float2> sprev{};
        Row3 P0{}, P1{};
        for (int y = y0 - 1; y <= y1; ++y) {
            Raw g[9];
#pragma unroll
            for (int i = 1; i < 9; ++i) g[i] = gn[i];
            const Row3 Rp = row3<S>(rn);
            p += pitch;
            if (y < y1) {
                load_g<S>(gn, p, plane, pitch);
                rn = IO::ld(p + pitch);
            }
            const Site<float2> s = row_site<S>(g, Rm, Rc, Rp);
            const Row3 P2 = row3(Eos<EOSP>::psi(L, site_rho(s, L.rho0), a.status, sp.live));
            if (y > y0) {
                const int ys = y - 1;
                float2 v[9];
                row_collide<S, MRT>(C, L.mrt_s, sprev, P0, P1, P2, v);
                row_store<S>(q, plane, pitch, sp.x, ys, nx, ny, sp.in0, sp.in1,
                             x0 < GW || xend > nx - GW || ys < GW || ys >= ny - GW, v);
            }
            q += pitch;
            sprev = s;
            P0 = P1;
            P1 = P2;
            Rm = Rc;
            Rc = Rp;
        }
    }
}

// ---------------------------------------------------------------- two steps a launch
__device__ __forceinline__ float ld_one(const float* p) {
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// k_rows2: two steps; a pair of warps marches down an item's rows.  The first
// warp takes the first step as k_rows does, on 64 columns of which 60 come
// out right, and hands its rows to the second through a ring of eight rows in
// shared memory; the second takes the second step on those and stores 56
// columns.  The lattice's periodic neighbours are read where they are (rows
// and columns wrapped), not from the images, which reach two sites only.
//
// One step a launch moves 72 bytes a site and step (FP32) and stops at 0.81 of
// the copy bandwidth; two move 36, and the kernel is bound by the FP32 pipe
// (72 % of its heavy half's cycles, 63 % of issue slots).  The batch instances
// hold the lattice's constants in registers beside the rows and spill (100
// bytes, MRT 28); the others do not.  Measured per step, 32 x 16 tile
// kernel -> this one: FP32 BGK 1024^2 19.2 -> 16.3 us, 1201^2 33.2 -> 21.6,
// 2100 x 1700 51.6 -> 46.2, 4096^2 221 -> 191, 8192^2 870 -> 706 (95 GLUPS);
// MRT 8192^2 984 -> 865; 512 lattices of 64^2 .. 512^2 804 -> 730, 100 of
// 64^2 .. 200^2 48 -> 40.  FP16 storage, which is not bound by DRAM, loses by
// the columns it computes twice (8192^2: k_rows 688, this one 778).
// Unrolling either row loop by 2 is 3 to 25 % slower; 64-bit addresses and a
// test per load instead of one per row cost 6 %.
template <int EOSP, bool MRT, bool ONE>
__global__ void __launch_bounds__(64 * kPairs, 2)
    k_rows2(StepArgs a, const __grid_constant__ LatDev lat0) {
    using S = StoreF32;
    using T = S::T;
    using IO = PairIO<S>;
    using Raw = IO::Raw;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ LatDev slat[ONE ? 1 : kPairs];
    __shared__ uint64_t bars[kPairs][2 * kPairDepth];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, pr = w % kPairs;
    Raw* const ring = reinterpret_cast<Raw*>(smem_raw) + pr * (kPairDepth * 9 * 32);  // [depth][9][32]
    uint64_t* const full = bars[pr];
    uint64_t* const empty = full + kPairDepth;
    const int t = blockIdx.x * kPairs + pr;
    int4 tl = make_int4(0, 0, 0, 0);
    bool on = t < a.ntiles;
    if (on) {
        tl = __ldg(&a.tiles[t]);
        // (a lattice with one step left is not this launch's)
        on = !a.quota || a.step + 2 <= __ldg(&a.quota[tl.x]);
    }
    if (w < kPairs && lane == 0) {
        // (failure-detection test: an armed item's rows never count as handed over)
        const uint32_t arrivals = a.starve == t + 1 ? 2 : 1;
        for (int k = 0; k < kPairDepth; ++k) {
            mbar_init(&full[k], arrivals);
            mbar_init(&empty[k], 1);
        }
        mbar_fence_init();
    }
    if (!ONE && w < kPairs && on)
        for (int k = lane; k < (int)(sizeof(LatDev) / 4); k += 32)
            reinterpret_cast<int*>(&slat[pr])[k] = __ldg(reinterpret_cast<const int*>(a.lats + tl.x) + k);
    __syncthreads();
    if (!on) return;
    const LatDev& L = ONE ? lat0 : slat[pr];
    const SiteConsts C = site_consts(L);
    const int nx = L.nx, ny = L.ny, pitch = L.pitch, gx = L.gx;
    const int64_t plane = L.plane;
    const int x0 = tl.y, y0 = tl.z, y1 = tl.z + item_rows(tl.w), xend = x0 + item_width(tl.w);
    const int x = x0 - 4 + 2 * lane;
    auto need = [&](int lo, int hi) {  // which of the lane's columns lie in lo .. hi
        return (unsigned)(x >= lo && x <= hi) | ((unsigned)(x + 1 >= lo && x + 1 <= hi) << 1);
    };
    Row3 P0{}, P1{};
    Site<float2> sprev{};
    if (w < kPairs) {
        // ------------------------------------------------------ first step
        const unsigned live = need(x0 - 3, xend + 2);
        const int c0 = ((x % nx) + nx) % nx, c1 = c0 + 1 == nx ? 0 : c0 + 1;
        const bool whole = __all_sync(0xffffffffu, !(c0 & 1) && c1 == c0 + 1);
        // byte offsets of the pair's place in a row of a plane (32 bits: the planes
        // of a lattice on this path are smaller than 4 GB)
        const char* const base = reinterpret_cast<const char*>(
            reinterpret_cast<const T*>(a.pop) + L.off_f[a.parity]);
        const uint32_t prow = (uint32_t)pitch * (uint32_t)sizeof(T);
        const uint32_t col = (uint32_t)(GY * pitch + gx + c0) * (uint32_t)sizeof(T);
        const int next = (c1 - c0) * (int)sizeof(T);
        auto down = [&](int y) { return y + 1 == ny ? 0 : y + 1; };
        auto at = [&](int i, uint32_t o) {
            return reinterpret_cast<const T*>(base + i * plane * (int64_t)sizeof(T) + o);
        };
        auto one = [&](int i, uint32_t o) {
            return make_float2(ld_one(at(i, o)), ld_one(at(i, o + (uint32_t)next)));
        };
        auto ld = [&](int i, uint32_t o) { return whole ? IO::ld(at(i, o)) : one(i, o); };
        auto load = [&](Raw g[9], Raw& rest, uint32_t om, uint32_t oc, uint32_t op) {
            if (whole) {
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    g[i] = IO::ld(at(i, plane_cy(i) == 0 ? oc : plane_cy(i) > 0 ? om : op));
                rest = IO::ld(at(0, op));
            } else {
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    g[i] = one(i, plane_cy(i) == 0 ? oc : plane_cy(i) > 0 ? om : op);
                rest = one(0, op);
            }
        };
        int yw = ((y0 - 4) % ny + ny) % ny;  // row y - 1, then the rows after it
        uint32_t om = (uint32_t)yw * prow + col;
        yw = down(yw);
        uint32_t oc = (uint32_t)yw * prow + col;
        yw = down(yw);
        uint32_t op = (uint32_t)yw * prow + col;
        Row3 Rm = row3<S>(ld(0, om)), Rc = row3<S>(ld(0, oc));
        Raw gn[9], rn;
        load(gn, rn, om, oc, op);
        for (int y = y0 - 3; y <= y1 + 2; ++y) {
            Raw g[9];
#pragma unroll
            for (int i = 1; i < 9; ++i) g[i] = gn[i];
            const Row3 Rp = row3<S>(rn);
            if (y < y1 + 2) {
                om = oc;
                oc = op;
                yw = down(yw);
                op = (uint32_t)yw * prow + col;
                load(gn, rn, om, oc, op);
            }
            const Site<float2> s = row_site<S>(g, Rm, Rc, Rp);
            const Row3 P2 = row3(Eos<EOSP>::psi(L, site_rho(s, L.rho0), a.status, live));
            if (y >= y0 - 1) {
                float2 v[9];
                row_collide<S, MRT>(C, L.mrt_s, sprev, P0, P1, P2, v);
                const unsigned n = (unsigned)(y - (y0 - 1)), slot = n % kPairDepth;  // row y0 - 2 + n
                if (n >= kPairDepth) {
                    const bool ok = mbar_wait_bounded(&empty[slot], (uint32_t)(n / kPairDepth - 1) & 1u,
                                                      a.wait_cycles);
                    if (!__all_sync(0xffffffffu, ok)) {
                        if (lane == 0) atomicOr(a.status + L.lattice, 2u);
                        return;
                    }
                }
                T* q = reinterpret_cast<T*>(ring + slot * (9 * 32) + lane);
#pragma unroll
                for (int i = 0; i < 9; ++i) IO::st(q + i * 64, v[i]);
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[slot]);
            }
            sprev = s;
            P0 = P1;
            P1 = P2;
            Rm = Rc;
            Rc = Rp;
        }
    } else {
        // ------------------------------------------------------ second step
        const unsigned live = need(x0 - 1, xend);
        const bool in0 = x >= x0 && x < xend, in1 = x >= x0 && x + 1 < xend;
        T* q = reinterpret_cast<T*>(a.pop) + L.off_f[a.parity ^ 1] +
               (int64_t)(y0 - 2 + GY) * pitch + gx + x;
        auto got = [&](unsigned n) {
            const bool ok =
                mbar_wait_bounded(&full[n % kPairDepth], (uint32_t)(n / kPairDepth) & 1u, a.wait_cycles);
            return __all_sync(0xffffffffu, ok);
        };
        auto row = [&](int i, unsigned n) { return ring[((n % kPairDepth) * 9 + i) * 32 + lane]; };
        bool ok = got(0) && got(1);
        Row3 Rm{}, Rc{};
        if (ok) {
            Rm = row3<S>(row(0, 0));
            Rc = row3<S>(row(0, 1));
        }
        for (int y = y0 - 1; y <= y1; ++y) {
            const unsigned n = (unsigned)(y - (y0 - 2));  // ring row of lattice row y
            ok = ok && got(n + 1);
            if (!ok) {
                if (lane == 0) atomicOr(a.status + L.lattice, 2u);
                return;
            }
            const Row3 Rp = row3<S>(row(0, n + 1));
            Raw g[9];
#pragma unroll
            for (int i = 1; i < 9; ++i) g[i] = row(i, n - plane_cy(i));
            const Site<float2> s = row_site<S>(g, Rm, Rc, Rp);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[(n - 1) % kPairDepth]);  // row y - 1 is done with
            const Row3 P2 = row3(Eos<EOSP>::psi(L, site_rho(s, L.rho0), a.status, live));
            if (y > y0) {
                const int ys = y - 1;
                float2 v[9];
                row_collide<S, MRT>(C, L.mrt_s, sprev, P0, P1, P2, v);
                row_store<S>(q, plane, pitch, x, ys, nx, ny, in0, in1,
                             x0 < GW || xend > nx - GW || ys < GW || ys >= ny - GW, v);
            }
            q += pitch;
            sprev = s;
            P0 = P1;
            P1 = P2;
            Rm = Rc;
            Rc = Rp;
        }
    }
}

// ---------------------------------------------------------------- resident lattices
// 16-byte packets between blocks: three values and the step's tag, written
// and read as one 128-bit access.
__device__ __forceinline__ uint4 ld_mail(const uint4* p) {
    uint64_t lo, hi;
    asm volatile(
        "{\n\t.reg .b128 v;\n\tld.relaxed.gpu.global.b128 v, [%2];\n\tmov.b128 {%0, %1}, v;\n\t}"
        : "=l"(lo), "=l"(hi)
        : "l"(p)
        : "memory");
    return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}
__device__ __forceinline__ void st_mail(uint4* p, uint4 v) {
    const uint64_t lo = (uint64_t)v.y << 32 | v.x, hi = (uint64_t)v.w << 32 | v.z;
    asm volatile(
        "{\n\t.reg .b128 v;\n\tmov.b128 v, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(p),
        "l"(lo), "l"(hi)
        : "memory");
}
template <class T>
__device__ __forceinline__ uint32_t to_bits(T v) {
    if constexpr (sizeof(T) == 4)
        return __float_as_uint(v);
    else
        return __half_as_ushort(v);
}
template <class T>
__device__ __forceinline__ T of_bits(uint32_t b) {
    if constexpr (sizeof(T) == 4)
        return __uint_as_float(b);
    else
        return __ushort_as_half((unsigned short)b);
}

// Planes a tile needs from the two rows (columns) before its first: 4 of the
// outer one, then 6 of the inner one; and from the two after its last: 6 of
// the inner, then 4 of the outer one.
//   rows:    0 2 5 6 | 0 1 3 2 5 6 | 0 1 3 4 7 8 | 0 4 7 8
//   columns: 0 1 5 8 | 0 2 4 1 5 8 | 0 2 4 3 6 7 | 0 3 6 7
__device__ __forceinline__ int halo_plane(bool cols, int k) {
    constexpr unsigned char R[20] = {0, 2, 5, 6, 0, 1, 3, 2, 5, 6, 0, 1, 3, 4, 7, 8, 0, 4, 7, 8};
    constexpr unsigned char Cc[20] = {0, 1, 5, 8, 0, 2, 4, 1, 5, 8, 0, 2, 4, 3, 6, 7, 0, 3, 6, 7};
    return cols ? Cc[k] : R[k];
}
// 0: outer before, 1: inner before, 2: inner after, 3: outer after
__device__ __forceinline__ int halo_line(int k) { return k < 4 ? 0 : k < 10 ? 1 : k < 16 ? 2 : 3; }

// k_resident: many time steps in one cooperative launch.  Every block keeps one
// tile (at most 60 columns) of a lattice in shared memory from the first step
// to the last; a step's halo goes from block to block in packets of three
// values and the step's number.  A reader polls a packet until it carries the
// number it waits for, so data and signal arrive together: no fence, no flag,
// no barrier across blocks, and global memory is read and written once a
// launch instead of once a step.
//
// What bounds it: latency.  A launch per step costs 5.2-5.4 us for any
// lattice up to about 256^2 (launch, first loads, psi barrier, stores and the
// end of the grid, one after another); here a step is psi and collision (950
// cycles at 64^2, 1450 at 256^2, 8800 for the 21 rows a tile of 777 x 611),
// packets out (1050, 1400, 1300) and packets in (2000, 2550, 4500 with the wait
// for the slowest neighbour): two trips to L2.  Measured per step, FP32, one
// launch per step in a graph -> here: 64^2 5.2 -> 2.0 us, 200^2 MRT 5.4 -> 2.5
// us, 256^2 5.3 -> 2.7 us, 777 x 611 11.0 -> 7.2 us.  Flags behind release
// fences instead of tagged packets took 3.0 us at 64^2 and 5.3 us at 256^2;
// 8-byte packets of one value 2.1 and 3.2 us.
//
// Rows j = 0 .. rows + 1 of a tile's psi are lattice rows y0 - 1 .. y0 + rows.
// A round is eight rows, one a warp: pulled state and psi of the round's
// rows, one barrier, collision of the round before.  The collision writes its
// rows in place: what a round still pulls lies after the rows of the round
// before, and the states pulled earlier are in registers.  Two blocks share an
// SM, so that one computes while the other waits for its halo.
//
// Two mailbox slots alternate by the step's number.  A slot's packet is
// overwritten two steps later, which its writer reaches only with its
// reader's packets of the step between, and the reader sent those after it
// had read the slot.  epoch counts a tile's steps over all launches, so a
// number never comes twice (all tiles of a handle are equal between
// launches).  Every wait is bounded: a block whose wait runs out raises
// status bit 2 and leaves, and its neighbours' waits run out in turn.
template <class S, int EOSP, bool MRT, bool ONE>
__global__ void __launch_bounds__(32 * kResWarps, 2)
    k_resident(const __grid_constant__ ResArgs m, const __grid_constant__ LatDev lat0) {
    using T = typename S::T;
    using IO = PairIO<S>;
    using Raw = typename IO::Raw;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const StepArgs& a = m.a;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const ResTile tl = m.tiles[blockIdx.x];
    const int x0 = tl.x0, wd = tl.wd, y0 = tl.y0, rows = tl.rows, xend = x0 + wd;
    const int RR = rows + 4;
    float2* psi = reinterpret_cast<float2*>(smem_raw);  // [rows + 2][32]
    uint2* mw = reinterpret_cast<uint2*>(psi + (rows + 2) * 32);  // packet table
    // packets: ten lines of the rows above and below, and of the columns left
    // and right, three values each; ten of two at each corner
    const int gw = (wd + 2) / 3, gr = (rows + 2) / 3, npack = 20 * (gw + gr) + 40;
    LatDev* slat = reinterpret_cast<LatDev*>(mw + npack);
    Raw* F = reinterpret_cast<Raw*>(slat + 1);  // [9][RR][32]
    T* const box = reinterpret_cast<T*>(F);
    if (!ONE) {
        for (int k = tid; k < (int)(sizeof(LatDev) / 4); k += blockDim.x)
            reinterpret_cast<int*>(slat)[k] = reinterpret_cast<const int*>(a.lats + tl.lattice)[k];
        __syncthreads();
    }
    const LatDev& L = ONE ? lat0 : *slat;
    const int nx = L.nx, ny = L.ny, pitch = L.pitch, gx = L.gx;
    const int64_t plane = L.plane;
    const Strip sp = strip_of(x0, xend, pitch, gx);
    const uint32_t epoch = m.epoch[blockIdx.x];
    // Packet u of the tile's own halo: its place in the box (.x, low half); and
    // the packet u that it sends: the values' place (.x, high half) and the
    // mailbox packet it goes to (.y, 20 bits).  Above that in .y: the number of
    // values (2 bits) and whether they lie along a column (received, sent).
    for (int u = tid; u < npack; u += 32 * kResWarps) {
        int q, rr, rc, sr, sc, pl, t, to, n;
        bool col = false;
        if (u < 20 * gw) {  // rows: received from above (lines 0, 1) and below
            q = u / gw;
            const int g = u - q * gw, ln = halo_line(q);
            pl = halo_plane(false, q);
            n = min(3, wd - 3 * g);
            rr = ln < 2 ? ln : rows + ln;
            rc = 3 * g + 2;
            // sent to the tile below (its lines 0, 1) and above, same columns
            sr = ln < 2 ? rows - 2 + ln : ln - 2;
            sc = 3 * g;
            t = ln < 2 ? tl.nbr[6] : tl.nbr[1];
            to = u;
        } else if (u < 20 * (gw + gr)) {  // columns: from the left and right
            const int v = u - 20 * gw;
            q = v / gr;
            const int g = v - q * gr, ln = halo_line(q);
            pl = halo_plane(true, q);
            n = min(3, rows - 3 * g);
            col = true;
            rr = 3 * g + 2;
            rc = ln < 2 ? ln : wd + ln;
            sr = 3 * g;
            sc = ln < 2 ? wd - 2 + ln : ln - 2;
            t = ln < 2 ? tl.nbr[4] : tl.nbr[3];
            to = 20 * (((ln < 2 ? tl.wd_e : tl.wd_w) + 2) / 3) + v;
        } else {  // corners: a row line's two columns left (k = 0) and right (k = 1)
            const int v = u - 20 * (gw + gr), k = v & 1;
            q = v >> 1;
            const int ln = halo_line(q);
            pl = halo_plane(false, q);
            n = 2;
            rr = ln < 2 ? ln : rows + ln;
            rc = k ? wd + 2 : 0;
            // a left corner (k = 0) comes from the tile left of it: this tile
            // sends its last two columns to the right, its first two to the left
            sr = ln < 2 ? rows - 2 + ln : ln - 2;
            sc = k ? 0 : wd - 2;
            t = ln < 2 ? (k ? tl.nbr[5] : tl.nbr[7]) : (k ? tl.nbr[0] : tl.nbr[2]);
            to = 20 * (((k ? tl.wd_w : tl.wd_e) + 2) / 3 + (ln < 2 ? tl.gr_s : tl.gr_n)) + v;
        }
        const uint32_t meta = (uint32_t)n | (uint32_t)col << 2;
        mw[u] = make_uint2((uint32_t)((pl * RR + rr) * 64 + rc) |
                               (uint32_t)((pl * RR + sr + 2) * 64 + sc + 2) << 16,
                           (uint32_t)(t * (2 * m.slot) + to) | meta << 20);
    }
    // the box from the lattice: rows y0 - 2 .. y0 + rows + 1
    {
        const T* p = reinterpret_cast<const T*>(a.pop) + L.off_f[a.parity] +
                     (int64_t)(y0 - 2 + GY) * pitch + gx + sp.xl;
        for (int r = w; r < RR; r += kResWarps)
#pragma unroll
            for (int i = 0; i < 9; ++i)
                F[(i * RR + r) * 32 + lane] = IO::ld(p + i * plane + (int64_t)r * pitch);
    }
    __syncthreads();
    const int nr = rows + 2;  // rows of psi: row j is y0 - 1 + j
    Site<float2> s[2];
    for (int st = 1; st <= m.nsteps; ++st) {
        const bool last = st == m.nsteps;
        // collision of row j from its state and psi's rows j - 1, j, j + 1
        auto finish_row = [&](int j, const Site<float2>& sj) {
            if (j < 1 || j > rows) return;
            const Row3 P0 = row3(psi[(j - 1) * 32 + lane]), P1 = row3(psi[j * 32 + lane]),
                       P2 = row3(psi[(j + 1) * 32 + lane]);
            float2 v[9];
            row_collide<S, MRT>(site_consts(L), L.mrt_s, sj, P0, P1, P2, v);
            if (!last) {
                T* q = box + (j + 1) * 64 + 2 * lane;
                if (sp.in1) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) IO::st(q + i * RR * 64, v[i]);
                } else if (sp.in0) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) q[i * RR * 64] = S::cv(v[i].x);
                }
            } else {
                const int y = y0 - 1 + j;
                T* q = reinterpret_cast<T*>(a.pop) + L.off_f[a.parity ^ 1] +
                       (int64_t)(y + GY) * pitch + gx + sp.x;
                row_store<S>(q, plane, pitch, sp.x, y, nx, ny, sp.in0, sp.in1,
                             x0 < GW || xend > nx - GW || y < GW || y >= ny - GW, v);
            }
        };
        int jb = 0;
        for (; jb < nr; jb += 2 * kResWarps) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = jb + u * kResWarps + w;
                if (jb + u * kResWarps < nr) {
                    if (j < nr) {
                        const int r = j + 1;
                        const Row3 Rm = row3<S>(F[(r - 1) * 32 + lane]),
                                   Rc = row3<S>(F[r * 32 + lane]),
                                   Rp = row3<S>(F[(r + 1) * 32 + lane]);
                        Raw g[9];
#pragma unroll
                        for (int i = 1; i < 9; ++i) g[i] = F[(i * RR + r - plane_cy(i)) * 32 + lane];
                        s[u] = row_site<S>(g, Rm, Rc, Rp);
                        psi[j * 32 + lane] =
                            Eos<EOSP>::psi(L, site_rho(s[u], L.rho0), a.status, sp.live);
                    }
                    __syncthreads();
                    if (j >= kResWarps) finish_row(j - kResWarps, s[u ^ 1]);
                }
            }
        }
        // the last round's rows
        {
            const int j = (nr - 1) / kResWarps * kResWarps + w;
            if (((nr - 1) / kResWarps) & 1)
                finish_row(j, s[1]);
            else
                finish_row(j, s[0]);
        }
        if (last) break;
        __syncthreads();  // the tile's new values are in the box
        const uint32_t tag = epoch + (uint32_t)st;
        uint4* const mail = m.mail + (tag & 1u) * m.slot;
        constexpr int NB = 3;  // packets a thread has in flight
        for (int u0 = tid; u0 < npack; u0 += NB * 32 * kResWarps) {
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (u0 + 32 * kResWarps * k < npack) {
                    const uint2 q = mw[u0 + 32 * kResWarps * k];
                    // (a line's last packet may read past its values: inside the box)
                    const int d = q.y >> 22 & 1 ? 64 : 1;
                    const T* v = box + (q.x >> 16);
                    st_mail(mail + (q.y & 0xfffff),
                            make_uint4(to_bits(v[0]), to_bits(v[d]), to_bits(v[2 * d]), tag));
                }
        }
        const uint4* in = mail + (uint64_t)blockIdx.x * (2 * m.slot);
        bool late = false;
        for (int u0 = tid; u0 < npack && !late; u0 += NB * 32 * kResWarps) {
            unsigned left = 0;
#pragma unroll
            for (int k = 0; k < NB; ++k) left |= (unsigned)(u0 + 32 * kResWarps * k < npack) << k;
            long long c0 = 0;
            for (int it = 0; left; ++it) {
                uint4 v[NB];
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if (left >> k & 1) v[k] = ld_mail(in + u0 + 32 * kResWarps * k);
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if ((left >> k & 1) && v[k].w == tag) {
                        const uint2 q = mw[u0 + 32 * kResWarps * k];
                        const int d = q.y >> 22 & 1 ? 64 : 1, n = q.y >> 20 & 3;
                        T* o = box + (q.x & 0xffffu);
                        o[0] = of_bits<T>(v[k].x);
                        if (n > 1) o[d] = of_bits<T>(v[k].y);
                        if (n > 2) o[2 * d] = of_bits<T>(v[k].z);
                        left &= ~(1u << k);
                    }
                if (it == 0)
                    c0 = clock64();
                else if (left && clock64() - c0 > a.wait_cycles) {
                    late = true;
                    break;
                }
            }
        }
        if (__syncthreads_or(late)) {
            if (tid == 0) atomicOr(&a.status[tl.lattice], 2u);
            return;
        }
    }
    if (tid == 0) m.epoch[blockIdx.x] = epoch + (uint32_t)m.nsteps;
}

// ---------------------------------------------------------------- launchers
template <class S, bool MRT, bool ONE>
cudaError_t resident_inst(const ResArgs* m, const LatDev* lat0, int grid, cudaStream_t st, int* occ) {
    const void* fn = (const void*)k_resident<S, EOS_DF, MRT, ONE>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
    if (e != cudaSuccess) return e;
    if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, fn, 32 * kResWarps, kResSmem);
    ResArgs args = *m;
    LatDev lat = lat0 ? *lat0 : LatDev{};
    void* p[] = {&args, &lat};
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(32 * kResWarps), p, kResSmem, st);
}

template <class S, bool MRT, bool ONE>
cudaError_t rows_inst(const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    const unsigned grid = (unsigned)((a.ntiles + kRowWarps - 1) / kRowWarps);
    k_rows<S, EOS_DF, MRT, ONE><<<grid, 32 * kRowWarps, 0, st>>>(a, lat0 ? *lat0 : LatDev{});
    return cudaGetLastError();
}

template <bool MRT, bool ONE>
cudaError_t pairs_inst(const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    constexpr int smem = (int)kPairSmem;
    const cudaError_t e = cudaFuncSetAttribute((const void*)k_rows2<EOS_DF, MRT, ONE>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((a.ntiles + kPairs - 1) / kPairs);
    k_rows2<EOS_DF, MRT, ONE><<<grid, 64 * kPairs, smem, st>>>(a, lat0 ? *lat0 : LatDev{});
    return cudaGetLastError();
}

}  // namespace

// (FP32 storage: the odd last steps of a server's requests only)
template <class S>
cudaError_t rows_any(int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    if constexpr (sizeof(typename S::T) == 4)
        return mrt || lat0 ? cudaErrorInvalidValue : rows_inst<S, false, false>(a, nullptr, st);
    else if (mrt)
        return lat0 ? rows_inst<S, true, true>(a, lat0, st) : rows_inst<S, true, false>(a, nullptr, st);
    else
        return lat0 ? rows_inst<S, false, true>(a, lat0, st) : rows_inst<S, false, false>(a, nullptr, st);
}

// One storage type: the launch (occ null), or its blocks per SM into *occ
// (lat0 not null: one lattice).
template <class S>
cudaError_t resident_any(int mrt, const ResArgs* m, const LatDev* lat0, int grid, cudaStream_t st,
                         int* occ) {
    if (mrt)
        return lat0 ? resident_inst<S, true, true>(m, lat0, grid, st, occ)
                    : resident_inst<S, true, false>(m, lat0, grid, st, occ);
    return lat0 ? resident_inst<S, false, true>(m, lat0, grid, st, occ)
                : resident_inst<S, false, false>(m, lat0, grid, st, occ);
}

}  // namespace pplbm
