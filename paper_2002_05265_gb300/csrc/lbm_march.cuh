// Time-fused step kernel: one launch advances a lattice by t <= TMAX time steps with one read
// and one write of its populations.
//
// A warp owns a strip of 64 columns, two neighbouring nodes per lane, and marches up the rows.
// At each row it loads the nine pulled rows, collides them (level 1, time step 1), keeps what
// level 2 will pull, collides row y - 1 of level 2 from that, and so on; level t is stored.  A level
// needs the rows y - 1, y, y + 1 of the level below: the populations with xi_y = -1 come from the row
// that level just produced, those with xi_y = 0 and +1 from one and two rows earlier, so nine pairs
// per level wait in the lane's own column of shared memory (or three of them in registers).  The
// neighbours in x are lanes: one shuffle per x-shifted population.  Warps share nothing, so there is
// no barrier.
// The price is redundant work at the strip's edges: every level spoils one node on each side
// (the outer lanes' results are discarded, adjacent strips overlap: 56 of 64 columns are stored at
// t = 4), and a march over H rows starts with rows of the lower levels that its neighbour in y also
// computes (t - 1 of level 1).
//
// Why: one step per launch moves 2 x 9 x s bytes per node update, and the FP32 kernels sit at
// the measured copy bandwidth with it (72 B per update, 0.98-1.02 of it); fused, a launch moves that
// per t updates, and what bounds it is the FP32 pipe (80-103 operations per update, collide_f32;
// ncu, 4096^2 K: pipe 66 % busy, issue 57 %, the rest register-port conflicts of three-operand
// instructions), reached by colliding the lane's two nodes with the two-wide FP32 instructions.
// Measured, us a step, one-step launches before and four-step launches after: 16384^2 FP32 K 2905 ->
// 1157, BGK 2824 -> 963; 4096^2 CHM 184 -> 74, BF16 116 -> 76; 2048^2 CM 48.8 -> 20.9; 1024^2 K 10.0 ->
// 7.1; eight 1024^2 lattices of all models 93 -> 42.1.
// A reference velocity (SHIFT) costs 18 %: 4096^2 K 77.2 us a step without, 90.9 with.
// Fewer or more levels: 3 at most 1.33x the time of 4 (4096^2 BGK), 5 1.05x, 6 1.2x (the edges).
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// Two neighbouring nodes' values of one population, as stored.
template <typename S> struct Pair16 {   // 16-bit storage: one register
    uint32_t v;
};
template <typename S> struct MarchPair {
    using type = Pair16<S>;
};
template <> struct MarchPair<float> {
    using type = F2;
};

// asynchronous copies global -> the lane's shared memory (cp.async); plain loads instead of
// them are moved by the compiler to where their values are first needed
__device__ __forceinline__ uint32_t shared_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int BYTES> __device__ __forceinline__ void fetch_bytes(void* d, const void* s) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(shared_addr(d)), "l"(s), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void fetch_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void pair_fetch(F2* d, const float* p) { fetch_bytes<8>(d, p); }
__device__ __forceinline__ void pair_fetch2(F2* d, const float* a, const float* b) {
    fetch_bytes<4>(d, a);
    fetch_bytes<4>(reinterpret_cast<float*>(d) + 1, b);
}
__device__ __forceinline__ void pair_store(float* p, F2 v) {
    float2 o;
    f2_split(v, o.x, o.y);
    *reinterpret_cast<float2*>(p) = o;
}
__device__ __forceinline__ void pair_store_lo(float* p, F2 v) { *p = f2_lo(v); }
// the pair one node to the left (node x takes x - 1) / right
__device__ __forceinline__ F2 pair_from_left(F2 v) {
    float lo, hi;
    f2_split(v, lo, hi);
    return f2_make(__shfl_up_sync(0xffffffffu, hi, 1), lo);
}
__device__ __forceinline__ F2 pair_from_right(F2 v) {
    float lo, hi;
    f2_split(v, lo, hi);
    return f2_make(hi, __shfl_down_sync(0xffffffffu, lo, 1));
}
__device__ __forceinline__ F2 pair_open(F2 v) { return v; }
__device__ __forceinline__ void pair_close(F2& p, F2 v) { p = v; }

template <typename S> __device__ __forceinline__ void pair_fetch(Pair16<S>* d, const S* p) { fetch_bytes<4>(d, p); }
// (two bytes are below cp.async's smallest copy)
template <typename S> __device__ __forceinline__ void pair_fetch2(Pair16<S>* d, const S* a, const S* b) {
    const uint32_t lo = *reinterpret_cast<const unsigned short*>(a), hi = *reinterpret_cast<const unsigned short*>(b);
    d->v = lo | (hi << 16);
}
template <typename S> __device__ __forceinline__ void pair_store(S* p, Pair16<S> v) {
    *reinterpret_cast<uint32_t*>(p) = v.v;
}
template <typename S> __device__ __forceinline__ void pair_store_lo(S* p, Pair16<S> v) {
    *reinterpret_cast<unsigned short*>(p) = (unsigned short)v.v;
}
template <typename S> __device__ __forceinline__ Pair16<S> pair_from_left(Pair16<S> v) {
    return Pair16<S>{__byte_perm(__shfl_up_sync(0xffffffffu, v.v, 1), v.v, 0x5432)};
}
template <typename S> __device__ __forceinline__ Pair16<S> pair_from_right(Pair16<S> v) {
    return Pair16<S>{__byte_perm(v.v, __shfl_down_sync(0xffffffffu, v.v, 1), 0x5432)};
}
__device__ __forceinline__ F2 pair_open(Pair16<__half> p) {
    __half2 h;
    memcpy(&h, &p.v, 4);
    return f2_make(__low2float(h), __high2float(h));
}
// a bfloat16 is the upper half of the FP32 with the same value
__device__ __forceinline__ F2 pair_open(Pair16<__nv_bfloat16> p) {
    return f2_make(__uint_as_float(p.v << 16), __uint_as_float(p.v & 0xffff0000u));
}
template <typename S> __device__ __forceinline__ void pair_close(Pair16<S>& p, F2 v) {
    float lo, hi;
    f2_split(v, lo, hi);
    p.v = pack2(S(), lo, hi);
}

constexpr int kMarchWarps = 8;    // most warps of a CTA; all of one lattice
// Most time steps of a launch, and the CTAs of kMarchWarps warps per SM the registers are sized for.
template <typename S> struct MarchForm {
    static constexpr int TMAX = 4;
    static constexpr int MINB = 2;
};
constexpr int kMarchSpan = 64;    // columns of a strip, discarded edges included
__host__ __device__ constexpr int march_edge(int t) { return (t + 1) / 2; }             // discarded lanes a side
__host__ __device__ constexpr int march_width(int t) { return kMarchSpan - 4 * march_edge(t); }   // columns stored

struct MarchEntry {
    const void* src;
    void* dst;
    long long plane;
    int nx, ny, pitch;
    int model;           // lbm::Model, extended equilibrium
    int strips;          // ceil(nx / march_width(t))
    int bands;           // bands of rows, ny / bands high; strips * bands marches, band after band
    unsigned begin;      // first CTA of this lattice
    float2 c[kNumConsts];   // the constant table, each entry twice (both halves of an F2)
};
struct MarchArgs {
    int n;
    int t;               // time steps of the launch, 1 .. TMAX
    MarchEntry e[kGroupMax];
};

__device__ __forceinline__ F2 f2_of(float2 v) { return f2_make(v.x, v.y); }
__device__ __forceinline__ F2 f2_of(float v) { return f2_make(v, v); }
// from a constant table, or one with every entry twice
template <typename E>
__device__ __forceinline__ Consts<F2> make_consts_f2(const E* t) {
    Consts<F2> c;
    c.w = f2_of(t[0]); c.w3 = f2_of(t[1]); c.w4 = f2_of(t[2]); c.rho0 = f2_of(t[3]);
    c.urx = f2_of(t[4]); c.ury = f2_of(t[5]);
    c.Xr = f2_of(t[12]); c.Yr = f2_of(t[13]);
    c.ka = f2_of(t[14]); c.kb = f2_of(t[15]); c.nkb = f2_of(t[26]);
    c.nw = f2_of(t[27]); c.nw3 = f2_of(t[28]); c.nw4 = f2_of(t[29]);
    c.nrho0 = f2_of(t[18]);
    c.ww3 = f2_of(t[19]); c.rr = f2_of(t[20]); c.qq = f2_of(t[21]);
    c.sw4 = f2_of(t[22]);
    c.nc3 = f2_of(t[23]); c.nc4 = f2_of(t[24]); c.sw1 = f2_of(t[25]);
    return c;
}

// Shared memory of a warp, in rows of 32 values (a lane only ever touches its own column, so no
// barrier is needed): the nine populations that travel from global memory, then for every level
// but the last what the next one will pull: the last two rows' three populations with xi_y = +1
// and, rolled, the last row's three with xi_y = 0.  It is kept small because what it takes of the
// SM's 256 KB is missing in the L1, where the travelling lines are allocated (measured, FP32
// 4096^2 BGK: 60 us a step with 147 KB per SM, 77 us with 184 KB, 94 us with 221 KB).
template <int TMAX, bool ROLL> constexpr int march_warp_rows = 9 + (TMAX - 1) * (ROLL ? 9 : 6);
template <typename S, bool ROLL> constexpr int march_smem_bytes =   // of one warp
    march_warp_rows<MarchForm<S>::TMAX, ROLL> * 32 * (int)sizeof(typename MarchPair<S>::type);

template <int MODEL, typename S, bool SHIFT>
__device__ __forceinline__ void march_collide(const typename MarchPair<S>::type (&in)[9],
                                              typename MarchPair<S>::type (&out)[9], const Consts<F2>& c) {
    F2 g[9], o[9], rho, ux, uy;
    // pull in x: populations with xi_x = +1 come from the left, xi_x = -1 from the right
#pragma unroll
    for (int i = 0; i < 9; ++i)
        g[i] = pair_open(ex_of(i) == 1 ? pair_from_left(in[i]) : (ex_of(i) == -1 ? pair_from_right(in[i]) : in[i]));
    collide<MODEL, 4, F2, SHIFT>(g, o, c, rho, ux, uy);
#pragma unroll
    for (int i = 0; i < 9; ++i) pair_close(out[i], o[i]);
}

// The row of level k + 1 below the row that level k just produced (o): takes what waits, leaves
// o for the next time, and collides (in place) unless that row is not complete yet.
template <int MODEL, typename S, bool SHIFT, typename Q>
__device__ __forceinline__ bool march_level(Q (&o)[9], Q (&z)[3], Q* p, bool ready, const Consts<F2>& c) {
    Q in[9];
    in[0] = z[0]; in[1] = z[1]; in[3] = z[2];
    in[2] = p[0]; in[5] = p[32]; in[6] = p[64];   // the row before last ...
    in[4] = o[4]; in[7] = o[7]; in[8] = o[8];
    z[0] = o[0]; z[1] = o[1]; z[2] = o[3];
    p[0] = o[2]; p[32] = o[5]; p[64] = o[6];      // ... makes room for this one
    if (ready) march_collide<MODEL, S, SHIFT>(in, o, c);
    return ready;
}
// Levels K + 1 .. t of the current row; true when o is a row of level t.
template <int K, int TMAX, int MODEL, typename S, bool SHIFT, typename Q>
__device__ __forceinline__ bool march_levels(Q (&o)[9], Q (&z)[TMAX][3], Q* own, int t, int i, const Consts<F2>& c) {
    if (K == t) return true;
    if constexpr (K < TMAX) {
        Q* p = own + (9 + (K - 1) * 6 + (i & 1) * 3) * 32;
        return march_level<MODEL, S, SHIFT>(o, z[K - 1], p, i >= 2 * K, c) &&
               march_levels<K + 1, TMAX, MODEL, S, SHIFT>(o, z, own, t, i, c);
    }
    return false;
}

// t time steps of the columns [x0, x0 + march_width(t)) and the rows [y0, y1) of a periodic
// lattice, from src to dst.  PAIRS: nx is even, so that a lane's two columns are neighbours in
// memory wherever the wrap in x puts them.  ROLL: the levels are a loop and everything that waits
// is in shared memory (a quarter of the code); otherwise they are unrolled and the populations
// with xi_y = 0 wait in registers.
template <int MODEL, typename S, bool SHIFT, int TMAX, bool PAIRS, bool ROLL>
__device__ __forceinline__ void march(const S* src, S* dst, int nx, int ny, int pitch, long long plane,
                                      const Consts<F2>& c, int t, int x0, int y0, int y1, int lane,
                                      typename MarchPair<S>::type* own) {
    using Q = typename MarchPair<S>::type;
    const int edge = march_edge(t);
    const int x = x0 + 2 * (lane - edge);
    int xa = x % nx;
    xa = xa < 0 ? xa + nx : xa;
    const int xb = xa + 1 == nx ? 0 : xa + 1;   // (PAIRS: never needed)
    const bool keep = lane >= edge && lane < 32 - edge && x < nx;
    // level 1 starts t - 1 rows below y0 and pulls from the rows around its own
    int yp = (y0 - t) % ny;
    yp = yp < 0 ? yp + ny : yp;
    long long om, oc, op = (long long)yp * pitch;
    auto advance = [&] {
        om = oc;
        oc = op;
        yp = yp + 1 == ny ? 0 : yp + 1;
        op = yp == 0 ? 0ll : op + pitch;
    };
    oc = 0;
    advance();
    advance();
    const int n = (y1 - y0) + 2 * (t - 1);   // rows of level 1
    auto fetch = [&] {   // the populations that level 1's next row pulls
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S* p = src + i * plane + (ey_of(i) == 1 ? om : (ey_of(i) == -1 ? op : oc));
            if constexpr (PAIRS) pair_fetch(own + i * 32, p + xa);
            else pair_fetch2(own + i * 32, p + xa, p + xb);
        }
        fetch_commit();
    };
    fetch();
    Q z[TMAX][3];
    S* out = dst + (long long)y0 * pitch + x;
#pragma unroll ROLL ? 1 : 2
    for (int i = 0; i < n; ++i) {
        Q cur[9], o[9];
        fetch_wait();
#pragma unroll
        for (int j = 0; j < 9; ++j) cur[j] = own[j * 32];
        if (i + 1 < n) {   // the next row travels while this one is collided
            advance();
            fetch();
        }
        march_collide<MODEL, S, SHIFT>(cur, o, c);
        bool done;
        if constexpr (ROLL) {
            int k = 1;
            Q* w = own + 9 * 32;
#pragma unroll 1
            for (; k < t; ++k, w += 9 * 32) {
                Q zk[3] = {w[0], w[32], w[64]};
                const bool ready = march_level<MODEL, S, SHIFT>(o, zk, w + (3 + (i & 1) * 3) * 32, i >= 2 * k, c);
                w[0] = zk[0]; w[32] = zk[1]; w[64] = zk[2];
                if (!ready) break;
            }
            done = k == t;
        } else {
            done = march_levels<1, TMAX, MODEL, S, SHIFT>(o, z, own, t, i, c);
        }
        if (done) {
            if (PAIRS || x + 1 < nx) {
                if (keep) {
#pragma unroll
                    for (int j = 0; j < 9; ++j) pair_store(out + j * plane, o[j]);
                }
            } else if (keep) {
#pragma unroll
                for (int j = 0; j < 9; ++j) pair_store_lo(out + j * plane, o[j]);
            }
            out += pitch;
        }
    }
}

// All lattices of a launch.  (Not persistent: a loop over tasks around the models' code costs 40-160
// bytes of spills a model.)  A CTA serves one lattice, so its model and constants are uniform over
// the CTA.  Its warps march side by side: strips overlap and their rows share lines, so that what
// one reads another finds in the caches.
template <typename S, bool SHIFT, bool PAIRS, bool ROLL>
__global__ void __launch_bounds__(32 * kMarchWarps, MarchForm<S>::MINB)
    march_kernel(const __grid_constant__ MarchArgs g) {
    // programmatic dependent launch: the next launch on the stream may be scheduled now, and this
    // one waits here until its predecessor has completed and its writes are visible
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int k = 0;
    while (k + 1 < g.n && blockIdx.x >= g.e[k + 1].begin) ++k;
    const MarchEntry& E = g.e[k];
    const int task = (int)(blockIdx.x - E.begin) * (int)(blockDim.x >> 5) + warp;
    const int band = task / E.strips;
    if (band >= E.bands) return;
    const int x0 = (task - band * E.strips) * march_width(g.t);
    const int y0 = (int)((long long)band * E.ny / E.bands), y1 = (int)((long long)(band + 1) * E.ny / E.bands);
    extern __shared__ __align__(16) unsigned char march_smem[];
    auto* own = reinterpret_cast<typename MarchPair<S>::type*>(march_smem) +
                warp * march_warp_rows<MarchForm<S>::TMAX, ROLL> * 32 + lane;
    const S* src = static_cast<const S*>(E.src);
    S* dst = static_cast<S*>(E.dst);
    const Consts<F2> c = make_consts_f2(E.c);
    asm volatile("griddepcontrol.wait;" ::: "memory");
#define LBM_MARCH(M)                                                                                              \
    march<M, S, SHIFT, MarchForm<S>::TMAX, PAIRS, ROLL>(src, dst, E.nx, E.ny, E.pitch, E.plane, c, g.t, x0, y0, y1, \
                                                        lane, own)
    switch (E.model) {
        case BGK: LBM_MARCH(BGK); break;
        case RM: LBM_MARCH(RM); break;
        case HM: LBM_MARCH(HM); break;
        case CM: LBM_MARCH(CM); break;
        case CHM: LBM_MARCH(CHM); break;
        case CUM: LBM_MARCH(CUM); break;
        case PR: LBM_MARCH(PR); break;
        default: LBM_MARCH(RR); break;
    }
#undef LBM_MARCH
}

}  // namespace lbm
