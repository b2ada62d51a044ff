// lbm_device.cuh -- device building blocks of the Ehrenfest-regularised
// lattice Boltzmann step (Brownlee, Gorban, Levesley 2007) for sm_103a.
//
// Layout in HBM: populations are SoA planes f[Q][ny][nxp] (x fastest, rows
// padded to nxp = round_up(nx, 32) elements so that every row starts on a
// 128-byte boundary).  Deviation storage keeps g_i = f_i - W_i rho0.
// All arithmetic is done in deviation variables (rho0 = 0 for FP64
// storage, 1 for the FP32 and FP16 forms; plain FP32 storage keeps each
// population as its exact difference from the FP32 weight), so the same
// code serves FP64, FP32 and the FP32/FP16 deviation forms.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace lbm {

// ---------------------------------------------------------------------------
// Lattices (Sec. 4.1: D1Q3 {0, -1, +1}; Sec. 4.2: D2Q9 0 rest, 1..4 E N W S,
// 5..8 NE NW SW SE, weights 4/9, 1/9, 1/36).  D1Q3 weights 2/3, 1/6, 1/6 are
// those of the rest-state quasiequilibrium of Sec. 4.1.
// ---------------------------------------------------------------------------
struct D2Q9 {
    static constexpr int Q = 9;
    __host__ __device__ static constexpr int cx(int i) {
        return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
    }
    __host__ __device__ static constexpr int cy(int i) {
        return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
    }
    __host__ __device__ static constexpr double w(int i) {
        return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
    }
    // population with the opposite velocity / with v_y reversed
    __host__ __device__ static constexpr int opp(int i) {
        return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5);
    }
    __host__ __device__ static constexpr int mir_y(int i) {
        return i == 2 ? 4 : i == 4 ? 2 : i == 5 ? 8 : i == 8 ? 5 : i == 6 ? 7 : i == 7 ? 6 : i;
    }
    static constexpr double sum_w_c2 = 2.0 / 3.0;   // sum_i W_i |v_i|^2
};

struct D1Q3 {
    static constexpr int Q = 3;
    __host__ __device__ static constexpr int cx(int i) { return i == 1 ? -1 : (i == 2 ? 1 : 0); }
    __host__ __device__ static constexpr int cy(int) { return 0; }
    __host__ __device__ static constexpr double w(int i) { return i == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
    __host__ __device__ static constexpr int opp(int i) { return i == 0 ? 0 : 3 - i; }
    __host__ __device__ static constexpr int mir_y(int i) { return i; }
    static constexpr double sum_w_c2 = 1.0 / 3.0;
};

static_assert(D2Q9::opp(1) == 3 && D2Q9::opp(2) == 4 && D2Q9::opp(3) == 1 && D2Q9::opp(4) == 2,
              "D2Q9 opposite of unit speeds");
static_assert(D2Q9::opp(5) == 7 && D2Q9::opp(6) == 8 && D2Q9::opp(7) == 5 && D2Q9::opp(8) == 6,
              "D2Q9 opposite of diagonals");

// ---------------------------------------------------------------------------
// Run parameters (passed by value to every kernel).
// ---------------------------------------------------------------------------
enum : int { EQ_POLY = 0, EQ_ENTROPIC = 1, EQ_ENERGY = 2, EQ_ENERGY_MLP = 3 };
enum : int { BC_BB = 0, BC_FREESLIP = 1, BC_INLET = 2, BC_OUTLET = 3, BC_PERIODIC = 4, BC_OUTLET_COPY = 5 };
enum : int { WALL_BOUNCE_BACK = 0, WALL_DIFFUSE = 1 };
enum : unsigned { ERR_NONFINITE = 1u, ERR_NEWTON = 2u, ERR_TIMEOUT = 4u, ERR_REPLAY = 8u };

struct Params {
    int nx, ny, nxp;
    long long plane;          // ny * nxp elements
    int eq;
    double beta, delta, rho0;
    float betaf, deltaf, rho0f;   // the same in FP32 (no FP64 work in FP32 kernels)
    int k;
    int bc[4];
    double rho_in, ux_in, uy_in;
    double gin[9];            // inlet populations f*(rho_in, u_in) in FP64, as the storage holds them
    int ox0, oy0, ow, oh;
    const void* src;          // post-collision populations of step t-1 (or pre-collision if prestream)
    void* dst;                // post-collision populations of step t
    int prestream;            // src holds pre-collision populations at their own sites
    // candidates and selection
    unsigned long long* cand_key;
    unsigned* cand_idx;
    unsigned* cand_count;
    int cand_per_block;
    int* sel_idx;
    unsigned long long* sel_key;   // keys of the selected candidates (written when not null)
    int* sel_count;
    // logs
    int* count_ring;
    double* probe_ring;
    int ring_cap;
    int probe_x, probe_y;
    long long* step;
    unsigned* err;
    // replay of given selections
    const int* replay_cnt;
    const long long* replay_off;
    const int* replay_idx;
    long long replay_t0, replay_n;
    // precision form: FP64 recheck of dS within recheck_band of delta
    int recheck;
    double recheck_band;
    // energy form
    const float* mlp;         // device copy of the network (FP32 master; rounded to BF16 at use)
    unsigned long long* newton_stats;   // it32, it64, sites, fails
    // completion ticket of the stream-collide blocks (the last block selects)
    unsigned* ticket;
    int grid_blocks;          // persistent grid size (resident blocks x SMs)
    unsigned* tile_counter;   // next tile to hand out (staged shapes)
    const int* tile_order;    // staged shapes: tile of each claim (null: row-major)
    int elbm;                 // ELBM collision (elbmLB) instead of LBGK (entropic f* only)
    int wall;                 // rule on the obstacle's faces: WALL_BOUNCE_BACK / WALL_DIFFUSE
    // slab of a run sharded in x: only columns [own_x0, own_x1) are the
    // slab's sites (the others are ghost copies of the neighbours' columns);
    // the stream-collide launch ends with the slab's own k best candidates
    // (select only), the global selection being applied afterwards
    int slab, own_x0, own_x1;
    int pad_[2];              // size a multiple of 16 bytes (bulk copies)
};

template <int Q, typename T> struct PopArr { T v[Q]; };

// ---------------------------------------------------------------------------
// Storage traits: load / store a population as a deviation in type T.
// ---------------------------------------------------------------------------
// kProject: the collision removes the rounding defects of the conserved
// moments of f - f* (conserve_neq below) -- FP32 storage, whose arithmetic
// error would otherwise exceed the storage rounding; FP64 arithmetic is
// exact enough, and FP16 storage rounding dominates its FP32 arithmetic.
// kPlain: plain FP32 storage (plain32): each population f is held as an FP32
// value, kept in the buffer as its exact difference g = f - fl32(W_i) from
// the FP32 weight, so that the FP32 arithmetic works on deviations for
// every FP32 form.
struct plain32 {
    float v;
};
template <typename S> struct Store;
template <> struct Store<double> {
    using T = double;
    static constexpr bool kProject = false, kPlain = false;
    __device__ static T load(const void* p, long long i) { return static_cast<const double*>(p)[i]; }
    __device__ static void store(void* p, long long i, T v) { static_cast<double*>(p)[i] = v; }
};
template <> struct Store<float> {
    using T = float;
    static constexpr bool kProject = true, kPlain = false;
    __device__ static T load(const void* p, long long i) { return static_cast<const float*>(p)[i]; }
    __device__ static void store(void* p, long long i, T v) { static_cast<float*>(p)[i] = v; }
};
template <> struct Store<plain32> {
    using T = float;
    static constexpr bool kProject = true, kPlain = true;
    __device__ static T load(const void* p, long long i) { return static_cast<const float*>(p)[i]; }
    __device__ static void store(void* p, long long i, T v) { static_cast<float*>(p)[i] = v; }
};
template <> struct Store<__half> {
    using T = float;
    static constexpr bool kProject = false, kPlain = false;
    __device__ static T load(const void* p, long long i) {
        return __half2float(static_cast<const __half*>(p)[i]);
    }
    __device__ static void store(void* p, long long i, T v) {
        static_cast<__half*>(p)[i] = __float2half_rn(v);
    }
};

// ---------------------------------------------------------------------------
// Geometry helpers.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool is_solid(const Params& P, int x, int y) {
    return P.ow > 0 && x >= P.ox0 && x < P.ox0 + P.ow && y >= P.oy0 && y < P.oy0 + P.oh;
}

// ---------------------------------------------------------------------------
// Quasiequilibria as deviations gs_i = f*_i - W_i rho0 in type T.
// ---------------------------------------------------------------------------

// Polynomial (Sec. 4.1 for D1Q3; standard second-order D2Q9 form).
// gs_i = W_i (drho + rho (3 c.u + 9/2 (c.u)^2 - 3/2 u^2)).
// The library is compiled without automatic multiply-add contraction; every
// fused multiply-add is written out, so each kernel that evaluates these
// functions produces the same bits (bit-exact checkpoint / resume).
template <typename T> constexpr bool kF64 = false;
template <> constexpr bool kF64<double> = true;

// Two FP32 values, one per site of a pair, worked on by the packed FP32
// instructions of sm_100 on (add, mul and fma .f32x2): each half is rounded as
// the scalar instruction rounds it, so a pair gives the bits of two scalar
// evaluations.  They take one issue slot for two results (measured 64
// instructions per SM and clock against 117 - 128 scalar ones: the FP32
// pipes' rate is the same), which leaves the other slots to loads,
// conversions and integer work.
// (The host versions only let the shared templates compile.)
#define LBM_HD __host__ __device__ __forceinline__
struct __align__(8) f2 {
    float x, y;
    f2() = default;
    LBM_HD f2(float a, float b) : x(a), y(b) {}
    LBM_HD explicit f2(float a) : x(a), y(a) {}
    LBM_HD explicit f2(double a) : x((float)a), y((float)a) {}
    LBM_HD explicit f2(int a) : x((float)a), y((float)a) {}
};
#ifdef __CUDA_ARCH__
__device__ __forceinline__ unsigned long long f2_pack(f2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ f2 f2_unpack(unsigned long long r) {
    f2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
#endif
LBM_HD f2 f2_fma(f2 a, f2 b, f2 c) {
#ifdef __CUDA_ARCH__
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_pack(a)), "l"(f2_pack(b)), "l"(f2_pack(c)));
    return f2_unpack(d);
#else
    return f2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
LBM_HD f2 operator+(f2 a, f2 b) {
#ifdef __CUDA_ARCH__
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_pack(a)), "l"(f2_pack(b)));
    return f2_unpack(d);
#else
    return f2(a.x + b.x, a.y + b.y);
#endif
}
LBM_HD f2 operator*(f2 a, f2 b) {
#ifdef __CUDA_ARCH__
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_pack(a)), "l"(f2_pack(b)));
    return f2_unpack(d);
#else
    return f2(a.x * b.x, a.y * b.y);
#endif
}
LBM_HD f2 operator-(f2 a, f2 b) { return f2_fma(b, f2(-1.0f), a); }   // a - b, rounded once
LBM_HD f2 operator-(f2 a) { return a * f2(-1.0f); }
#undef LBM_HD

template <typename T> __host__ __device__ __forceinline__ T dfma(T a, T b, T c);
template <> __host__ __device__ __forceinline__ float dfma<float>(float a, float b, float c) { return fmaf(a, b, c); }
template <> __host__ __device__ __forceinline__ double dfma<double>(double a, double b, double c) { return fma(a, b, c); }
template <> __host__ __device__ __forceinline__ f2 dfma<f2>(f2 a, f2 b, f2 c) { return f2_fma(a, b, c); }

// v . u for lattice velocity components in {-1, 0, 1}: additions only.
template <typename L, typename T>
__host__ __device__ __forceinline__ T cdotu(int i, T ux, T uy) {
    const T a = L::cx(i) == 1 ? ux : -ux;
    const T b = L::cy(i) == 1 ? uy : -uy;
    if (L::cx(i) == 0) return L::cy(i) == 0 ? T(0) : b;
    if (L::cy(i) == 0) return a;
    return a + b;
}

// Populations i and opp(i) share (v.u)^2 and have opposite v.u, so each
// pair is evaluated once: gs = W (c0 + 9/2 rho (v.u)^2) +- W 3 rho (v.u),
// c0 = drho - 3/2 rho u^2.
template <typename L, typename T>
__host__ __device__ __forceinline__ void feq_poly(T drho, T rho, T ux, T uy, T* gs) {
    const T usq = dfma<T>(ux, ux, uy * uy);
    const T c0 = dfma<T>(T(-1.5) * rho, usq, drho);
    const T r45 = T(4.5) * rho, r3 = T(3) * rho;
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        if (i == 0) {
            gs[0] = T(L::w(0)) * c0;
        } else if (i < L::opp(i)) {
            const T cu = cdotu<L, T>(i, ux, uy);
            const T w = T(L::w(i));
            const T a = dfma<T>(r45 * cu, cu, c0);
            const T b = r3 * cu;
            gs[i] = w * (a + b);
            gs[L::opp(i)] = w * (a - b);
        }
    }
}

// Run parameters in the arithmetic type T.
template <typename T> struct Par;
template <> struct Par<float> {
    __device__ static float beta(const Params& P) { return P.betaf; }
    __device__ static float delta(const Params& P) { return P.deltaf; }
    __device__ static float rho0(const Params& P) { return P.rho0f; }
};
template <> struct Par<double> {
    __device__ static double beta(const Params& P) { return P.beta; }
    __device__ static double delta(const Params& P) { return P.delta; }
    __device__ static double rho0(const Params& P) { return P.rho0; }
};

// ---------------------------------------------------------------------------
// Stored values and the deviations the arithmetic works on.  FP64 storage
// holds f (rho0 = 0); FP32 / FP16 deviation storage holds g = f - W_i rho0
// (rho0 = 1); plain FP32 storage holds the FP32 value of f, kept as the
// exact difference g = f - fl32(W_i).  FP32 arithmetic takes rho0 = 1 for
// every FP32 / FP16 form.
// ---------------------------------------------------------------------------

// FP32 to FP64 by integer operations: the conversion instruction runs on the
// FP64 pipe (two per SM and clock), and does so even where a predicate turns
// it off.  Subnormal values are scaled by 2^64 first; exponent 255 (infinity,
// NaN) becomes 2047.
__device__ __forceinline__ double widen(float x) {
    const bool small = (__float_as_uint(x) & 0x7fffffffu) < 0x00800000u;
    const unsigned b = __float_as_uint(small ? x * 0x1p64f : x), m = b & 0x7fffffffu;
    unsigned e = small ? (896u - 64u) << 20 : 896u << 20;
    if (m >= 0x7f800000u) e = 1792u << 20;
    if (m == 0u) e = 0u;
    return __hiloint2double((int)(((m >> 3) + e) | (b & 0x80000000u)), (int)(b << 29));
}

// FP64 value of population i whose stored deviation is g (FP64 storage holds
// f itself, the deviation forms have rho0 = 1).
template <typename L, typename S>
__device__ __forceinline__ double pop_f64(int i, typename Store<S>::T g) {
    if constexpr (sizeof(typename Store<S>::T) == 8) return g;
    else if constexpr (Store<S>::kPlain) return widen(g) + (double)(float)L::w(i);
    else return widen(g) + L::w(i);
}

// Deviation of a population whose value f was computed in FP64 (initial and
// imported states), as a stored field holds it: plain FP32 rounds f, the
// deviation forms round f - W_i rho0.
template <typename L, typename S>
__device__ __forceinline__ typename Store<S>::T dev_of_f64(const Params& P, int i, double f) {
    using T = typename Store<S>::T;
    if constexpr (Store<S>::kPlain) return (float)f - (float)L::w(i);
    else return (T)(f - L::w(i) * P.rho0);
}

// A deviation computed in the arithmetic, rounded as the storage rounds it:
// plain FP32 storage rounds f = g + fl32(W_i) to FP32 (the difference with
// fl32(W_i) is then exact when f lies within a factor two of W_i); the other
// forms round at the store itself.
template <typename L, typename S>
__device__ __forceinline__ typename Store<S>::T store_round(int i, typename Store<S>::T g) {
    if constexpr (Store<S>::kPlain) {
        const float w = (float)L::w(i);
        return (g + w) - w;
    } else {
        (void)i;
        return g;
    }
}

// Conserved moments of the nonequilibrium part d = f - f*: zero in exact
// arithmetic, since f* has the conserved moments of f (mass and momentum
// (lbgkLB), and the energy 2E for the energy-constrained quasiequilibrium,
// Sec. 3.3).  The FP32 evaluation of f* leaves errors of a few ulps in each
// f*_i, whose sums the over-relaxed collision f' = f - 2 beta d (beta ~ 1)
// would turn into a drift of the conserved quantities by about twice their
// value per step, the same at every site of a smooth flow.  They are removed
// by subtracting the combination W_i (a + b . v_i + e |v_i|^2) of the
// collision invariants that has the same moments as d (D2Q9: sum W = 1,
// sum W v v = I/3, sum W |v|^2 = 2/3, sum W |v|^4 = 8/9; e = 0 without the
// energy constraint; D1Q3: sum W v^2 = 1/3).  The sums are of the small
// nonequilibrium parts, so the conserved moments of the result are exact to
// their rounding; in exact arithmetic nothing changes.
template <typename L, int EQ, typename T>
__device__ __forceinline__ void conserve_neq(T* d) {
    if constexpr (L::Q == 9) {
        const T D0 = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
        const T Dx = ((d[1] - d[3]) + (d[5] - d[6])) + (d[8] - d[7]);
        const T Dy = ((d[2] - d[4]) + (d[5] - d[8])) + (d[6] - d[7]);
        T a = D0, e = T(0.0f);
        if constexpr (EQ >= EQ_ENERGY) {
            const T DE = ((d[1] + d[2]) + (d[3] + d[4])) + T(2.0f) * ((d[5] + d[6]) + (d[7] + d[8]));
            a = dfma<T>(T(-1.5f), DE, T(2.0f) * D0);     // a = 2 D0 - 3/2 DE
            e = dfma<T>(T(2.25f), DE, T(-1.5f) * D0);    // e = 9/4 DE - 3/2 D0
        }
        // W_i (a + 3 v_i . D + e |v_i|^2), weights 4/9, 1/9, 1/36
        const T m1 = (a + e) * T(1.0f / 9.0f), px = Dx * T(1.0f / 3.0f), py = Dy * T(1.0f / 3.0f);
        const T m5 = dfma<T>(T(2.0f), e, a) * T(1.0f / 36.0f), qx = Dx * T(1.0f / 12.0f), qy = Dy * T(1.0f / 12.0f);
        d[0] = d[0] - a * T(4.0f / 9.0f);
        d[1] = d[1] - (m1 + px);
        d[3] = d[3] - (m1 - px);
        d[2] = d[2] - (m1 + py);
        d[4] = d[4] - (m1 - py);
        const T s1 = m5 + qy, s2 = m5 - qy;
        d[5] = d[5] - (s1 + qx);
        d[6] = d[6] - (s1 - qx);
        d[7] = d[7] - (s2 - qx);
        d[8] = d[8] - (s2 + qx);
    } else {
        const T D0 = (d[0] + d[1]) + d[2];
        const T Dx = d[2] - d[1];
        const T m = D0 * T(1.0f / 6.0f), p = Dx * T(0.5f);   // W (D0 + 3 v Dx), W = 1/6
        d[0] = d[0] - D0 * T(2.0f / 3.0f);
        d[1] = d[1] - (m - p);
        d[2] = d[2] - (m + p);
    }
}

// 1 / x: FP32 from the hardware approximation refined by one Newton-Raphson
// step r + r (1 - x r) (the relative error e of the seed becomes ~e^2, below
// one ulp); FP64 from the hardware's approximation r0 (special function
// unit, not the FP64 pipe), with e = 1 - x r0: r0 (1 + e + e^2), whose error
// e^3 is below 2^-57 -- three FP64 operations instead of a division's ten.
template <typename T> __host__ __device__ __forceinline__ T recip(T x);
template <> __host__ __device__ __forceinline__ float recip<float>(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
#else
    return 1.0f / x;
#endif
}
template <> __host__ __device__ __forceinline__ double recip<double>(double x) {
#ifdef __CUDA_ARCH__
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
#else
    return 1.0 / x;
#endif
}

template <> __host__ __device__ __forceinline__ f2 recip<f2>(f2 x) {
    return f2(recip<float>(x.x), recip<float>(x.y));
}

// sigma = sqrt(1 + q) - 1, q >= 0, to the rounding of sigma itself (a square
// root rounded near 1 leaves an error that is the same at every site of a quiet
// region, and it adds up).  FP32: q / (1 + sqrt(1 + q)).  FP64: from the
// hardware's approximation r of 1 / sqrt(x), x = 1 + q: with s = x r,
// e = 1 - s r and the residual d = q - (s - 1) (s + 1),
// sigma = s - 1 + d r (1/2 + 3/8 e) up to e^3 (below 2^-57) -- nine FP64
// operations.  Against extended precision the f* of it are 42 % (D1Q3) and 33 %
// (D2Q9) closer than the printed formula in correctly rounded FP64.
template <typename T> __host__ __device__ __forceinline__ T root_excess(T q);
template <> __host__ __device__ __forceinline__ float root_excess<float>(float q) {
    return q * recip<float>(1.0f + sqrtf(1.0f + q));
}
template <> __host__ __device__ __forceinline__ double root_excess<double>(double q) {
#ifdef __CUDA_ARCH__
    const double x = 1.0 + q;
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double s = x * r, e = fma(-s, r, 1.0), s0 = s - 1.0, d = fma(-s0, s + 1.0, q);
    return fma(d * r, fma(0.375, e, 0.5), s0);
#else
    return q / (1.0 + sqrt(1.0 + q));
#endif
}
template <> __host__ __device__ __forceinline__ f2 root_excess<f2>(f2 q) {
    const f2 x = f2(1.0f) + q;
    return q * recip<f2>(f2(1.0f) + f2(sqrtf(x.x), sqrtf(x.y)));
}

// Entropic for mass and momentum, by axis.  Sec. 4.1's closed form (with the
// left/right labels read so that the momentum is +rho u) is rho times
//   rest (2/3)(2 - s), moving (1/6)(2 s - 1 +- 3 u), s = sqrt(1 + 3 u^2),
// and the product formula of Sec. 4.2 is the product of two such axes: its
// factors are (2 - s) ((2 u + s) / (1 - u))^{+-1} = 2 s - 1 +- 3 u, as
// (2 - s)(2 + s) = 3 (1 - u^2).  With sigma = s - 1 = 3 u^2 / (1 + s) an axis's
// factors are 1 + A, A = -sigma (rest), 2 sigma +- 3 u, so
//   f*_i - W_i rho0 = W_i (drho + rho (A + B + A B)),  drho = rho - rho0,
// without the cancellation of f*_i - W_i rho0 and without divisions (the
// printed form takes six; in FP32 an update took 290 instructions with it).
template <typename T>
__host__ __device__ __forceinline__ void entropic_axis(T u, T* A) {
    const T u3 = T(3) * u;
    const T sigma = root_excess<T>(u3 * u);
    A[0] = -sigma;
    const T two = sigma + sigma;
    A[1] = two + u3;
    A[2] = two - u3;
}
// ZERO0: the caller's rho0 is zero (FP64 storage; drho = rho).
template <typename L, typename T, bool ZERO0 = false>
__host__ __device__ __forceinline__ void feq_entropic(T drho, T rho, T ux, T uy, T* gs) {
    if constexpr (L::Q == 3 && kF64<T>) {
        // the printed form on rho / 6, correctly rounded (quotient, residual,
        // correction): a rounded weight's error would be the same at every
        // site and step, a drift of the mass (5e-14 after 500 steps)
        const T c = T(1.0 / 6.0), q = rho * c, r6 = dfma<T>(dfma<T>(T(-6), q, rho), c, q);
        const T u3 = T(3) * ux, sigma = root_excess<T>(u3 * ux);
        const T a = dfma<T>(T(2), sigma, T(1));   // 2 s - 1
        gs[0] = T(4) * r6 * (T(1) - sigma);
        gs[1] = r6 * (a - u3);
        gs[2] = r6 * (a + u3);
        if constexpr (!ZERO0)
            for (int i = 0; i < 3; i++) gs[i] -= T(L::w(i)) * (rho - drho);
        return;
    }
    T A[3];
    entropic_axis<T>(ux, A);
    if constexpr (L::Q == 3) {
        // populations rest, left, right
        gs[0] = T(L::w(0)) * dfma<T>(rho, A[0], drho);
        gs[1] = T(L::w(1)) * dfma<T>(rho, A[2], drho);
        gs[2] = T(L::w(2)) * dfma<T>(rho, A[1], drho);
    } else {
        T B[3], R[3], D[3];
        entropic_axis<T>(uy, B);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R[j] = rho * A[j];
            D[j] = dfma<T>(rho, B[j], drho);
        }
#pragma unroll
        for (int i = 0; i < L::Q; i++) {
            const int j = L::cx(i) < 0 ? 2 : L::cx(i), k = L::cy(i) < 0 ? 2 : L::cy(i);
            gs[i] = T(L::w(i)) * dfma<T>(R[j], B[k], R[j] + D[k]);
        }
    }
}

// Boundary equilibrium from (rho, u): polynomial or entropic formula (the
// energy forms use the isothermal entropic formula, whose energy
// multiplier is zero).
template <typename L, typename T>
__host__ __device__ __forceinline__ void feq_rho_u(int eq, T rho, T ux, T uy, T rho0, T* gs) {
    if (eq == EQ_POLY) feq_poly<L, T>(rho - rho0, rho, ux, uy, gs);
    else feq_entropic<L, T>(rho - rho0, rho, ux, uy, gs);
}

// ---------------------------------------------------------------------------
// Nonequilibrium entropy (DelS).
// With x_i = (f_i - f*_i) / f*_i and phi(x) = (1+x) ln(1+x) - x >= 0,
//   sum_i f*_i phi(x_i) = sum_i f_i ln(f_i/f*_i) - sum_i (f_i - f*_i),
// which is dS because f and f* share their density.  The phi form has no
// first-order cancellation.  phi is evaluated by its Taylor series
// sum_{n>=2} (-1)^n x^n / (n (n-1)) for small |x| and from log1p otherwise.
// Outside the positive cone (some f_i < 0 or f*_i <= 0) dS = +inf.
// ---------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ T phi_fn(T x);

template <> __device__ __forceinline__ float phi_fn<float>(float x) {
    if (fabsf(x) <= 0.25f) {
        // terms n = 2..13; truncation < 1e-9 relative at |x| = 1/4
        float p = -1.0f / 156.0f;
        p = fmaf(p, x, 1.0f / 132.0f);
        p = fmaf(p, x, -1.0f / 110.0f);
        p = fmaf(p, x, 1.0f / 90.0f);
        p = fmaf(p, x, -1.0f / 72.0f);
        p = fmaf(p, x, 1.0f / 56.0f);
        p = fmaf(p, x, -1.0f / 42.0f);
        p = fmaf(p, x, 1.0f / 30.0f);
        p = fmaf(p, x, -1.0f / 20.0f);
        p = fmaf(p, x, 1.0f / 12.0f);
        p = fmaf(p, x, -1.0f / 6.0f);
        p = fmaf(p, x, 0.5f);
        return x * x * p;
    }
    if (x <= -1.0f) return 1.0f;  // f_i = 0: 0 ln 0 - (0 - f*) = f*
    return fmaf(1.0f + x, log1pf(x), -x);
}

// (FP64 takes 64 cycles per warp instruction and SM quarter, whatever the
// lanes or the dependences: what counts is the number of operations, over
// both branches when a warp's lanes take both.  log1p alone takes about as many
// as both sums here.)
template <> __device__ __forceinline__ double phi_fn<double>(double x) {
    if (fabs(x) <= 0.0625) {
        // terms n = 2..17; truncation < 1e-18 relative at |x| = 1/16
        double p = 0.0;
#pragma unroll
        for (int n = 17; n >= 2; n--) {
            const double c = ((n & 1) ? -1.0 : 1.0) / (double(n) * double(n - 1));
            p = n == 17 ? c : fma(p, x, c);
        }
        return x * x * p;
    }
    if (x >= -0.5 && x <= 1.0) {
        // ln(1 + x) = 2 artanh(t), t = x / (2 + x): |t| <= 1/3, artanh(t) =
        // t sum t^{2k} / (2k + 1), k <= 16 (truncation < 2e-18)
        const double t = x * recip<double>(2.0 + x), z = t * t;
        double q = 1.0 / 33.0;
#pragma unroll
        for (int k = 15; k >= 0; k--) q = fma(q, z, 1.0 / double(2 * k + 1));
        return fma((1.0 + x) * (t + t), q, -x);
    }
    if (x <= -1.0) return 1.0;
    return fma(1.0 + x, log1p(x), -x);
}

// Exact dS of one site in type T; +inf outside the positive cone.
template <typename L, typename T>
__device__ __forceinline__ T delta_s_exact(const T* g, const T* gs, T rho0) {
    bool bad = false;
    T x[L::Q], fs[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        fs[i] = dfma<T>(T(L::w(i)), rho0, gs[i]);
        const T f = dfma<T>(T(L::w(i)), rho0, g[i]);
        bad |= !(fs[i] > T(0)) || (f < T(0));
        if constexpr (kF64<T>) x[i] = (g[i] - gs[i]) * recip<T>(fs[i]);
        else x[i] = (g[i] - gs[i]) / fs[i];
    }
    if (bad) return T(INFINITY);
    T s = T(0);
#pragma unroll
    for (int i = 0; i < L::Q; i++) s = dfma<T>(fs[i], phi_fn<T>(x[i]), s);
    return s;
}

// Out-of-line copy for the rare sites that the bound below does not clear.
template <typename L, typename T>
__device__ __noinline__ T delta_s_slow(PopArr<L::Q, T> g, PopArr<L::Q, T> gs, T rho0) {
    return delta_s_exact<L, T>(g.v, gs.v, rho0);
}

// Division-free bound that clears a site (dS <= delta) without evaluating
// dS.  With d_i = f_i - f*_i, x_i = d_i / f*_i and m <= min_i f*_i / W_i:
//   Q = sum_i d_i^2 / W_i >= m sum_i d_i^2 / f*_i  and  x_i^2 <= Q / (W_min m^2),
// so Q <= m^2 W_min / 16 gives |x_i| <= 1/4 (hence f_i > 0), where
// phi(x) <= 0.5478 x^2, and then dS = sum f* phi(x) <= 0.55 Q / m.
// The site is cleared when m > 0, 16 Q <= W_min m^2 and 0.55 Q <= delta m.
// Polynomial f*: f*_i / W_i = rho (1 + 3 v.u + 9/2 (v.u)^2 - 3/2 u^2) >=
// rho (1 - 3 (|u_x| + |u_y|) - 3/2 u^2) = m.  Other f*: m = min_i f*_i / W_i.
// FP64 storage evaluates the bound in FP32 (FP64 operations are what its
// update is bound by), with magnitudes cut to 20 bits (abs_float, integer
// operations) and a relative margin of 2^-16 on each side, far above the
// roundings: a site is cleared only if the FP64 bound clears it too, and one
// near the limit gets its exact dS as any other site that is not cleared.
// The populations, f* and delta enter divided by the power of two of the
// site's density (dS is linear in it), so that the bound holds at every
// density FP64 represents.  Squares that FP32 loses (|d| below 2^-60 of the
// density) are covered by a floor of Q, 2^-99 unless every d is zero; m is
// kept above 2^-40, where m^2 and the floor are far from FP32's limits.

// |x| / 2^s as FP32, truncated to 20 significant bits (0 below 2^-126, infinity
// from 2^128 on and for NaN), without an FP64 operation.  scale: (s + 896) << 20.
constexpr int kNoScale = 896 << 20;
__device__ __forceinline__ float abs_float(double x, int scale) {
    const int h = __double2hiint(x) & 0x7fffffff;
    return __int_as_float(min(max(h - scale, 0), 0x0ff00000) << 3);
}

template <typename L, typename T, int EQ>
__device__ __forceinline__ bool ds_cleared(const T* d, const T* gs, T rho, T ux, T uy, T rho0, T delta) {
    // the bound's arithmetic type
    constexpr bool narrow = kF64<T>;
    using B = float;
    int scale = kNoScale;   // of the density (not below 2^-896: the difference in abs_float stays in range)
    if constexpr (narrow) scale = max((__double2hiint(rho) & 0x7ff00000) - (127 << 20), 0);
    B q0 = B(0), q1 = B(0), q2 = B(0);
    int any = 0;   // bits of the d
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        B di;
        if constexpr (narrow) {
            di = abs_float(d[i], scale);
            any |= (__double2hiint(d[i]) & 0x7fffffff) | __double2loint(d[i]);
        } else {
            di = d[i];
        }
        if (L::w(i) == L::w(0)) q0 = fmaf(di, di, q0);
        else if (L::w(i) == L::w(1)) q1 = fmaf(di, di, q1);
        else q2 = fmaf(di, di, q2);
    }
    constexpr double wmin = L::Q == 9 ? 1.0 / 36.0 : 1.0 / 6.0;
    B Q = fmaf(q0, B(1.0 / L::w(0)), fmaf(q1, B(1.0 / L::w(1)), L::Q == 9 ? q2 * B(1.0 / L::w(5)) : B(0)));
    B m;
    if constexpr (narrow) {
        if constexpr (EQ == 0) {
            const B vx = abs_float(ux, kNoScale) * B(1.0 + 0x1p-18), vy = abs_float(uy, kNoScale) * B(1.0 + 0x1p-18);
            m = abs_float(rho, scale) * fmaf(B(-1.5), fmaf(vx, vx, vy * vy), fmaf(B(-3), vx + vy, B(1)));
        } else {
            m = B(INFINITY);
#pragma unroll
            for (int i = 0; i < L::Q; i++)
                m = fminf(m, gs[i] > T(0) ? abs_float(gs[i], scale) * B(1.0 / L::w(i)) : B(-1));
        }
        Q = any ? fmaxf(Q * B(1.0 + 0x1p-16), B(0x1p-99)) : B(0);
        m *= B(1.0 - 0x1p-16);
        const B ad = abs_float(delta, scale);
        const B dl = delta > T(0) ? ad * B(1.0 - 0x1p-16) : ad * B(-1.0 - 0x1p-16);
        return (rho > T(0)) & (m > B(0x1p-40)) & (B(16.0 / wmin) * Q <= m * m) & (B(0.55) * Q <= dl * m);
    } else {
        if constexpr (EQ == 0) {
            const B usq = fmaf(ux, ux, uy * uy);
            m = rho * fmaf(B(-1.5), usq, fmaf(B(-3), fabsf(ux) + fabsf(uy), B(1)));
        } else {
            m = B(INFINITY);
#pragma unroll
            for (int i = 0; i < L::Q; i++) m = fminf(m, fmaf(gs[i], B(1.0 / L::w(i)), rho0));
        }
        return (m > B(0)) && (B(16.0 / wmin) * Q <= m * m) && (B(0.55) * Q <= delta * m);
    }
}

// The bound for a pair of sites, the same operations half by half: bit 0 and
// bit 1 set where the pair's first and second site are cleared.
template <typename L, int EQ>
__device__ __forceinline__ unsigned ds_cleared_pair(const f2* d, const f2* gs, f2 rho, f2 ux, f2 uy, float rho0,
                                                    float delta) {
    f2 q0(0.0f), q1(0.0f), q2(0.0f);
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        if (L::w(i) == L::w(0)) q0 = f2_fma(d[i], d[i], q0);
        else if (L::w(i) == L::w(1)) q1 = f2_fma(d[i], d[i], q1);
        else q2 = f2_fma(d[i], d[i], q2);
    }
    constexpr double wmin = 1.0 / 36.0;
    const f2 Q = f2_fma(q0, f2(1.0 / L::w(0)), f2_fma(q1, f2(1.0 / L::w(1)), q2 * f2(1.0 / L::w(5))));
    f2 m;
    if constexpr (EQ == 0) {
        const f2 usq = f2_fma(ux, ux, uy * uy), a(fabsf(ux.x), fabsf(ux.y)), b(fabsf(uy.x), fabsf(uy.y));
        m = rho * f2_fma(f2(-1.5f), usq, f2_fma(f2(-3.0f), a + b, f2(1.0f)));
    } else {
        m = f2(INFINITY);
#pragma unroll
        for (int i = 0; i < L::Q; i++) {
            const f2 v = f2_fma(gs[i], f2(1.0 / L::w(i)), f2(rho0));
            m = f2(fminf(m.x, v.x), fminf(m.y, v.y));
        }
    }
    const f2 a = f2((float)(16.0 / wmin)) * Q, b = m * m, c = f2(0.55f) * Q, e = f2(delta) * m;
    return ((m.x > 0.0f) & (a.x <= b.x) & (c.x <= e.x) ? 1u : 0u) |
           ((m.y > 0.0f) & (a.y <= b.y) & (c.y <= e.y) ? 2u : 0u);
}

// Monotone map of a double onto uint64 (larger double <=> larger key).
__device__ __forceinline__ unsigned long long ds_key(double d) {
    unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// ---------------------------------------------------------------------------
// Free flight with boundary rules (Sec. 3 map Theta_tau; Sec. 4.2).
// Pre-collision deviation populations at fluid site (x, y) from the
// post-collision field src.  Rules where x - v_i leaves the fluid:
//   x side: PERIODIC wraps, INLET = f*(rho_in, u_in) (computed once in FP64 by
//           the host, Params::gin), OUTLET = f*(rho, u of
//           column nx-2 in the same row), BB = own opposite population;
//   y side: PERIODIC wraps, FREESLIP = population (v_x, -v_y) of (x - v_x, y),
//           BB = own opposite population;
//   solid source: own opposite population (half-way bounce-back), or with
//           wall = WALL_DIFFUSE the diffuse kinetic wall (diffuse_wall).
// The x rule is applied first (inlet and outlet win at corners).
// ---------------------------------------------------------------------------

// Diffuse kinetic wall at rest (Maxwell's diffuse reflection, the kinetic
// boundary condition cited in Sec. 4.2): the wall re-emits the mass it
// absorbed as its rest quasiequilibrium W_i rho_w.  The links in mask
// (source inside the obstacle) enter holding f'_{-i}(x), the absorbed
// populations, and leave with
//   f_i = W_i (sum_{j in mask} f'_{-j}) / (sum_{j in mask} W_j).
// The same map holds for deviations g = f - W rho0 (the W_i rho0 parts
// cancel), so it applies to every storage form as it stands.
template <typename L, typename T>
__device__ __forceinline__ void diffuse_wall(unsigned mask, T* g) {
    T absorbed = T(0), wsum = T(0);
#pragma unroll
    for (int i = 0; i < L::Q; i++)
        if ((mask >> i) & 1u) {
            absorbed += g[i];
            wsum += T(L::w(i));
        }
    const T rho_w = absorbed / wsum;
#pragma unroll
    for (int i = 0; i < L::Q; i++)
        if ((mask >> i) & 1u) g[i] = T(L::w(i)) * rho_w;
}

// Quasiequilibrium f*(rho, u) evaluated in FP64 and held as the storage
// holds a population (dev_of_f64): the initial state.
template <typename L, typename S>
__device__ __forceinline__ void bc_equilibrium(const Params& P, double rho, double ux, double uy,
                                               typename Store<S>::T* g) {
    double fs[L::Q];
    feq_rho_u<L, double>(P.eq, rho, ux, uy, 0.0, fs);
#pragma unroll
    for (int i = 0; i < L::Q; i++) g[i] = dev_of_f64<L, S>(P, i, fs[i]);
}

// Outlet rule of Sec. 4.2: the quasiequilibrium of the density and velocity
// of column nx - 2 (stored deviations v), in the run's arithmetic (the
// callers round it as the storage holds a population).
template <typename L, typename T>
__device__ __forceinline__ void outlet_equilibrium(const Params& P, const T* v, T* g) {
    const T rho0 = Par<T>::rho0(P);
    T drho = T(0), jx = T(0), jy = T(0);
#pragma unroll
    for (int j = 0; j < L::Q; j++) {
        drho += v[j];
        jx += T(L::cx(j)) * v[j];
        jy += T(L::cy(j)) * v[j];
    }
    const T rho = rho0 + drho;
    feq_rho_u<L, T>(P.eq, rho, jx / rho, jy / rho, rho0, g);
}

// Sites whose nine sources lie in the fluid (almost all) load them at once.
// The others resolve every population to one load (plane, column, row) by
// selects and load them together too: the rules cost their instructions, not
// a chain of dependent branches and loads.
template <typename L, typename S>
__device__ void gather_site(const Params& P, int x, int y, typename Store<S>::T* g) {
    using T = typename Store<S>::T;
    const long long s0 = (long long)y * P.nxp + x;
    const bool inside = x >= 1 && x <= P.nx - 2 && (L::Q == 3 || (y >= 1 && y <= P.ny - 2));
    const bool near = P.ow > 0 && x >= P.ox0 - 1 && x <= P.ox0 + P.ow && y >= P.oy0 - 1 && y <= P.oy0 + P.oh;
    if (P.prestream || (inside && !near)) {
        const long long shift = P.prestream ? 0 : 1;
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            g[i] = Store<S>::load(P.src, i * P.plane + s0 - shift * (L::cy(i) * (long long)P.nxp + L::cx(i)));
        return;
    }
    unsigned wall_mask = 0u, in_mask = 0u, out_mask = 0u;
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
        const int cx = L::cx(i), cy = L::cy(i);
        // source (sx, sy) of plane i; done: the rule is settled
        int sx = x - cx, sy = y - cy;
        bool own = false, mirror = false, done = false;   // own opposite population; population (v_x, -v_y)
        if (cx != 0 && (sx < 0 || sx >= P.nx)) {
            const int kind = sx < 0 ? P.bc[0] : P.bc[1];
            if (kind == BC_INLET) in_mask |= 1u << i;
            if (kind == BC_OUTLET) out_mask |= 1u << i;
            own = kind != BC_PERIODIC && kind != BC_OUTLET_COPY;   // (inlet, outlet: replaced below)
            done = own;
            // zero-gradient outflow: the column beyond the side is a copy
            // of the side column; the y and obstacle rules then apply
            sx = kind == BC_PERIODIC ? (sx < 0 ? sx + P.nx : sx - P.nx) : x;
        }
        if (cy != 0 && !done && (sy < 0 || sy >= P.ny)) {
            const int kind = sy < 0 ? P.bc[2] : P.bc[3];
            done = kind != BC_PERIODIC;
            mirror = kind == BC_FREESLIP;
            own = done && !mirror;
            sy = kind == BC_PERIODIC ? (sy < 0 ? sy + P.ny : sy - P.ny) : y;
        }
        if (i > 0 && !done && is_solid(P, sx, sy)) {
            own = true;
            if (P.wall == WALL_DIFFUSE) wall_mask |= 1u << i;
        }
        const int plane = own ? L::opp(i) : (mirror ? L::mir_y(i) : i);
        const long long at = own ? s0 : (long long)sy * P.nxp + sx;
        g[i] = Store<S>::load(P.src, plane * P.plane + at);
    }
    if (out_mask) {
        T v[L::Q], gout[L::Q];
        const long long sp = (long long)y * P.nxp + (P.nx - 2);
#pragma unroll
        for (int j = 0; j < L::Q; j++) v[j] = Store<S>::load(P.src, j * P.plane + sp);
        outlet_equilibrium<L, T>(P, v, gout);
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            if ((out_mask >> i) & 1u) g[i] = store_round<L, S>(i, gout[i]);
    }
    if (in_mask) {
#pragma unroll
        for (int i = 0; i < L::Q; i++)
            if ((in_mask >> i) & 1u) g[i] = (T)P.gin[i];
    }
    if (wall_mask) diffuse_wall<L, T>(wall_mask, g);
}

// ---------------------------------------------------------------------------
// Block-wide top-k by radix select.
// Elements e in [0, n) with keys key[e] (uint64, larger = better) and unique
// indices idx[e]; total order (key descending, idx ascending).  The function
// finds the threshold so that exactly k (< n) elements are selected:
// selected(e) <=> (key & kmask) > kpre, or (key & kmask) == kpre and
// (all_tied or (~idx & imask) >= ipre).  Digits of 8 bits from the most
// significant differing bit down; the idx phase runs only when more than the
// needed number of elements share the exact threshold key.
// key/idx may point to shared or global memory.  All threads of the block
// must call it; scratch is shared memory supplied by the caller.
// ---------------------------------------------------------------------------
struct TopkScratch {
    unsigned hist[256];
    unsigned long long red_or[32], red_and[32];
    unsigned long long kpre, kmask;
    unsigned ipre, imask;
    int need;           // elements still to take among the tied group
    int all_tied;
    int digit;          // result of the last radix pass
    unsigned above;     // elements in digits above it
    int hi;             // most significant bit where keys differ (-1: none)
    unsigned long long diff;
};

struct Thresh {
    unsigned long long kpre, kmask;
    unsigned ipre, imask;
    int all_tied;
    __device__ __forceinline__ bool selected(unsigned long long key, unsigned id) const {
        const unsigned long long km = key & kmask;
        if (km != kpre) return km > kpre;
        if (all_tied) return true;
        return ((~id) & imask) >= ipre;
    }
};

// one radix pass over a digit [lo, lo+width) of the value returned by getv
// for elements matching the current prefix; updates prefix/need.
template <typename GetV, typename Match>
__device__ void radix_pass(TopkScratch& sc, int n, int lo, int width, GetV getv, Match match) {
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int b = tid; b < 256; b += nt) sc.hist[b] = 0;
    __syncthreads();
    const unsigned dmask = (1u << width) - 1u;
    if (tid == 0) { sc.digit = 0; sc.above = 0; }
    for (int e = tid; e < n; e += nt) {
        if (match(e)) atomicAdd(&sc.hist[(unsigned)(getv(e) >> lo) & dmask], 1u);
    }
    __syncthreads();
    if (tid < 32) {
        // bins b = 255..0 scanned from the top: lane l owns bins 8l..8l+7
        unsigned c[8], tot = 0;
#pragma unroll
        for (int j = 0; j < 8; j++) { c[j] = sc.hist[tid * 8 + j]; tot += c[j]; }
        // inclusive suffix sum over lanes (lane 31 holds the top bins)
        unsigned suf = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_down_sync(0xffffffffu, suf, o);
            if (tid + o < 32) suf += v;
        }
        unsigned above = suf - tot;   // elements in bins above this lane's bins
        const unsigned need = (unsigned)sc.need;
        // the lane whose range contains the need-th element from the top
        const bool mine = above < need && need <= suf;
        if (mine) {
            unsigned acc = above;
            for (int j = 7; j >= 0; j--) {
                if (acc + c[j] >= need) {
                    sc.digit = tid * 8 + j;
                    sc.above = acc;
                    break;
                }
                acc += c[j];
            }
        }
    }
    __syncthreads();
}

template <typename KeyAt, typename IdAt>
__device__ Thresh block_topk(TopkScratch& sc, int n, int k, KeyAt keyat, IdAt idat) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    // common bits of all keys: skip digits where every key agrees
    unsigned long long o = 0, a = ~0ull;
    for (int e = tid; e < n; e += nt) { const unsigned long long v = keyat(e); o |= v; a &= v; }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        o |= __shfl_xor_sync(0xffffffffu, o, s);
        a &= __shfl_xor_sync(0xffffffffu, a, s);
    }
    if (lane == 0) { sc.red_or[warp] = o; sc.red_and[warp] = a; }
    __syncthreads();
    if (tid == 0) {
        unsigned long long oo = 0, aa = ~0ull;
        for (int w = 0; w < (nt + 31) / 32; w++) { oo |= sc.red_or[w]; aa &= sc.red_and[w]; }
        const unsigned long long diff = oo ^ aa;
        const int hi = diff ? 63 - __clzll(diff) : -1;
        const unsigned long long above_hi = hi >= 63 ? 0ull : (~0ull << (hi + 1));
        sc.kmask = above_hi;
        sc.kpre = aa & above_hi;
        sc.need = k;
        sc.all_tied = 0;
        sc.ipre = 0;
        sc.imask = 0;
        sc.hi = hi;
        sc.diff = diff;
    }
    __syncthreads();
    const int hi = sc.hi;
    const unsigned long long diff = sc.diff;
    const int lo_bit = diff ? __ffsll((long long)diff) - 1 : 0;
    bool done = (hi < 0);   // all keys equal: go to the idx phase
    for (int top = hi; !done && top >= lo_bit; top -= 8) {
        const int lo = top - 7 > lo_bit ? top - 7 : lo_bit;
        const int width = top - lo + 1;
        const unsigned long long kpre = sc.kpre, kmask = sc.kmask;
        radix_pass(sc, n, lo, width, keyat,
                   [&](int e) { return (keyat(e) & kmask) == kpre; });
        if (tid == 0) {
            const unsigned long long dm = ((1ull << width) - 1ull) << lo;
            sc.kpre |= (unsigned long long)sc.digit << lo;
            sc.kmask |= dm;
            sc.need -= (int)sc.above;
            if (sc.hist[sc.digit] == (unsigned)sc.need) sc.all_tied = 1;
        }
        __syncthreads();
        if (sc.all_tied) done = true;
    }
    if (!sc.all_tied) {
        // the threshold key is fully determined; lower bits are common to all
        if (tid == 0) {
            // complete kpre with the common low bits
            unsigned long long low = (lo_bit > 0) ? ((1ull << lo_bit) - 1ull) : 0ull;
            sc.kpre = (sc.kpre & ~low) | (keyat(0) & low);
            sc.kmask = ~0ull;
        }
        __syncthreads();
        const unsigned long long T = sc.kpre;
        // idx phase on ~idx (larger ~idx = smaller idx) among key == T
        for (int top = 31; top >= 0; top -= 8) {
            const int lo = top - 7;
            const unsigned ipre = sc.ipre, imask = sc.imask;
            radix_pass(sc, n, lo, 8, [&](int e) { return (unsigned long long)(~idat(e)); },
                       [&](int e) { return keyat(e) == T && ((~idat(e)) & imask) == ipre; });
            if (tid == 0) {
                sc.ipre |= (unsigned)sc.digit << lo;
                sc.imask |= 0xffu << lo;
                sc.need -= (int)sc.above;
                if (sc.hist[sc.digit] == (unsigned)sc.need) sc.all_tied = 2;
            }
            __syncthreads();
            if (sc.all_tied) break;
        }
    }
    Thresh t;
    t.kpre = sc.kpre;
    t.kmask = sc.kmask;
    t.ipre = sc.ipre;
    t.imask = sc.imask;
    t.all_tied = sc.all_tied == 1;
    __syncthreads();
    return t;
}

}  // namespace lbm
