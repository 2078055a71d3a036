// setup.cu -- kernels that initialise, inspect or export the lattice; none of
// them runs inside a time step.
#include <cfloat>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "lbsq_internal.cuh"

namespace lbsq {

constexpr int kB = 256;

__device__ __forceinline__ bool grid_cell(const Lattice& L, int64_t& n, int& x, int& y, int& z) {
    n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= L.N) return false;
    cell_coords(L, n, x, y, z);
    return true;
}

static unsigned grid_for(int64_t N) { return (unsigned)((N + kB - 1) / kB); }

// Every population at rest equilibrium w_i rho0 (Sec. III).
__global__ void k_fill_rest(const Lattice L) {
    int64_t n;
    int x, y, z;
    if (!grid_cell(L, n, x, y, z)) return;
    for (int i = 0; i < Q; ++i) store_abs(L, (int64_t)i * L.Np + n, i, wgt(i) * L.rho0);
}

// Equilibrium of given fields, w_i rho (1 + 3 c.u + 9/2 (c.u)^2 - 3/2 u.u)
// (incompressible: w_i (rho + rho0 (3 c.u + 9/2 (c.u)^2 - 3/2 u.u))), into
// the read slots of parity q.  rho[N], u[3][N] on the device.
__global__ void k_set_eq(const Lattice L, const double* rho, const double* u, int q) {
    int64_t n;
    int x, y, z;
    if (!grid_cell(L, n, x, y, z)) return;
    const double r = rho[n], ux = u[n], uy = u[L.N + n], uz = u[2 * L.N + n];
    const double uu = ux * ux + uy * uy + uz * uz;
    for (int i = 0; i < Q; ++i) {
        const double cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
        const double fe = L.inc ? wgt(i) * (r + L.rho0 * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
                                : wgt(i) * r * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
        store_abs(L, read_slot(L, i, x, y, z, q), i, fe);
    }
}

// f[19][N] (absolute values) <-> read slots of parity q.
__global__ void k_set_pop(const Lattice L, const double* f, int q) {
    int64_t n;
    int x, y, z;
    if (!grid_cell(L, n, x, y, z)) return;
    for (int i = 0; i < Q; ++i) store_abs(L, read_slot(L, i, x, y, z, q), i, f[(int64_t)i * L.N + n]);
}

__global__ void k_get_pop(const Lattice L, double* f, int q) {
    int64_t n;
    int x, y, z;
    if (!grid_cell(L, n, x, y, z)) return;
    for (int i = 0; i < Q; ++i) f[(int64_t)i * L.N + n] = load_abs(L, read_slot(L, i, x, y, z, q), i);
}

// ---- density and momentum of a cell
//
// rho = rho0 + sum g_i and j = sum g_i c_i of the stored deviations, summed in
// 64-bit fixed point (unit 2^(k0 - 60), k0 the exponent of rho0).  The integer
// sums are exact; what rounds is the conversion, which cuts a deviation off at
// the unit, 2^-60 rho0 or less (to_fx: FP64 below 2^-8 rho0, FP32 below 2^-37;
// 19 terms err by less than an ulp of rho, where FP64 sums erred by several).
// What bounds a read-out kernel is this GPU's FP64 rate, not memory: one FP64
// warp instruction takes the SM's pipe 16 cycles, the issue slots of 64
// others, and the sums in FP64 took about 100 per cell (256^3: 4.7 ms on even
// steps, 7.2 ms on odd ones, 3 % of the DRAM bandwidth).  A deviation becomes
// a fixed-point number in about 10 integer instructions, a 64-bit add takes
// two.  256^3 after: FP64 0.50 / 0.58 ms (even / odd steps,
// 0.46 ms at the copy rate), FP32 and 16 bits 0.43 ms.
// Cells with a deviation outside 0.15 rho0 (NaN and Inf included) or a
// density that is not positive take the FP64 sums of moments_general.
struct MomentK {
    int fx;             // fixed point usable: rho0 within 2^+-60
    int k0;             // exponent of rho0
    unsigned thr64;     // high word of 0.15 * 2^k0
    int kf;             // k0 plus the exponent of the storage's scale
    unsigned thr32;     // FP32 bits of 0.15 * 2^kf
    float inv_unit_rho; // (float)2^(k0 - 60)
    long long rho0_fx;  // rho0 in fixed point (exact)
    double inv_rho0;
};

static MomentK moment_constants(const Lattice& L) {
    MomentK k{};
    int e = 0;
    std::frexp(L.rho0, &e);
    k.k0 = e - 1;
    k.fx = k.k0 >= -60 && k.k0 <= 60;
    if (!k.fx) return k;
    const double b = std::ldexp(0.15, k.k0);
    unsigned long long bits;
    memcpy(&bits, &b, 8);
    k.thr64 = (unsigned)(bits >> 32);
    k.kf = k.k0 + std::ilogb(L.scale);
    const float bf = std::ldexp(0.15f, k.kf);
    memcpy(&k.thr32, &bf, 4);
    k.inv_unit_rho = std::ldexp(1.0f, k.k0 - 60);
    k.rho0_fx = (long long)std::ldexp(L.rho0, 60 - k.k0);
    k.inv_rho0 = 1.0 / L.rho0;
    return k;
}

// A stored value as an integer in units of 2^(k0 - 60); ok is cleared when it
// lies outside the range.  FP64: the mantissa shifted into place, truncated
// below 2^-60 rho0 (exact for |g| >= 2^-8 rho0).
__device__ __forceinline__ long long to_fx(uint2 w, const MomentK& K, bool& ok) {
    ok = ok && (w.y & 0x7fffffffu) < K.thr64;
    const unsigned e = (w.y >> 20) & 0x7ffu;
    const unsigned long long m =
        ((unsigned long long)((w.y & 0xfffffu) | 0x100000u) << 32 | (unsigned long long)w.x) << 10;
    const unsigned sh = umin((unsigned)(1025 + K.k0) - e, 63u);
    const long long v = (long long)(m >> sh), sg = (long long)((int)w.y >> 31);
    return (v ^ sg) - sg;
}
// FP32 (in the storage's units): exact for |g| >= 2^-37 rho0.  A conversion
// instruction to 64 bits per value made the kernel slower than these integer
// ones (256^3 FP32: 0.82 ms).
__device__ __forceinline__ long long to_fx(float g, const MomentK& K, bool& ok) {
    const unsigned b = __float_as_uint(g), e = (b >> 23) & 0xffu;
    ok = ok && (b & 0x7fffffffu) < K.thr32;
    const unsigned long long m = (unsigned long long)(((b & 0x7fffffu) | 0x800000u) << 7) << 32;
    const unsigned sh = umin((unsigned)(129 + K.kf) - e, 63u);
    const long long v = (long long)(m >> sh), sg = (long long)((int)b >> 31);
    return (v ^ sg) - sg;
}

// v 2^k as a double (to nearest), in integer arithmetic: a conversion
// instruction would take the FP64 pipe.
__device__ __forceinline__ double fx_to_double(long long v, int k) {
    unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    m <<= lz;
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // the implicit bit adds one to the exponent
    const unsigned long long bits = ((unsigned long long)(1085 - lz + k) << 52) + r;
    return __longlong_as_double((long long)(bits | (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// FP64 sums of the deviations of cell (x, y, z): v = {sum g, sum g c}.
__device__ __noinline__ void moments_general(const Lattice& L, int64_t n, int q, double v[4]) {
    int x, y, z;
    cell_coords(L, n, x, y, z);
    v[0] = v[1] = v[2] = v[3] = 0.0;
    for (int i = 0; i < Q; ++i) {
        const int64_t s = read_slot(L, i, x, y, z, q);
        const double g = L.storage == ST_F64 ? ((const double*)L.F)[s] : (double)load_dev(L, s);
        v[0] += g;
        v[1] += g * cx(i);
        v[2] += g * cy(i);
        v[3] += g * cz(i);
    }
}

// Fixed-point sums m = {sum g, sum g c} of cell n from the read slots of
// parity P; false where they do not hold.
template <int S, int P>
__device__ __forceinline__ bool moments_fx(const Lattice& L, uint32_t n, const MomentK& K, long long m[4]) {
    using T = typename std::conditional<S == ST_F64, uint2, typename StoreT<S>::T>::type;
    const T* F = (const T*)L.F;
    const uint32_t Np = (uint32_t)L.Np;  // 19 Np < 2^32
    T w[Q];
    if constexpr (P == 0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) w[i] = ld_stream(F + ((uint32_t)i * Np + n));
    } else {
        const uint32_t nx = L.nx, ny = L.ny, nz = L.nz;
        const uint32_t r = n / nx, x = n - r * nx, z = r / ny, y = r - z * ny;
        const uint32_t xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
        const uint32_t ys[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
        const uint32_t zs[3] = {z == 0 ? nz - 1 : z - 1, z, z == nz - 1 ? 0 : z + 1};
#pragma unroll
        for (int i = 0; i < Q; ++i)
            w[i] = ld_stream(F + ((uint32_t)opp(i) * Np + xs[1 - cx(i)] + nx * (ys[1 - cy(i)] + ny * zs[1 - cz(i)])));
    }
    bool ok = true;
    long long s = 0, j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        long long v;
        if constexpr (S == ST_F64) v = to_fx(w[i], K, ok);
        else if constexpr (S == ST_F32) v = to_fx(w[i], K, ok);
        else if constexpr (S == ST_F16) v = to_fx(__half2float(w[i]), K, ok);
        else v = to_fx(__bfloat162float(w[i]), K, ok);
        s += v;
        if (cx(i)) j[0] += cx(i) > 0 ? v : -v;
        if (cy(i)) j[1] += cy(i) > 0 ? v : -v;
        if (cz(i)) j[2] += cz(i) > 0 ? v : -v;
    }
    m[0] = s;
    for (int a = 0; a < 3; ++a) m[1 + a] = j[a];
    return ok && K.fx && K.rho0_fx + s > (1ll << 55);
}

// rho = sum f_i and u = j / rho of fluid cells (Sec. III; incompressible
// equilibrium: u = j / rho0); 0 in solid cells.  1 / rho: an FP32 estimate and
// two Newton steps in FP64 (4 FP64 instructions; the estimate's relative error
// of 2^-23 squares at each), then one product per component: within two units
// in the last place of the quotient.
template <int S, int P>
__global__ void __launch_bounds__(kB) k_fields(const Lattice L, const int32_t* own, double* rho, double* u,
                                               const MomentK K) {
    const int64_t n = (int64_t)blockIdx.x * kB + threadIdx.x;
    if (n >= L.N) return;
    const bool fluid = own[n] == 0;
    long long m[4];
    const bool ok = moments_fx<S, P>(L, (uint32_t)n, K, m);
    double r = 0.0, v[3] = {0.0, 0.0, 0.0};
    if (fluid && ok) {
        const long long rf = K.rho0_fx + m[0];
        r = fx_to_double(rf, K.k0 - 60);
        double inv = K.inv_rho0;
        if (!L.inc) {
            const float seed = __frcp_rn(__ll2float_rn(rf) * K.inv_unit_rho);
            inv = (double)seed;
            inv = __fma_rn(inv, __fma_rn(-r, inv, 1.0), inv);
            inv = __fma_rn(inv, __fma_rn(-r, inv, 1.0), inv);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fx_to_double(m[1 + a], K.k0 - 60) * inv;
    } else if (fluid) {
        double g[4];
        moments_general(L, n, P, g);
        r = L.rho0 + g[0];
        const double den = L.inc ? L.rho0 : r;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = r != 0.0 ? g[1 + a] / den : 0.0;
    }
    if (rho) __stcs(rho + n, r);
    if (u) {
#pragma unroll
        for (int a = 0; a < 3; ++a) __stcs(u + a * L.N + n, v[a]);
    }
}

// Mass and momentum of the fluid: per-block partials, then a one-block pass
// that sums them in block order (a fixed order, hence reproducible bits).
// A thread sums the deviations of its cells (kMassCells of them, kB apart) and
// counts them; the rest density enters as rho0 times the count.  256^3 with
// the copy back: 5.7 - 7.5 ms before the fixed-point sums, 0.5 - 0.6 ms now.
constexpr int kMassCells = 8;
template <int S, int P>
__global__ void __launch_bounds__(kB) k_mass_partial(const Lattice L, const int32_t* own, double* part,
                                                     const MomentK K) {
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    int count = 0;
    for (int c = 0; c < kMassCells; ++c) {
        const int64_t n = ((int64_t)blockIdx.x * kMassCells + c) * kB + threadIdx.x;
        if (n >= L.N) break;
        if (own[n] != 0) continue;
        ++count;
        long long m[4];
        if (moments_fx<S, P>(L, (uint32_t)n, K, m)) {
            for (int k = 0; k < 4; ++k) v[k] += fx_to_double(m[k], K.k0 - 60);
        } else {
            double g[4];
            moments_general(L, n, P, g);
            for (int k = 0; k < 4; ++k) v[k] += g[k];
        }
    }
    v[0] += L.rho0 * (double)count;
    __shared__ double sm[kB / 32][4];
    for (int k = 0; k < 4; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
        for (int k = 0; k < 4; ++k) sm[warp][k] = v[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int w = 0; w < kB / 32; ++w)
            for (int k = 0; k < 4; ++k) t[k] += sm[w][k];
        for (int k = 0; k < 4; ++k) part[(size_t)blockIdx.x * 4 + k] = t[k];
    }
}

// Threads (j, k), j < kB / 4, sum component k of blocks j, j + kB / 4, ...;
// then one thread per component adds the kB / 4 sums in order.
__global__ void k_mass_final(const double* part, int nblocks, double* out) {
    __shared__ double sm[kB];
    const int k = threadIdx.x & 3;
    double t = 0.0;
    for (int b = threadIdx.x >> 2; b < nblocks; b += kB / 4) t += part[(size_t)b * 4 + k];
    sm[threadIdx.x] = t;
    __syncthreads();
    if (threadIdx.x < 4) {
        double s = 0.0;
        for (int j = 0; j < kB / 4; ++j) s += sm[4 * j + k];
        out[k] = s;
    }
}

// Count cells a new sphere would cover that are already solid.
__global__ void k_sphere_overlap(const Lattice L, const int32_t* own, double px, double py, double pz, double R,
                                 int W, int* count) {
    const long long total = (long long)W * W * W;
    const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= total) return;
    const int lx = (int)floor(px - R) - 2, ly = (int)floor(py - R) - 2, lz = (int)floor(pz - R) - 2;
    const int x = wrapi(lx + (int)(b % W), L.nx), y = wrapi(ly + (int)((b / W) % W), L.ny),
              z = wrapi(lz + (int)(b / ((long long)W * W)), L.nz);
    const double dx = min_image((double)x - px, L.nx), dy = min_image((double)y - py, L.ny),
                 dz = min_image((double)z - pz, L.nz);
    if (inside_sphere(dx, dy, dz, R) && own[cell_index(L, x, y, z)] != 0) atomicAdd(count, 1);
}

// Plane wall: count sphere-owned cells of the layer (kind[] maps id-1 -> kind),
// then claim the fluid cells of the layer (cells of other walls stay theirs).
__global__ void k_plane_overlap(const Lattice L, const int32_t* own, const int* kind, int axis, int index,
                                int* count) {
    int64_t n;
    int c[3];
    if (!grid_cell(L, n, c[0], c[1], c[2])) return;
    if (c[axis] != index) return;
    const int o = own[n];
    if (o != 0 && kind[o - 1] == BODY_SPHERE) atomicAdd(count, 1);
}

__global__ void k_plane_claim(const Lattice L, int32_t* own, int axis, int index, int id) {
    int64_t n;
    int c[3];
    if (!grid_cell(L, n, c[0], c[1], c[2])) return;
    if (c[axis] == index && own[n] == 0) own[n] = id;
}

// A round tube along z (BodyParams::tube): solid nodes already held by a
// sphere, counted; free solid nodes claimed for body `id`.
__global__ void k_tube_overlap(const Lattice L, const int32_t* own, const int* kind, const BodyParams q, int* count) {
    int64_t n;
    int c[3];
    if (!grid_cell(L, n, c[0], c[1], c[2])) return;
    if (!tube_solid(q, c[0], c[1])) return;
    const int o = own[n];
    if (o != 0 && kind[o - 1] == BODY_SPHERE) atomicAdd(count, 1);
}

__global__ void k_tube_claim(const Lattice L, int32_t* own, const BodyParams q, int id) {
    int64_t n;
    int c[3];
    if (!grid_cell(L, n, c[0], c[1], c[2])) return;
    if (tube_solid(q, c[0], c[1]) && own[n] == 0) own[n] = id;
}

// Work flag for set-up passes: body k (or all if k < 0) re-classifies (and
// its node margin restarts) or not.
__global__ void k_set_flags(BodyAcc* acc, int nb, int k, int reclass) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nb || (k >= 0 && j != k)) return;
    acc[j].reclass = reclass;
    if (reclass) acc[j].margin_bits = (unsigned long long)__double_as_longlong(DBL_MAX);
}

// A read-out of a few hundred bytes: `words` 64-bit words of src after the
// device error word, so that the host gets both in one copy.
__global__ void k_gather(const int* err, const unsigned long long* src, int words, unsigned long long* dst) {
    const int t = threadIdx.x;
    if (t == 0) dst[0] = (unsigned long long)(unsigned)*err;
    for (int w = t; w < words; w += blockDim.x) dst[1 + w] = src[w];
}

// ---------------------------------------------------------------- launchers

void launch_gather(const int* err, const void* src, int words, void* dst, cudaStream_t st) {
    k_gather<<<1, 64, 0, st>>>(err, (const unsigned long long*)src, words, (unsigned long long*)dst);
}

// f(storage, parity) with both as compile-time constants.
template <class Fn>
static void with_storage(int storage, int q, Fn f) {
    auto parity = [&](auto S) {
        if (q == 0) f(S, std::integral_constant<int, 0>{});
        else f(S, std::integral_constant<int, 1>{});
    };
    switch (storage) {
        case ST_F64: parity(std::integral_constant<int, ST_F64>{}); break;
        case ST_F32: parity(std::integral_constant<int, ST_F32>{}); break;
        case ST_F16: parity(std::integral_constant<int, ST_F16>{}); break;
        default: parity(std::integral_constant<int, ST_BF16>{}); break;
    }
}

void launch_fill_rest(const Lattice& L, cudaStream_t st) { k_fill_rest<<<grid_for(L.N), kB, 0, st>>>(L); }
void launch_set_eq(const Lattice& L, const double* rho, const double* u, int q, cudaStream_t st) {
    k_set_eq<<<grid_for(L.N), kB, 0, st>>>(L, rho, u, q);
}
void launch_set_pop(const Lattice& L, const double* f, int q, cudaStream_t st) {
    k_set_pop<<<grid_for(L.N), kB, 0, st>>>(L, f, q);
}
void launch_get_pop(const Lattice& L, double* f, int q, cudaStream_t st) {
    k_get_pop<<<grid_for(L.N), kB, 0, st>>>(L, f, q);
}
void launch_fields(const Lattice& L, const int32_t* own, double* rho, double* u, int q, cudaStream_t st) {
    const MomentK K = moment_constants(L);
    const unsigned g = grid_for(L.N);
    with_storage(L.storage, q, [&](auto S, auto P) {
        k_fields<decltype(S)::value, decltype(P)::value><<<g, kB, 0, st>>>(L, own, rho, u, K);
    });
}
int mass_partial_blocks(const Lattice& L) { return (int)((L.N + kB * kMassCells - 1) / (kB * kMassCells)); }
void launch_mass(const Lattice& L, const int32_t* own, double* part, double* out, int q, cudaStream_t st) {
    const MomentK K = moment_constants(L);
    const int nb = mass_partial_blocks(L);
    with_storage(L.storage, q, [&](auto S, auto P) {
        k_mass_partial<decltype(S)::value, decltype(P)::value><<<nb, kB, 0, st>>>(L, own, part, K);
    });
    k_mass_final<<<1, kB, 0, st>>>(part, nb, out);
}
void launch_sphere_overlap(const Lattice& L, const int32_t* own, const double* pos, double R, int W, int* count,
                           cudaStream_t st) {
    const long long total = (long long)W * W * W;
    k_sphere_overlap<<<(unsigned)((total + kB - 1) / kB), kB, 0, st>>>(L, own, pos[0], pos[1], pos[2], R, W, count);
}
void launch_plane_overlap(const Lattice& L, const int32_t* own, const int* kind, int axis, int index, int* count,
                          cudaStream_t st) {
    k_plane_overlap<<<grid_for(L.N), kB, 0, st>>>(L, own, kind, axis, index, count);
}
void launch_plane_claim(const Lattice& L, int32_t* own, int axis, int index, int id, cudaStream_t st) {
    k_plane_claim<<<grid_for(L.N), kB, 0, st>>>(L, own, axis, index, id);
}
void launch_tube_overlap(const Lattice& L, const int32_t* own, const int* kind, const BodyParams& q, int* count,
                         cudaStream_t st) {
    k_tube_overlap<<<grid_for(L.N), kB, 0, st>>>(L, own, kind, q, count);
}
void launch_tube_claim(const Lattice& L, int32_t* own, const BodyParams& q, int id, cudaStream_t st) {
    k_tube_claim<<<grid_for(L.N), kB, 0, st>>>(L, own, q, id);
}
void launch_set_flags(BodyAcc* acc, int nb, int k, int reclass, cudaStream_t st) {
    k_set_flags<<<(nb + kB - 1) / kB, kB, 0, st>>>(acc, nb, k, reclass);
}


// Shell stencil of a sphere of radius R for k_body_fused: the offsets o from
// the centre's node floor(r) for which some centre fraction f in [0,1]^3 puts
// |o - f|^2 inside the bounds of in_shell widened by 1, packed as
// (ox + 512) | (oy + 512) << 10 | (oz + 512) << 20, in (z, y, x) order.
// Requires R <= kStencilMaxR.
std::vector<uint32_t> shell_stencil(double R) {
    const double lo2 = R > 1.5 ? (R - 1.5) * (R - 1.5) - 0.25 : -1.0;
    const double hi2 = (R + 2.0) * (R + 2.0) + 0.25;
    const int m = (int)std::ceil(R + 4.0);
    std::vector<uint32_t> v;
    for (int oz = -m; oz <= m; ++oz)
        for (int oy = -m; oy <= m; ++oy)
            for (int ox = -m; ox <= m; ++ox) {
                const int o[3] = {ox, oy, oz};
                double dmin = 0.0, dmax = 0.0;
                for (int a = 0; a < 3; ++a) {
                    const double t = o[a];
                    const double nearest = t < 0.0 ? -t : (t > 1.0 ? t - 1.0 : 0.0);
                    const double farthest = std::max(std::fabs(t), std::fabs(t - 1.0));
                    dmin += nearest * nearest;
                    dmax += farthest * farthest;
                }
                if (dmin < hi2 + 1.0 && dmax > lo2 - 1.0)
                    v.push_back((uint32_t)(ox + 512) | (uint32_t)(oy + 512) << 10 | (uint32_t)(oz + 512) << 20);
            }
    return v;
}

}  // namespace lbsq
