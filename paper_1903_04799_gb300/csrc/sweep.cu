// sweep.cu -- fused stream + collide over the whole lattice of a context
// (Sec. III, Eq. "lb"); the per-cell arithmetic is in sweep_body.cuh.
//
// Grid (x-blocks, y-blocks, z-planes).  The update is the in-place AA pattern
// (see lbsq_internal.cuh): even steps read and write a cell's own 19 slots,
// odd steps read and write its 19 neighbour slots.  The kernels are
// geometry-free: solid cells are swept too (their slots are private to them,
// and every slot a fluid cell reads from a solid neighbour is rewritten by the
// link kernel after the sweep), so no flag field is read.
#include <algorithm>

#include "sweep_body.cuh"

namespace lbsq {

// Every kernel comes in two forms: NEAR = false over grid rows (modes 0 and
// 1), NEAR = true over the rows of the window (mode 2).
template <int S, int P, bool NATIVE, bool NEAR>
__global__ void __launch_bounds__(256) k_sweep(const SweepArgs a) {
    dep_wait();
    dep_launch();
    const uint32_t skey = S == ST_BF16 ? sr_step_key(a) : 0u;  // before any exit (see sr_step)
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (NEAR) {
        near_rows(a, [&](int y, int z, bool active) {
            if (active && x < a.nx) sweep_one<S, P, NATIVE>(a, x, y, z, skey);
        });
    } else {
        int y, z;
        if (!sweep_at(a, blockIdx.y * blockDim.y + threadIdx.y, y, z) || x >= a.nx) return;
        sweep_one<S, P, NATIVE>(a, x, y, z, skey);
    }
}

// FP64 storage, double-float collision (sweep_df.cuh), one cell per thread.
// lambda_e = 1: three blocks per SM (80 registers, 56 bytes of spill): 24 warps
// per SM hide the loads better than 16.  The general relaxation has more live
// values; at 80 registers it spills 128 bytes, and 160 x 144 x 130 takes 161 us
// per step against 159 at two blocks per SM.  The near form, with its loop over
// rows, runs at two blocks too.
template <int P, bool LE1, bool NEAR>
__global__ void __launch_bounds__(256, NEAR || !LE1 ? 2 : 3) k_sweep_df(const SweepArgs a) {
    dep_wait();
    dep_launch();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (NEAR) {
        near_rows(a, [&](int y, int z, bool active) {
            if (active && x < a.nx) sweep_one_df<P, LE1>(a, x, y, z);
        });
    } else {
        int y, z;
        if (!sweep_at(a, blockIdx.y, y, z) || x >= a.nx) return;
        sweep_one_df<P, LE1>(a, x, y, z);
    }
}

template <int S, int P, bool NEAR>
__global__ void __launch_bounds__(256, 2) k_sweep2(const SweepArgs a) {
    dep_wait();
    dep_launch();
    const uint32_t skey = S == ST_BF16 ? sr_step_key(a) : 0u;  // before any exit (see sr_step)
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if constexpr (NEAR) {
        near_rows(a, [&](int y, int z, bool active) {
            if (active && x0 < a.nx) sweep_two<S, P>(a, x0, y, z, skey);
        });
    } else {
        int y, z;
        const bool go = sweep_at(a, blockIdx.y * blockDim.y + threadIdx.y, y, z);
        if (x0 >= a.nx || y >= a.ny) return;
        sweep_two<S, P>(a, x0, y, z, skey, go);
    }
}

// 16-bit storages with nx % 4 == 0, nx <= 768: blocks of whole rows, four
// cells per thread (see sweep_four_rows); dynamic shared memory of
// 10 x rows x nx elements on odd steps.
template <int S, int P, bool NEAR>
__global__ void __launch_bounds__(P == 0 ? 256 : 192, 2) k_sweep4r(const SweepArgs a) {
    dep_wait();
    dep_launch();
    extern __shared__ unsigned short rowbuf[];
    const uint32_t skey = S == ST_BF16 ? sr_step_key(a) : 0u;  // before any exit (see sr_step)
    if constexpr (NEAR) {
        near_rows(a, [&](int y, int z, bool active) {
            sweep_four_rows<S, P>(a, y, z, active, rowbuf, skey);
            if (P == 1) __syncthreads();  // the row buffer is reused
        });
    } else {
        int y, z;
        const bool go = sweep_at(a, blockIdx.y * blockDim.y + threadIdx.y, y, z);
        sweep_four_rows<S, P>(a, y < a.ny ? y : 0, z, go, rowbuf, skey);
    }
}

// Which of the `count` consecutive cells from n0 on are swept, as a bit mask
// (modes 0 and 1).
__device__ __forceinline__ unsigned cells_swept(const SweepArgs& a, uint32_t n0, uint32_t count) {
    const unsigned all = (1u << count) - 1u;
    if (a.zmode == 0) return all;
    const int4 w = __ldg(reinterpret_cast<const int4*>(a.win));
    const uint32_t nx = a.nx, ny = a.ny;
    uint32_t r = n0 / nx, x = n0 - r * nx;
    unsigned in = 0;  // cells in the window
    for (uint32_t k = 0; k < count;) {
        const uint32_t run = umin(count - k, nx - x);  // cells of row r
        int rz = (int)(r / ny) - w.x, ry = (int)(r % ny) - w.z;
        rz += rz < 0 ? a.nz : 0;
        ry += ry < 0 ? a.ny : 0;
        if (rz < w.y && ry < w.w) in |= ((1u << run) - 1u) << k;
        k += run;
        x = 0;
        ++r;
    }
    return all & ~in;
}

// Even steps (modes 0 and 1) of rows that the forms above do not fit: four
// consecutive cells per thread in 16 bits (sweep_four_flat), two in FP32, those
// `ahead` cells further prefetched into L2.  The cells at the lattice's end
// that fill no chunk, and the chunks that the window's border cuts, go one by
// one.
template <int S>
__global__ void __launch_bounds__(256, 2) k_sweep_flat(const SweepArgs a, uint32_t ahead) {
    dep_wait();
    dep_launch();
    const uint32_t skey = S == ST_BF16 ? sr_step_key(a) : 0u;  // before any exit (see sr_step)
    using T = typename StoreT<S>::T;
    constexpr uint32_t W = S == ST_F32 ? 2 : 4;
    const uint32_t N = (uint32_t)a.nx * (uint32_t)a.ny * (uint32_t)a.nz;
    const uint32_t n0 = W * (blockIdx.x * blockDim.x + threadIdx.x);
    if (n0 >= N) return;
    if (ahead && n0 + ahead < N) {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            asm volatile("prefetch.global.L2 [%0];" ::"l"((const T*)a.F + ((Off)i * (Off)a.Np + n0 + ahead)));
    }
    const unsigned take = cells_swept(a, n0, umin(W, N - n0));
    if (take == (1u << W) - 1u) {
        if constexpr (S == ST_F32) sweep_two_flat(a, n0);
        else sweep_four_flat<S>(a, n0, skey);
    } else {
        for (uint32_t k = 0; k < W; ++k)
            if (take >> k & 1u) sweep_one_call<S, 0>(a, (int)(n0 + k), 0, 0, skey);  // own slots only: any cell as x
    }
}

// 16-bit storages with nx % 4 == 0, odd steps of split sweeps: four cells per
// thread without shared memory (see sweep_four_odd), blocks of at most 192
// threads (167 registers, no spill; at 256 threads the 128-register cap
// spills 72-80 bytes and measured 3-4 % slower).
template <int S, bool NEAR>
__global__ void __launch_bounds__(192, 2) k_sweep4o(const SweepArgs a) {
    dep_wait();
    dep_launch();
    const uint32_t skey = S == ST_BF16 ? sr_step_key(a) : 0u;  // before any exit (see sr_step)
    const int x0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if constexpr (NEAR) {
        near_rows(a, [&](int y, int z, bool active) {
            if (active && x0 < a.nx) sweep_four_odd<S>(a, x0, y, z, skey, true);
        });
    } else {
        int y, z;
        const bool go = sweep_at(a, blockIdx.y * blockDim.y + threadIdx.y, y, z);
        if (x0 >= a.nx || y >= a.ny) return;
        sweep_four_odd<S>(a, x0, y, z, skey, go);
    }
}

// Shape of a sweep launch: bx x by threads, xblocks blocks along a row, grid
// planes and rows gz, gy, blocks per SM that reside together.
struct Rows {
    int bx, by, xblocks, gz, gy, resident;
};

static int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

// Planes ahead for the L2 prefetch of the sources (SweepArgs::pf): just past
// the planes that the resident blocks (two per SM for FP32, three for FP64)
// cover; FP32 adds two more.
// Measured on GB300, whole-lattice sweeps:
//   FP32 (two-cell form, 256^3): 0.959 -> 0.990 of the copy bandwidth;
//   FP64 (double-float form): 256^3 0.65 -> 0.75 at 1 or 2 planes ahead,
//     0.66 at 4, 0.60 at 5; 192^3 0.56 -> 0.72; 128^3 0.64 -> 0.78;
//   16-bit sweeps: see prefetch_ahead16.
// Far sweeps of split steps prefetch from 200 MB of populations on
// (far_prefetch).  Below, the step is as long as its body kernels' chain, whose
// code the prefetched lines, which enter L2 at normal priority, evict; above,
// the far sweep sets the pace.  One squirmer, us per step without / with:
//   FP32 128^3 (159 MB) 45 / 56, 144^3 (227 MB) 82 / 76, 160^3 106 / 94, 192^3
//   169 / 155, 250^3 371 / 355, 256^3 377 / 375; partially saturated cells
//   160^3 120 / 109, 256^3 420 / 414;
//   FP64 96^3 (134 MB) 48.1 / 51.2, 112^3 (213 MB) 82.7 / 83.9, 128^3 109 / 108,
//   144^3 188 / 170, 160^3 236 / 210, 250^3 916 / 825;
//   FP16 96^3 24.2 / 24.5, 160^3 (156 MB) 69.3 / 70.1, 192^3 (269 MB) 110 / 105,
//   250^3 225 / 221; BF16 160^3 76.6 / 77.0, 192^3 121 / 114.
static bool far_prefetch(const SweepArgs& a, int storage) {
    return a.zmode != 1 || 19 * a.Np * storage_bytes(storage) >= 200000000;
}
// A near sweep prefetches nothing: its window is a few planes deep (250^3 pair
// in BF16, whole step: 341 -> 334 us without).
static int prefetch_ahead(const SweepArgs& a, int storage, const Rows& r) {
    if (a.zmode == 2 || !far_prefetch(a, storage)) return 0;
    const long long per_plane = (long long)r.xblocks * ((r.gy + r.by - 1) / r.by);
    const long long resident = (long long)r.resident * sm_count();
    const int ahead = (int)((resident + per_plane - 1) / per_plane) + (storage == ST_F32 ? 2 : 0);
    return ahead < a.nz ? ahead : 0;
}

// Planes ahead for the L2 prefetch of the 16-bit sweeps (sweep_four_rows on
// even steps, sweep_two on odd steps): `extra` past the planes the resident
// blocks (two per SM) cover.  Measured on GB300 at 256^3 over both parities,
// against no prefetch: FP16 0.765 -> 0.807 with the even steps' (2 past; 0 or
// 4: the same within 0.3 %), -> 0.840 with the odd steps' too (0 past; 2 or
// 4: within 0.4 %); BF16 0.679 -> 0.703 -> 0.710.  Split sweeps prefetch
// too: the 256^3 pusher's whole step, FP16 0.2516 -> 0.2468 ms, BF16 0.2841 ->
// 0.2850 ms.  (An earlier measurement of the two-cell form prefetching on both
// parities, 0.745 -> 0.684, was taken before the sweeps' traffic was marked
// evict-first.)
static int prefetch_ahead16(const SweepArgs& a, const Rows& r, int extra) {
    if (a.zmode == 2 || !far_prefetch(a, ST_F16)) return 0;
    const long long per_plane = (long long)r.xblocks * ((r.gy + r.by - 1) / r.by);
    const long long resident = 2LL * sm_count();
    const int ahead = (int)((resident + per_plane - 1) / per_plane) + extra;
    return ahead < a.nz ? ahead : 0;
}

// Launch of one of the kernels above: bx x by threads, x blocks of bx threads
// along a row.  Rows of the lattice (modes 0 and 1) take a grid of their own;
// the near sweep a wave of `resident` blocks per SM that stride over the
// window, at most one block per by rows of its bound gz x gy.
template <class K>
static void launch_rows(K far_kernel, K near_kernel, const SweepArgs& a, const Rows& r, size_t smem, cudaStream_t st,
                        bool dep) {
    const dim3 block(r.bx, r.by);
    if (a.zmode != 2) {
        launch(far_kernel, dim3(r.xblocks, (r.gy + r.by - 1) / r.by, r.gz), block, smem, st, dep, a);
        return;
    }
    const long long want = ((long long)r.gz * r.gy + r.by - 1) / r.by;
    const long long wave = std::max(1, r.resident * sm_count() / r.xblocks);
    launch(near_kernel, dim3(r.xblocks, (unsigned)std::min(want, wave), 1), block, smem, st, dep, a);
}

template <bool LE1>
static void launch_df(const SweepArgs& a, int parity, const Rows& r, cudaStream_t st, bool dep) {
    if (parity == 0) launch_rows(k_sweep_df<0, LE1, false>, k_sweep_df<0, LE1, true>, a, r, 0, st, dep);
    else launch_rows(k_sweep_df<1, LE1, false>, k_sweep_df<1, LE1, true>, a, r, 0, st, dep);
}

// k_sweep_flat.  Whole-lattice steps (both parities) against the one- and
// two-cell forms: 250^3 FP16 241 -> 207 us, BF16 252 -> 217; 251^3 FP16 259 ->
// 217, BF16 375 -> 278; without the prefetch 250^3 FP16 215, BF16 227.
//
// Small lattices keep those forms, whose more numerous threads hide more
// latency; what counts is their threads, the cells with rows padded to whole
// warps.  One-cell / flat, whole-lattice steps: FP16 33^3 2.6 / 3.1 us, 45^3 3.4
// / 4.0, 59^3 4.4 / 4.9, 61^3 4.9 / 4.9, 65^3 6.2 / 5.4, 5 x 100 x 100 4.8 / 4.1;
// BF16 51^3 4.4 / 5.1, 65^3 8.2 / 6.7; FP32 33^3 2.6 / 3.0, 45^3 3.6 / 3.6, 51^3
// 4.1 / 3.9, 65^3 7.0 / 6.7, 7 x 50 x 60 2.3 / 2.7.
static bool flat_pays(const SweepArgs& a, int storage) {
    const int64_t threads = (int64_t)(a.nx + 31) / 32 * 32 * a.ny * a.nz;
    return threads >= (storage == ST_F32 ? 130000 : 240000);
}
template <int S>
static void launch_flat(const SweepArgs& a, cudaStream_t st, bool dep) {
    const uint32_t N = (uint32_t)a.nx * a.ny * a.nz, cells = (S == ST_F32 ? 2 : 4) * 256;
    const uint32_t ahead = 2u * sm_count() * cells + 2u * a.nx * a.ny;
    launch(k_sweep_flat<S>, (N + cells - 1) / cells, 256, 0, st, dep, a, ahead < N && far_prefetch(a, S) ? ahead : 0u);
}

template <int S>
static void launch_s(SweepArgs a, int parity, int variant, int gz, int gy, cudaStream_t st, bool dep) {
    const int nx = a.nx;
    auto rows = [&](int cells, int max_bx, int threads, int resident) {
        const int units = nx / cells;
        const int bx = std::min(max_bx, (units + 31) / 32 * 32);
        return Rows{bx, std::max(1, threads / bx), (units + bx - 1) / bx, gz, gy, resident};
    };
    if constexpr (S == ST_F64) {
        Rows r = rows(1, 256, 1, 3);
        if (variant == 1) {  // FP64 arithmetic
            r.resident = 2;
            if (parity == 0) launch_rows(k_sweep<S, 0, true, false>, k_sweep<S, 0, true, true>, a, r, 0, st, dep);
            else launch_rows(k_sweep<S, 1, true, false>, k_sweep<S, 1, true, true>, a, r, 0, st, dep);
            return;
        }
        if (a.zmode == 2 || !a.K.df.le1) r.resident = 2;
        a.pf = prefetch_ahead(a, S, r);
        if (a.K.df.le1) launch_df<true>(a, parity, r, st, dep);
        else launch_df<false>(a, parity, r, st, dep);
        return;
    }
    if constexpr (S == ST_F16 || S == ST_BF16) {
        // default: even steps in whole-row four-cell blocks (aligned 8-byte
        // chunks: 0.86 of the copy bandwidth at 256^3, against 0.74 for two
        // cells), odd steps in the two-cell form (0.63 before the L2
        // prefetch; the whole-row form's odd steps, with their x-shifts
        // through shared memory, measured 0.62), or in split sweeps as below
        const bool rows4 = nx % 4 == 0 && nx <= 768;
        // even steps of rows that whole-row blocks do not fit: four cells
        // regardless of rows.  Whole-lattice steps (both parities) against the
        // one- and two-cell forms: 250^3 FP16 241 -> 207 us, BF16 252 -> 217;
        // 251^3 FP16 259 -> 217, BF16 375 -> 278.  Where whole rows fit, the two
        // are equal in bare sweeps (256^3: 204 us) and the rows faster in split
        // ones (256^3 pusher FP16 222 against 226 us: no divisions for the window)
        if (variant == 0 && parity == 0 && a.zmode != 2 && !rows4 && flat_pays(a, S)) {
            launch_flat<S>(a, st, dep);
            return;
        }
        // odd steps of split sweeps (far and near, mode 1 and 2): four cells per
        // thread.  Measured on GB300, 256^3 pusher, whole step against the
        // two-cell form: FP16 0.242 -> 0.232 ms, BF16 with stochastic rounding
        // 0.260 -> 0.252 ms (BF16 to nearest 0.243 -> 0.245).  In
        // whole-lattice sweeps the two-cell form stays ahead (bare 256^3 step:
        // FP16 0.210 against 0.214 ms, BF16 to nearest 0.211 against 0.223),
        // so they keep it; why the split steps favour four cells is not known.
        if (variant == 0 && parity == 1 && nx % 4 == 0 && a.zmode != 0) {
            const Rows r = rows(4, 64, 192, 2);
            a.pf = prefetch_ahead16(a, r, 0);
            launch_rows(k_sweep4o<S, false>, k_sweep4o<S, true>, a, r, 0, st, dep);
            return;
        }
        if ((variant == 3 || (variant == 0 && parity == 0)) && rows4) {
            // odd steps (more live values) in blocks of at most 192 threads
            const int tx = nx / 4, ty = std::max(1, (parity == 0 ? 256 : 192) / tx);
            const Rows r{tx, ty, 1, gz, gy, 2};
            if (parity == 0) {
                a.pf = prefetch_ahead16(a, r, 2);
                launch_rows(k_sweep4r<S, 0, false>, k_sweep4r<S, 0, true>, a, r, 0, st, dep);
            } else {
                const size_t smem = (size_t)10 * ty * nx * sizeof(unsigned short);
                launch_rows(k_sweep4r<S, 1, false>, k_sweep4r<S, 1, true>, a, r, smem, st, dep);
            }
            return;
        }
    }
    if constexpr (S != ST_F64) {
        if (variant != 1 && nx % 2 == 0) {
            const Rows r = rows(2, 128, 256, 2);
            if (S == ST_F32) a.pf = prefetch_ahead(a, S, r);
            else a.pf = parity == 1 ? prefetch_ahead16(a, r, 0) : 0;
            if (parity == 0) launch_rows(k_sweep2<S, 0, false>, k_sweep2<S, 0, true>, a, r, 0, st, dep);
            else launch_rows(k_sweep2<S, 1, false>, k_sweep2<S, 1, true>, a, r, 0, st, dep);
            return;
        }
        // FP32 with odd nx, even steps: two cells regardless of rows (whole-lattice
        // steps: 251^3 382 -> 361 us, 125 x 99 x 111 25.6 -> 25.1).  Odd steps keep
        // one cell: pairs across odd rows, every access scalar and every second
        // element left to another instruction, took 408 us.  In split steps of
        // lattices that fit L2 the window's divisions cost what the pairs gain
        // (one squirmer, one cell / flat: 99^3 25.5 / 25.3, 111 x 111 x 112, 105 MB,
        // 31.8 / 31.3, 121 x 121 x 122, 136 MB, 40.1 / 39.3, 131^3 57.6 / 53.4, 161^3
        // 105 / 97, 201^3 214 / 195).
        if (S == ST_F32 && variant == 0 && parity == 0 && flat_pays(a, S) &&
            (a.zmode == 0 || (a.zmode == 1 && 19 * a.Np * 4 > (128 << 20)))) {
            launch_flat<S>(a, st, dep);
            return;
        }
        // Blocks of 128 threads: one row of few cells per block left the GPU
        // starting blocks (one about every nanosecond: 7 x 200 x 300, 60 000 rows,
        // FP32 35 -> 14 us per step, FP16 34 -> 14; 5 x 100 x 100 6.9 -> 4.1).
        const Rows r = rows(1, 256, 128, 4);
        // (no L2 prefetch: 125 x 99 x 111 FP16 16.9 us per step without, 19.1 with)
        if (parity == 0) launch_rows(k_sweep<S, 0, false, false>, k_sweep<S, 0, false, true>, a, r, 0, st, dep);
        else launch_rows(k_sweep<S, 1, false, false>, k_sweep<S, 1, false, true>, a, r, 0, st, dep);
    }
}

// variant: 0 = default (FP64: double-float collision, one cell per thread;
// FP32: two cells per thread (even nx); FP16 / BF16: even steps as 3 or
// k_sweep_flat, odd steps as 2, or four cells per thread without shared memory in split
// sweeps), 1 = one cell per thread (FP64: FP64 arithmetic), 2 = two
// cells per thread where possible (not FP64), 3 = FP16 / BF16: four cells per
// thread in blocks of whole rows on both parities, odd-step x-shifts through
// shared memory (nx % 4 == 0, nx <= 768; else as 2).
// zmode / win / gz / gy: cell selection (see SweepArgs); gz and gy = grid
// planes and rows (nz and ny for modes 0 and 1, upper bounds of the window's
// z and y lengths for mode 2).  Odd steps sweep the planes in descending
// order.  dep: a dependent launch (see dep_wait).
void launch_sweep(const Lattice& L, double lambda_e, double lambda_o, int parity, int variant, int zmode,
                  const int* win, int gz, int gy, cudaStream_t st, bool dep) {
    SweepArgs a = sweep_args(L, lambda_e, lambda_o);
    a.zmode = zmode;
    a.win = win;
    a.reverse = parity;
    a.sr_writer = zmode != 2;  // of a split step's two sweeps, the far one advances the step counter
    if (gz <= 0 || gy <= 0) return;
    switch (L.storage) {
        case ST_F64: launch_s<ST_F64>(a, parity, variant, gz, gy, st, dep); break;
        case ST_F32: launch_s<ST_F32>(a, parity, variant, gz, gy, st, dep); break;
        case ST_F16: launch_s<ST_F16>(a, parity, variant, gz, gy, st, dep); break;
        default: launch_s<ST_BF16>(a, parity, variant, gz, gy, st, dep); break;
    }
}

}  // namespace lbsq
