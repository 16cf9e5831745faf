// Inverse 2-D C2R transform at n = 64: tiles of 4 planes, even and odd rows ky by two teams of warps, two CTAs per SM.
//
// The half spectrum of a tile (66 KB) arrives as two TMA boxes, the even and the odd rows ky, in a ring of three; each
// team of 4 warps transforms the 16 rows of its box in place and then runs the columns over them alone: the even rows add to the samples of a column a
// 32-point real transform g, x[r] += g[r mod 32], the odd ones Re(i^v t[j]) with r = j + 16v and t one 16-point
// transform over rows (those above n/2 are conjugates) times 2 w_64^{-j}.  Only then do the teams exchange half of what
// they hold, and each completes half of the rows r of every column.
//
// Packed fp32 pairs (f32x2.cuh) of two adjacent columns.  Per tile and team of 128 threads:
//   B. two threads per row: the first butterfly of a decimation in frequency yields the even and the odd columns, the
//      two halves of a packed value; a second one splits the 32 pairs over the two threads, 16 points each;
//   A. thread = (plane, pair of columns): 16 rows, 32-point real or 16-point complex transform;
//   C. 8 values to the other team through shared memory, last butterfly, scale, cropped rows straight to the result.
// Row ky = 0 carries ky = n/2 as (re, im); the bins kx > n/2 of both are conjugates and are not read (GemmParams::herm_n).
// With spatial tiling a row of the matrix is a window and the crop goes to its place in the larger plane.
//
// Bound by the loads: rows of 16 bytes (4 planes) arrive at 1.3 cycles each and SM at best, 40 us for 8,192 planes, and by
// the wait for the odd rows, which are requested when a tile's even ones are in registers.  8,192 planes of 64 x 64 71 ->
// 61 us (57 x 57 the same), 2,048 of 57 x 57 25.6 -> 23.5, against whole rows and columns per thread in one CTA per SM with
// two staging tiles.  Tiles of 8 planes (rows of 32 bytes, one CTA per SM, 16 warps): 76 us.
#pragma once

#include "fft_big.cuh"

namespace fc {

struct Inv64Geom {
    static constexpr int N = 64, M = 32, NC = 33, G = 4, TEAM = 128, T = 2 * TEAM, HI = 16, RING = 3, MINB = 2;
    static constexpr size_t STAGE = (size_t)2 * N * HI * G * 4;  // a box: [part*N + kx][hi][plane], ky = 2 hi + lo
    // the same box as rows of 32 pairs in 16-byte units (re, re', im, im'); pitches: eight lanes = four planes x two rows (B)
    // and lanes over the pairs (A) are conflict-free
    static constexpr int RP = N / 2 + 4, PP = HI * RP + 1;
    static constexpr size_t ROWS = (size_t)G * PP * 16;
    static constexpr size_t BUF = ((ROWS > STAGE ? ROWS : STAGE) + 127) / 128 * 128;
    static constexpr size_t STAGE_NY = (size_t)2 * N * G * 4;
    static constexpr size_t SMEM = RING * BUF + STAGE_NY;
};

__device__ __forceinline__ void fk_tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                               uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}
__device__ __forceinline__ void inv64_team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(Inv64Geom::TEAM) : "memory");
}

__global__ void __launch_bounds__(Inv64Geom::T, Inv64Geom::MINB)
c2r_inv64_kernel(const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmNy,
                 const __grid_constant__ FftParams p) {
    using Gm = Inv64Geom;
    constexpr int N = Gm::N, M = Gm::M, G = Gm::G, RP = Gm::RP, PP = Gm::PP, RING = Gm::RING, PITCH = Gm::HI * G;
    extern __shared__ __align__(128) unsigned char fc_smem[];
    __shared__ __align__(8) unsigned long long bars[RING + 1];
    __shared__ volatile int dead;           // a load never landed: the tile is walked to its end, nothing more is stored
    __shared__ int asked, asked_ny;         // boxes and rows n/2 requested so far (written by thread 0)
    const float* sNy = reinterpret_cast<const float*>(fc_smem + RING * Gm::BUF);
    const uint32_t bar_ny = fk_smem_u32(&bars[RING]);
    const int team = threadIdx.x / Gm::TEAM, tid = threadIdx.x - team * Gm::TEAM, warp = tid >> 5, lane = tid & 31;
    const int gA = tid >> 5, mA = lane;                     // A: plane, pair of columns
    const int tpr = p.tiles_per_row;
    const F2 scale = f2_pack(p.scale, p.scale);
    const bool acc = p.accumulate != 0;

    dep_trigger();
    if (threadIdx.x == 0) {
        for (int s = 0; s <= RING; ++s) fk_mbar_init(fk_smem_u32(&bars[s]), 1);
        dead = asked = asked_ny = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    dep_wait();                     // no global access above this line

    // The boxes of this CTA's tiles form one sequence: the even, then the odd rows of a tile; box b has buffer b % RING.
    int rq_tile = blockIdx.x, rq_box = 0, rq_s = 0;
    auto request = [&]() {          // one thread
        if (rq_tile >= p.num_tiles || dead) return;
        const int row = rq_tile / tpr, c0 = (rq_tile - row * tpr) * G;
        const uint32_t bar = fk_smem_u32(&bars[rq_s]);
        fk_mbar_expect_tx(bar, (uint32_t)Gm::STAGE);
        fk_tma_load_5d(fk_smem_u32(fc_smem + rq_s * Gm::BUF), &tmS, c0, row, rq_box, 0, 0, bar);
        ++asked;
        if (++rq_s == RING) rq_s = 0;
        rq_box ^= 1;
        if (rq_box == 0) rq_tile += gridDim.x;
    };
    auto request_ny = [&](int tile) {       // row n/2, which travels with row 0; one thread
        if (tile >= p.num_tiles || dead) return;
        const int row = tile / tpr, c0 = (tile - row * tpr) * G;
        fk_mbar_expect_tx(bar_ny, (uint32_t)Gm::STAGE_NY);
        fk_tma_load_4d(fk_smem_u32(sNy), &tmNy, c0, row, M, 0, bar_ny);
        ++asked_ny;
    };
    if (threadIdx.x == 0) {
        request();
        request_ny(blockIdx.x);
        request();
        request();
    }
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (!dead && !fk_wait_or_report(bar, parity, p.wait_cycles, p.status)) dead = 1;
    };

    int s0 = 0;                     // buffer of the even rows; the odd rows have the next one
    uint32_t lap = 0, ny_phase = 0; // lap: parity of how often buffer s0 has been used
    for (int tile = blockIdx.x; tile < p.num_tiles; tile += gridDim.x) {
        const int row = tile / tpr, c0 = (tile - row * tpr) * G;
        const int s1 = s0 + 1 == RING ? 0 : s0 + 1, mine = team == 0 ? s0 : s1;
        unsigned char* buf = fc_smem + mine * Gm::BUF;
        wait(fk_smem_u32(&bars[mine]), team == 0 || s1 != 0 ? lap : lap ^ 1u);
        if (team == 0) {
            // The packed row X_0 + i X_{N/2}.  Both rows are Hermitian in kx and their bins kx > N/2 are never read:
            // the thread of kx <= N/2 also forms the value at N - kx.
            wait(bar_ny, ny_phase);
            ny_phase ^= 1u;
            float* st = reinterpret_cast<float*>(buf);
            for (int i = tid; i < G * (M + 1); i += Gm::TEAM) {
                const int g = i & (G - 1), kx = i / G;
                float* a = st + kx * PITCH + g;
                const float x0r = a[0], x0i = a[N * PITCH], xnr = sNy[kx * G + g], xni = sNy[(N + kx) * G + g];
                a[0] = x0r - xni;
                a[N * PITCH] = x0i + xnr;
                if (kx > 0 && kx < M) {
                    float* b = st + (N - kx) * PITCH + g;
                    b[0] = x0r + xni;
                    b[N * PITCH] = xnr - x0i;
                }
            }
            inv64_team_sync(team);
            if (tid == 0) request_ny(tile + gridDim.x);
        }

        // ---- B: rows; lanes run over the planes, then over four adjacent rows ----
        {
            F2 zr[16], zi[16];
            const float* st = reinterpret_cast<const float*>(buf) + (warp >> 1) * 32 + lane;
            auto half = [&](auto Q) __attribute__((always_inline)) {
                constexpr int q = decltype(Q)::value;
                auto first = [&](auto Kk, F2& re, F2& im) __attribute__((always_inline)) {
                    constexpr int k = decltype(Kk)::value;
                    constexpr float c = Tw<64, k>::c, s = Tw<64, k>::s;
                    const float ar = st[k * PITCH], ai = st[(N + k) * PITCH];
                    const float br = st[(M + k) * PITCH], bi = st[(N + M + k) * PITCH];
                    const float dr = ar - br, di = ai - bi;
                    re = f2_pack(ar + br, vfma(-s, di, c * dr));
                    im = f2_pack(ai + bi, vfma(s, dr, c * di));
                };
                static_for<16>([&](auto J) __attribute__((always_inline)) {
                    constexpr int j = decltype(J)::value;
                    F2 ar, ai, br, bi;
                    first(J, ar, ai);
                    first(std::integral_constant<int, j + 16>{}, br, bi);
                    if constexpr (q == 0) {
                        zr[j] = ar + br; zi[j] = ai + bi;
                    } else {
                        const F2 dr = ar - br, di = ai - bi;
                        if constexpr (j == 0) {
                            zr[j] = dr; zi[j] = di;
                        } else {
                            constexpr float c = Tw<32, j>::c, s = Tw<32, j>::s;
                            zr[j] = vfma(-s, di, vmul(c, dr));
                            zi[j] = vfma(s, dr, vmul(c, di));
                        }
                    }
                });
            };
            if ((warp & 1) == 0) half(std::integral_constant<int, 0>{});
            else                 half(std::integral_constant<int, 1>{});
            inv64_team_sync(team);                          // the box is in registers: the buffer takes the rows
            cfft<16, true>(zr, zi);                         // pair m = 2k + q of columns
            ulonglong2* rp = reinterpret_cast<ulonglong2*>(buf) + (lane & (G - 1)) * PP + ((warp >> 1) * (32 / G) + lane / G) * RP + (warp & 1);
            static_for<16>([&](auto K) __attribute__((always_inline)) {
                constexpr int k = decltype(K)::value;
                rp[2 * k] = make_ulonglong2(zr[k].b, zi[k].b);
            });
        }
        inv64_team_sync(team);

        // ---- A: columns; (u[j], v[j]) = (g[j], g[j + 16]) or t[j] ----
        F2 u[16], v[16];
        ulonglong2* col = reinterpret_cast<ulonglong2*>(buf) + gA * PP + mA;
        if (team == 0) {
            F2 Xr[17], Xi[17], g[32];
            static_for<16>([&](auto K) __attribute__((always_inline)) {             // row ky = 2k
                constexpr int k = decltype(K)::value;
                const ulonglong2 x = col[k * RP];
                Xr[k].b = x.x; Xi[k].b = x.y;
            });
            Xr[16] = Xi[0]; Xi[0] = Xi[16] = F2{0};
            // the even rows are in registers: their buffer takes the next tile's odd ones
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            inv64_team_sync(team);
            if (tid == 0) request();
            irfft<32>(Xr, Xi, g);
            static_for<16>([&](auto J) __attribute__((always_inline)) { u[decltype(J)::value] = g[decltype(J)::value]; v[decltype(J)::value] = g[decltype(J)::value + 16]; });
        } else {
            static_for<16>([&](auto Mm) __attribute__((always_inline)) {            // row ky = 4m + 1, above n/2 a conjugate
                constexpr int m = decltype(Mm)::value;
                const ulonglong2 x = col[(m < 8 ? 2 * m : 31 - 2 * m) * RP];
                u[m].b = x.x;
                v[m].b = x.y;
                if constexpr (m >= 8) v[m] = -v[m];
            });
            asm volatile("bar.arrive 3, %0;" ::"n"(Gm::T) : "memory");      // (the rows are in registers: see C)
            cfft<16, true>(u, v);
            static_for<16>([&](auto J) __attribute__((always_inline)) {
                constexpr int j = decltype(J)::value;
                constexpr float c = 2.0f * Tw<64, j>::c, s = 2.0f * Tw<64, j>::s;
                const F2 a = u[j], b = v[j];
                u[j] = vfma(-s, b, vmul(c, a));
                v[j] = vfma(s, a, vmul(c, b));
            });
        }
        // ---- C: team 0 completes j < 8, team 1 the others; what the other team needs passes through the buffer of the odd rows ----
        col = reinterpret_cast<ulonglong2*>(fc_smem + s1 * Gm::BUF) + gA * PP + mA;
        if (team == 0) asm volatile("bar.sync 3, %0;" ::"n"(Gm::T) : "memory");
        static_for<8>([&](auto I) __attribute__((always_inline)) {
            constexpr int i = decltype(I)::value;
            col[(team == 0 ? i : i + 8) * RP] = team == 0 ? make_ulonglong2(u[i + 8].b, v[i + 8].b) : make_ulonglong2(u[i].b, v[i].b);
            if (team == 1) { u[i] = u[i + 8]; v[i] = v[i + 8]; }
        });
        __syncthreads();
        const bool gone = dead;                             // (the waits of this tile are over, those of the next not begun)
        F2 e[8], f[8], tr[8], ti[8];
        static_for<8>([&](auto I) __attribute__((always_inline)) {
            constexpr int i = decltype(I)::value;
            const ulonglong2 x = col[(team == 0 ? i + 8 : i) * RP];
            const F2 a{x.x}, b{x.y};
            e[i] = team == 0 ? u[i] : a;  f[i] = team == 0 ? v[i] : b;
            tr[i] = team == 0 ? a : u[i]; ti[i] = team == 0 ? b : v[i];
        });
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();                                    // the buffer may take another box
        if (gone) break;
        if (threadIdx.x == 0) request();
        {
            // crop: rows [r0, r0 + hc) and columns [x0, x0 + wc) of the transform
            int hc = p.h, wc = p.w, r0 = 0, x0 = 0, pitch = p.w;
            float* base = p.real_out + ((size_t)row * p.C + c0 + gA) * (size_t)(hc * wc);
            if (p.win) {
                const int nt = p.nty * p.ntx, sp = row / nt, t = row - sp * nt, ty = t / p.ntx, tx = t - ty * p.ntx;
                hc = min(hc, p.H - ty * p.step_y);
                wc = min(wc, p.W - tx * p.step_x);
                r0 = p.oy; x0 = p.ox; pitch = p.W;
                base = p.real_out + ((size_t)sp * p.C + c0 + gA) * ((size_t)p.H * p.W) + (size_t)(ty * p.step_y) * p.W + tx * p.step_x;
            }
            const int c = 2 * mA - x0, j0 = team * 8 - r0;  // of this thread's first sample inside the crop
            const bool lo = gA < p.C - c0 && c >= 0 && c < wc, hi = gA < p.C - c0 && c + 1 >= 0 && c + 1 < wc;
            float* o = base + (long long)j0 * pitch + c;
            const bool paired = lo && hi && (((int)(reinterpret_cast<uintptr_t>(o) >> 2) | pitch) & 1) == 0;
            auto rows = [&](auto&& put) __attribute__((always_inline)) {
                static_for<4>([&](auto V) __attribute__((always_inline)) {
                    static_for<8>([&](auto I) __attribute__((always_inline)) {
                        constexpr int w = decltype(V)::value, i = decltype(I)::value;
                        const F2 x = w == 0 ? e[i] + tr[i] : w == 1 ? f[i] - ti[i] : w == 2 ? e[i] - tr[i] : f[i] + ti[i];
                        if ((unsigned)(j0 + i + 16 * w) < (unsigned)hc) put(o + (i + 16 * w) * pitch, f2_mul(x, scale));
                    });
                });
            };
            if (paired) {
                rows([&](float* q, F2 x) __attribute__((always_inline)) {
                    if (acc) x = x + F2{*reinterpret_cast<const unsigned long long*>(q)};
                    *reinterpret_cast<unsigned long long*>(q) = x.b;
                });
            } else if (lo || hi) {
                rows([&](float* q, F2 x) __attribute__((always_inline)) {
                    float a, b;
                    f2_unpack(x, a, b);
                    if (acc) {
                        if (lo) a += q[0];
                        if (hi) b += q[1];
                    }
                    if (lo) q[0] = a;
                    if (hi) q[1] = b;
                });
            }
        }
        if ((s0 += 2) >= RING) { s0 -= RING; lap ^= 1u; }
    }
    if (threadIdx.x == 0 && dead) {
        fk_ring_drain(fk_smem_u32(&bars[0]), RING, asked);
        fk_ring_drain(bar_ny, 1, asked_ny);
    }
}

// A single tile is no faster here than in the plain kernel, whose whole tile is requested at once: 64 tiles 8.7 against
// 9.7 us, 144 9.9 against 10.7, 288 14.7 against 12.8 (57 x 57).  So this kernel takes over where the plain one, with
// its one CTA per SM, would need a second round.
static inline bool inv64_pays(int n, const FftParams& p) {
    constexpr int G = Inv64Geom::G;
    return n == 64 && (long long)p.R * ((p.C + G - 1) / G) > fft_sm_count();
}

static cudaError_t launch_c2r_inv64(FftParams p, cudaStream_t st) {
    using Gm = Inv64Geom;
    if (!fill_tiling<Gm::G>(p)) return cudaErrorInvalidValue;
    CUtensorMap tm, tmny;
    memset(&tm, 0, sizeof(tm));
    memset(&tmny, 0, sizeof(tmny));
    if (!big_make_class_map<64, 2>(&tm, p.spec_in, p, Gm::G) || !big_make_map<64>(&tmny, p.spec_in, p, 1, Gm::G)) return cudaErrorInvalidValue;
    int grid = 0;
    const cudaError_t e = persistent_grid(reinterpret_cast<const void*>(c2r_inv64_kernel), Gm::T, Gm::SMEM, p.num_tiles, &grid);
    if (e != cudaSuccess) return e;
    // Never as a dependent of the contraction: its CTAs are then placed in the order in which SMs come free, neighbouring tiles
    // two by two on one SM, and the loads take longer (158 rows of 159 planes, accGrad 377 -> 333 us without; 298 of 134
    // with 13 x 13 crops 566 -> 459; 297 .. 444 tiles 1.7 us less, 149 .. 296 and 800 .. 1,200 no difference).
    return dep_launch(false, c2r_inv64_kernel, dim3(grid), dim3(Gm::T), Gm::SMEM, st, tm, tmny, p);
}

}  // namespace fc
