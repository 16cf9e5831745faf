// Inverse 2-D C2R transform of large planes (n = 128: the half spectrum of a tile of 8 planes, the least
// that give the frequency-major rows 32 bytes, is 528 KB and does not fit shared memory), and the
// pieces it shares with the forward transform of fft_split.cuh.
//
// The mirror image of the forward transform: a work item is a tile of 8 planes and one eighth of the rows ky,
// those congruent to +-r modulo 16 for class r = 0 .. 7.  The bins of a class add to the samples x[j + 8v]
// (j < 8, v < 16) of a column twice the real part of w_16^{-rv} t_r[j], where t_r is ONE 8-point transform over
// the class's rows, times w_128^{-rj}; class 0 (ky = 0 mod 8) leaves the terms r = 0 and 8 of the same sum.  So
// each class leaves 8 complex values per column, and the last step of a tile is one 16-point real transform per
// (column, j): no 1-D transform spans two items.  The values pass through a scratch area in global memory,
// 512 KB per tile in flight, rewritten for every tile; the spectra, read once, and the result pass through the
// L2 as first to leave, so that the scratch stays there.
// A tile belongs to a cluster of CL = 1, 2, 4 or 8 CTAs, which share its classes and then its planes (big_cluster).
//
// Per item, 512 threads, packed fp32 pairs (f32x2.cuh) of two adjacent columns:
//   B. the two residues of a class arrive as TMA boxes of 8 planes x 4 rows, in a ring of six; a team of 8 warps per
//      box, eight threads per row: the first butterfly of a decimation in frequency yields the even and the odd
//      columns, the two halves of a packed value; 8 points, a twiddle, an exchange in shared memory, 8 points,
//      written back in place;
//   A. thread = (plane, pair of columns): 8 rows, 8-point FFT, twiddle, coalesced 16-byte stores to the scratch.
//   C. after the last item, thread = (pair of columns, j): 16-point transform, scale, cropped rows to the result.
// Row ky = 0 carries ky = n/2 as (re, im) (Section 5.2).  Only the columns and rows inside the crop are computed from
// A on, so that a filter gradient costs little more than the spectrum's loads.
//
// Bound by the chain of an item: at 6,500 - 8,500 cycles per 64 KB it is 1.5 - 2 times what its loads take (4,400); the
// shared-memory pipe is busy for 2,600 of them.  Against whole rows and whole columns, with the half spectrum of a
// tile in the scratch and two lanes of a warp per column: 4,096 planes of 128 x 128 226 -> 183 us, 12,288 of 118 x 118
// 663 -> 545, 91 of 97 x 101 20.6 -> 15.4; 4,096 filter gradients of 5 x 5 176 -> 128.  Tried and not kept: four classes
// with 16-point transforms (195 and 135 us: one item's loads ahead instead of two); a 17th warp for the loads (no
// registers left for step C; 20.5 against 15.4 us for 91 planes).
#pragma once

#include "fft_kernels.cuh"

namespace fc {

constexpr int BIG_MAX_SMS = 160;  // scratch is sized for this many tiles in flight

struct BigGeom {
    static constexpr int N = 128, M = 64, NC = 65, G = 8, T = 512, TEAM = 256, CLASSES = 8, HI = 4, RING = 6;
    static constexpr size_t STAGE = (size_t)2 * N * HI * G * 4;  // a box: [part*N + kx][hi][plane]
    // the same box as rows of 64 pairs of columns in 16-byte units (re, re', im, im'); pair m = a + 8b stands at 9a + b:
    // lanes over the planes (B) and lanes over the pairs (A) are conflict-free
    static constexpr int RP = 72, PP = HI * RP + 1;
    static constexpr size_t ROWS = (size_t)G * PP * 16;
    static constexpr size_t BUF = ((ROWS > STAGE ? ROWS : STAGE) + 127) / 128 * 128;
    static constexpr size_t STAGE_NY = (size_t)2 * N * G * 4;
    static constexpr size_t SMEM = RING * BUF + STAGE_NY;
    // scratch of a tile: [class][plane][j][pair], 16 bytes each
    static constexpr int S_J = 64, S_PLANE = 8 * S_J, S_CLASS = G * S_PLANE;
    static constexpr size_t SCRATCH_PER_TILE = (size_t)CLASSES * S_CLASS * 16;
};

static inline size_t big_scratch_bytes(int n) {
    return n == 128 ? (size_t)BIG_MAX_SMS * BigGeom::SCRATCH_PER_TILE : 0;
}

// Planar spectrum [2][N][NC][R][ld] seen as a 4-D tensor (col, row, ky, part*N + kx):
// bin = kx*NC + ky and the parts are N*NC bins apart, so the last stride is uniform.
template <int N>
static bool big_make_map(CUtensorMap* map, const float* spec, const FftParams& p, int box_ky, int planes = 8) {
    tc_encode_fn enc = tc_get_encode();
    if (!enc) return false;
    constexpr int NC = N / 2 + 1;
    const cuuint64_t mat = (cuuint64_t)p.R * p.ld * 4;
    cuuint64_t dims[4] = {(cuuint64_t)p.C, (cuuint64_t)p.R, (cuuint64_t)NC, (cuuint64_t)2 * N};
    cuuint64_t strides[3] = {(cuuint64_t)p.ld * 4, mat, mat * NC};
    cuuint32_t box[4] = {(cuuint32_t)planes, 1u, (cuuint32_t)box_ky, (cuuint32_t)2 * N};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(spec), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// w_64^{t k} (between the two 8-point steps of a row of 64 pairs), both components duplicated for packed
// operations, and w_128^{t + 8r} (the butterfly between the halves of a pair)
struct BigTwiddles { unsigned long long c[8][8], s[8][8]; float ec[8][8], es[8][8]; };
constexpr BigTwiddles make_big_twiddles() {
    BigTwiddles w{};
    for (int t = 0; t < 8; ++t)
        for (int k = 0; k < 8; ++k) {
            w.c[t][k] = f2_const(static_cast<float>(cx_cos2pi(t * k, 64)));
            w.s[t][k] = f2_const(static_cast<float>(cx_sin2pi(t * k, 64)));
            w.ec[t][k] = static_cast<float>(cx_cos2pi(t + 8 * k, 128));
            w.es[t][k] = static_cast<float>(cx_sin2pi(t + 8 * k, 128));
        }
    return w;
}
__constant__ BigTwiddles c_big_tw = make_big_twiddles();
// (re, im) times w = (c, -s)
__device__ __forceinline__ void big_rotate(F2& re, F2& im, unsigned long long c_, unsigned long long s_) {
    const F2 c{c_}, s{s_};
    const F2 x = f2_fma(s, im, f2_mul(c, re));
    im = f2_mul(c, im) - f2_mul(s, re);
    re = x;
}
// [2][N][NC][R][ld] as (col, row, lo, hi, part*N + kx) with ky = L hi + lo; boxes of all hi
template <int N, int L>
static bool big_make_class_map(CUtensorMap* map, const float* spec, const FftParams& p, int planes = 8) {
    tc_encode_fn enc = tc_get_encode();
    if (!enc) return false;
    constexpr int NC = N / 2 + 1, HI = N / 2 / L;
    const cuuint64_t mat = (cuuint64_t)p.R * p.ld * 4;
    cuuint64_t dims[5] = {(cuuint64_t)p.C, (cuuint64_t)p.R, L, HI, (cuuint64_t)2 * N};
    cuuint64_t strides[4] = {(cuuint64_t)p.ld * 4, mat, mat * L, mat * NC};
    cuuint32_t box[5] = {(cuuint32_t)planes, 1u, 1u, (cuuint32_t)HI, (cuuint32_t)2 * N};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float*>(spec), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
__device__ __forceinline__ void fk_tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1,
                                                int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
        ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void fk_tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                               int c2, int c3, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// The same for data that a kernel reads once: its lines are the first to leave the L2.
__device__ __forceinline__ void fk_tma_load_4d_once(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                                    int c2, int c3, uint32_t bar) {
    unsigned long long once;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(once)
        : "memory");
}
__device__ __forceinline__ void fk_tma_load_5d_once(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                                    int c4, uint32_t bar) {
    unsigned long long once;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "l"(once)
        : "memory");
}
// Barrier over the CTAs of a tile; orders their accesses to the scratch.
__device__ __forceinline__ void big_tile_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Barrier over the team that works on one box.
__device__ __forceinline__ void big_team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(BigGeom::TEAM) : "memory");
}

// Phase A of class R: 8 rows of a pair of columns (row(box, hi) -> 16-byte unit), 8-point FFT, twiddle; put(j, value).
// release() comes when the rows are in registers.
template <int R, class Row, class Release, class Put>
__device__ __forceinline__ void big_column(Row&& row, Release&& release, Put&& put) {
    if constexpr (R == 0) {
        F2 Xr[9], Xi[9], g[16];
        static_for<8>([&](auto K) __attribute__((always_inline)) {              // row ky = 8k
            constexpr int k = decltype(K)::value;
            const ulonglong2 v = row(k & 1, k / 2);
            Xr[k].b = v.x; Xi[k].b = v.y;
        });
        Xr[8] = Xi[0]; Xi[0] = Xi[8] = F2{0};
        release();
        irfft<16>(Xr, Xi, g);
        static_for<8>([&](auto J) __attribute__((always_inline)) {              // terms 0 and 8 of the last step
            constexpr int j = decltype(J)::value;
            put(J, make_ulonglong2(vmul(0.5f, g[j] + g[j + 8]).b, vmul(0.5f, g[j] - g[j + 8]).b));
        });
    } else {
        F2 ar[8], ai[8];
        static_for<8>([&](auto Mm) __attribute__((always_inline)) {             // row ky = 16m + R, above n/2 a conjugate
            constexpr int m = decltype(Mm)::value;
            const ulonglong2 v = m < 4 ? row(0, m) : row(1, 7 - m);
            ar[m].b = v.x;
            ai[m].b = v.y;
            if constexpr (m >= 4) ai[m] = -ai[m];
        });
        release();
        cfft<8, true>(ar, ai);
        static_for<8>([&](auto J) __attribute__((always_inline)) {
            constexpr int j = decltype(J)::value;
            if constexpr (j == 0) {
                put(J, make_ulonglong2(ar[0].b, ai[0].b));
            } else {
                constexpr float c = Tw<128, R * j>::c, s = Tw<128, R * j>::s;
                put(J, make_ulonglong2(vfma(-s, ai[j], vmul(c, ar[j])).b, vfma(s, ar[j], vmul(c, ai[j])).b));
            }
        });
    }
}

__global__ void __launch_bounds__(BigGeom::T, 1)
c2r_big_kernel(const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmNy,
               const __grid_constant__ FftParams p, ulonglong2* __restrict__ scratch_all, const int cl) {
    using Gm = BigGeom;
    constexpr int N = Gm::N, M = Gm::M, G = Gm::G, RP = Gm::RP, PP = Gm::PP, RING = Gm::RING, PITCH = Gm::HI * G;
    extern __shared__ __align__(128) unsigned char fc_smem[];
    __shared__ __align__(8) unsigned long long bars[RING + 1];
    __shared__ volatile int dead;           // a load never landed: the tile is walked to its end, nothing more is stored
    __shared__ int asked, asked_ny;         // boxes and rows n/2 requested so far (written by thread 0)
    const float* sNy = reinterpret_cast<const float*>(fc_smem + RING * Gm::BUF);
    const uint32_t bar_ny = fk_smem_u32(&bars[RING]);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t = warp & 7, team = warp >> 3;               // B: part of the row, box
    const int gA = tid >> 6, mA = tid & 63;                 // A: plane, pair of columns; C: j, pair of columns
    const int hc = p.h, wc = p.w, hw = hc * wc, tpr = p.tiles_per_row;
    const int pairs = (wc + 1) >> 1, nj = min(8, hc);       // inside the crop
    const F2 scale = f2_pack(p.scale, p.scale);
    const int rank = (int)blockIdx.x % cl, group = (int)blockIdx.x / cl, groups = (int)gridDim.x / cl;
    const int K = Gm::CLASSES / cl;                         // items of a tile that this CTA takes
    ulonglong2* scratch = scratch_all + (size_t)group * (Gm::SCRATCH_PER_TILE / 16);
    const int tiles = group < p.num_tiles ? (p.num_tiles - group + groups - 1) / groups : 0;
    const int items = K * tiles;

    dep_trigger();
    if (tid == 0) {
        for (int s = 0; s <= RING; ++s) fk_mbar_init(fk_smem_u32(&bars[s]), 1);
        dead = asked = asked_ny = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    dep_wait();                     // no global access above this line

    // The items of this CTA over all its tiles form one sequence; item i has buffers 2i and 2i + 1 modulo RING.
    auto request = [&](int i) {     // one thread
        if (i >= items || dead) return;
        const int tile = group + (i / K) * groups, cls = rank * K + i % K, s = 2 * i % RING;
        const int row = tile / tpr, c0 = (tile - row * tpr) * G;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint32_t bar = fk_smem_u32(&bars[s + b]);
            fk_mbar_expect_tx(bar, (uint32_t)Gm::STAGE);
            fk_tma_load_5d_once(fk_smem_u32(fc_smem + (s + b) * Gm::BUF), &tmS, c0, row, b == 0 ? cls : (cls == 0 ? 8 : 16 - cls), 0, 0, bar);
        }
        asked += 2;
    };
    auto request_ny = [&](int tile) {       // row n/2, which travels with row 0; one thread
        if (rank != 0 || tile >= p.num_tiles || dead) return;
        const int row = tile / tpr, c0 = (tile - row * tpr) * G;
        fk_mbar_expect_tx(bar_ny, (uint32_t)Gm::STAGE_NY);
        fk_tma_load_4d_once(fk_smem_u32(sNy), &tmNy, c0, row, M, 0, bar_ny);
        ++asked_ny;
    };
    if (tid == 0) {
        request(0);
        request_ny(group);
        request(1);
        request(2);
    }
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (!dead && !fk_wait_or_report(bar, parity, p.wait_cycles, p.status)) dead = 1;
    };

    int i = 0;
    uint32_t ny_phase = 0;
    bool gone = false;              // from then on only the cluster's barriers are walked
    for (int tile = group; tile < p.num_tiles; tile += groups) {
        const int row = tile / tpr, c0 = (tile - row * tpr) * G;
        const int gcount = min(G, p.C - c0);
#pragma unroll 1
        for (int k = 0; k < K && !gone; ++k, ++i) {
            const int cls = rank * K + k, s = 2 * i % RING;
            // ---- B: rows of one residue ----
            {
                unsigned char* buf = fc_smem + (s + team) * Gm::BUF;
                wait(fk_smem_u32(&bars[s + team]), (uint32_t)(2 * i / RING) & 1u);
                if (cls == 0 && team == 0) wait(bar_ny, ny_phase);
                F2 zr[8], zi[8];
                {
                    const float* st = reinterpret_cast<const float*>(buf) + t * PITCH + lane;
                    const bool packed = cls == 0 && team == 0 && lane < G;              // row ky = 0
                    const float* ny = sNy + t * G + (lane & 7);
                    static_for<8>([&](auto U) {
                        constexpr int u = decltype(U)::value;
                        float ar = st[(8 * u) * PITCH], ai = st[(N + 8 * u) * PITCH];
                        float br = st[(M + 8 * u) * PITCH], bi = st[(N + M + 8 * u) * PITCH];
                        if (packed) {       // X_0 + i X_{N/2}: one complex row that carries both real rows
                            ar -= ny[(N + 8 * u) * G];      ai += ny[(8 * u) * G];
                            br -= ny[(N + M + 8 * u) * G];  bi += ny[(M + 8 * u) * G];
                        }
                        // even columns from the sum, odd ones from the difference times w_128^{-(t + 8u)}
                        const float c = c_big_tw.ec[t][u], sn = c_big_tw.es[t][u];
                        const float dr = ar - br, di = ai - bi;
                        zr[u] = f2_pack(ar + br, vfma(-sn, di, c * dr));
                        zi[u] = f2_pack(ai + bi, vfma(sn, dr, c * di));
                    });
                }
                cfft<8, true>(zr, zi);
                big_team_sync(team);                        // the box is in registers: the buffer takes the rows
                ulonglong2* rp = reinterpret_cast<ulonglong2*>(buf) + (lane & 7) * PP + (lane >> 3) * RP;
                static_for<8>([&](auto U) {
                    constexpr int u = decltype(U)::value;
                    if constexpr (u > 0) {                  // w_64^{-t u}
                        const F2 c{c_big_tw.c[t][u]}, sn{c_big_tw.s[t][u]};
                        const F2 x = f2_mul(c, zr[u]) - f2_mul(sn, zi[u]);
                        zi[u] = f2_fma(sn, zr[u], f2_mul(c, zi[u]));
                        zr[u] = x;
                    }
                    rp[9 * u + t] = make_ulonglong2(zr[u].b, zi[u].b);
                });
                big_team_sync(team);
                static_for<8>([&](auto U) {
                    const ulonglong2 v = rp[9 * t + decltype(U)::value];
                    zr[decltype(U)::value].b = v.x; zi[decltype(U)::value].b = v.y;
                });
                cfft<8, true>(zr, zi);                      // pair m = t + 8u of columns
                static_for<8>([&](auto U) {
                    constexpr int u = decltype(U)::value;
                    rp[9 * t + u] = make_ulonglong2(zr[u].b, zi[u].b);
                });
            }
            __syncthreads();
            // ---- A: columns ----
            {
                const ulonglong2* r0 = reinterpret_cast<const ulonglong2*>(fc_smem + s * Gm::BUF) + gA * PP + 9 * (mA & 7) + (mA >> 3);
                auto rowv = [&](int box, int hi) __attribute__((always_inline)) { return r0[box * (int)(Gm::BUF / 16) + hi * RP]; };
                auto release = [&]() __attribute__((always_inline)) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncthreads();                        // the rows are in registers: the buffers take the item after next
                    if (tid == 0) {
                        request(i + RING / 2);
                        if (cls == 0) request_ny(tile + groups);
                    }
                };
                ulonglong2* dst = scratch + (size_t)cls * Gm::S_CLASS + gA * Gm::S_PLANE + mA;
                const int live = gA < gcount && mA < pairs ? nj : 0;
                auto put = [&](auto J, ulonglong2 v) __attribute__((always_inline)) {
                    constexpr int j = decltype(J)::value;
                    if (j < live) __stcg(dst + j * Gm::S_J, v);
                };
                switch (cls) {
                    case 0: big_column<0>(rowv, release, put); break;
                    case 1: big_column<1>(rowv, release, put); break;
                    case 2: big_column<2>(rowv, release, put); break;
                    case 3: big_column<3>(rowv, release, put); break;
                    case 4: big_column<4>(rowv, release, put); break;
                    case 5: big_column<5>(rowv, release, put); break;
                    case 6: big_column<6>(rowv, release, put); break;
                    default: big_column<7>(rowv, release, put); break;
                }
            }
        }
        if (rank == 0) ny_phase ^= 1u;
        big_tile_sync();                                    // the scratch is complete
        gone = dead;

        // ---- C: last step of the columns, crop ----
        if (!gone && gA < nj && mA < pairs) {
            const int j = gA, m = mA;
            const ulonglong2* src = scratch + j * Gm::S_J + m;
#pragma unroll 1
            for (int g0 = rank; g0 < gcount; g0 += 2 * cl) {
                ulonglong2 in[2][8];                        // two planes' loads in flight
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (g0 + b * cl < gcount)
#pragma unroll
                        for (int r = 0; r < 8; ++r) in[b][r] = __ldcg(src + r * Gm::S_CLASS + (g0 + b * cl) * Gm::S_PLANE);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int g = g0 + b * cl;
                    if (g >= gcount) break;
                    F2 Xr[9], Xi[9], x[16];
                    Xr[0].b = in[b][0].x; Xr[8].b = in[b][0].y; Xi[0] = Xi[8] = F2{0};
#pragma unroll
                    for (int r = 1; r < 8; ++r) { Xr[r].b = in[b][r].x; Xi[r].b = in[b][r].y; }
                    irfft<16>(Xr, Xi, x);                   // row j + 8v
                    float* const plane = p.real_out + ((size_t)row * p.C + c0 + g) * hw;
                    float* o = plane + (size_t)j * wc + 2 * m;
                    const int step = 8 * wc;
                    if (((wc | ((int)(reinterpret_cast<uintptr_t>(plane) >> 2))) & 1) == 0) {
#pragma unroll
                        for (int v = 0; v < 16; ++v, o += step) {
                            if (j + 8 * v >= hc) break;
                            F2 z = f2_mul(x[v], scale);
                            if (p.accumulate) z = z + F2{*reinterpret_cast<const unsigned long long*>(o)};
                            float lo, hi;
                            f2_unpack(z, lo, hi);
                            __stcs(reinterpret_cast<float2*>(o), make_float2(lo, hi));
                        }
                    } else {
                        const bool two = 2 * m + 1 < wc;
#pragma unroll
                        for (int v = 0; v < 16; ++v, o += step) {
                            if (j + 8 * v >= hc) break;
                            float lo, hi;
                            f2_unpack(f2_mul(x[v], scale), lo, hi);
                            if (p.accumulate) {
                                lo += *o;
                                if (two) hi += o[1];
                            }
                            __stcs(o, lo);
                            if (two) __stcs(o + 1, hi);
                        }
                    }
                }
            }
        }
        big_tile_sync();                                    // the scratch may be rewritten
    }
    if (tid == 0 && dead) {
        fk_ring_drain(fk_smem_u32(&bars[0]), RING, asked);
        fk_ring_drain(bar_ny, 1, asked_ny);
    }
}

// CTAs that share a tile: as many as find SMs (clusters of eight and four stay inside a GPC, so that not all SMs can
// hold them), else two, whose rounds are finer than those of one; one where a round of single CTAs takes all tiles and
// these are less than half full, so that step C, which a pair would share, is short.
// Planes of 120 x 120, us with 1 / 2 / 4 / 8 CTAs: 3 tiles 48 / 30 / 19.5 / 15; 18 tiles 48 / 30 / 20.5 / 25.5; 36 tiles
// 49 / 30 / 36 / 40; 144 tiles 63.5 / 58 / 102 / 141; 512 tiles 234 / 179 / 375 / 487.  96 tiles of 3 planes 36 / 40 / 46 / 77.
static inline int big_cluster(long long tiles, int planes, int slots) {
    if (16 * tiles <= slots) return 8;
    if (6 * tiles <= slots) return 4;
    return 2 * tiles > slots && tiles <= slots && 2 * planes <= BigGeom::G ? 1 : 2;
}

static cudaError_t launch_c2r_big(FftParams p, float* scratch, size_t scratch_bytes, cudaStream_t st) {
    using Gm = BigGeom;
    if (!fill_tiling<Gm::G>(p)) return cudaErrorInvalidValue;
    CUtensorMap tm, tmny;
    memset(&tm, 0, sizeof(tm));
    memset(&tmny, 0, sizeof(tmny));
    if (!big_make_class_map<128, 16>(&tm, p.spec_in, p) || !big_make_map<128>(&tmny, p.spec_in, p, 1))
        return cudaErrorInvalidValue;
    int slots = 0;
    const cudaError_t e = persistent_grid(reinterpret_cast<const void*>(c2r_big_kernel), Gm::T, Gm::SMEM, 1 << 20, &slots);
    if (e != cudaSuccess) return e;
    const int cl = big_cluster(p.num_tiles, p.C, slots);
    long long groups = slots / cl;
    if (groups < 1) groups = 1;
    if (groups > p.num_tiles) groups = p.num_tiles;
    const long long fit = (long long)(scratch_bytes / Gm::SCRATCH_PER_TILE);
    if (fit < 1) return cudaErrorInvalidValue;
    if (groups > fit) groups = fit;
    const dim3 grid((unsigned)(groups * cl));
    ulonglong2* sc = reinterpret_cast<ulonglong2*>(scratch);
    return dep_launch({p.overlap != 0, cl}, c2r_big_kernel, grid, dim3(Gm::T), Gm::SMEM, st, tm, tmny, p, sc, cl);
}

// Which plane sizes take the transforms of this file and fft_split.cuh.
static inline bool big_planes(int n) { return n == 128; }

}  // namespace fc
