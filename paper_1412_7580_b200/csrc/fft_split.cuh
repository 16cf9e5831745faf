// Forward 2-D R2C transform of large planes (n = 128) with the rows ky split over CTAs.
//
// The half spectrum of a tile of 8 planes (528 KB) does not fit shared memory, and 8 planes are the
// least that give the frequency-major rows the 32 bytes the memory system needs.  So a work item is
// a tile of 8 planes and ONE FOURTH of the rows ky: the rows (r, 8 - r) mod 8 for class r = 0 .. 3.
// Every item reads all samples of its planes -- the four items of a tile run next to each other, so
// that the samples come from HBM once and from the L2 three times -- but computes only its own rows:
// the first butterflies of a decimation in frequency leave 16 of the 128 points of a column, one
// 16-point transform yields the rows ky = 8m + r, m < 16, and those above n/2 are the conjugates of
// the rows 8m' + (8 - r) (Section 5.2: Hermitian symmetry).  No work is done twice, except loads, and
// nothing passes through a scratch area between the two 1-D passes.
//
// Per item, 512 threads, packed fp32 pairs (f32x2.cuh) of two adjacent columns:
//   A. thread = (plane, pair of columns): coalesced loads straight into the first butterflies, 16-point FFT,
//      16 rows to shared memory ([plane][row][pair], 16 bytes per element);
//   B. thread = (row, t of 8): a row of 64 pairs is 8 pairs per thread, a twiddle, an exchange in place (the
//      slots a thread writes are the slots it has read), 8 more points; the halves of a pair are then the
//      transforms of the even and the odd columns and one last butterfly between them completes the row.
//      Results form the staging tile [lo][part * n + kx][hi][plane], which overlays the rows;
//   C. one TMA store per residue lo of the rows (ky = 8 hi + lo): boxes of 8 planes x 8 hi x 2n.
// Row ky = 0 carries ky = n/2 as (re, im) and is taken apart in the staging tile.  The store of an
// item overlaps phase A of the next, whose samples are requested into the L2 one item ahead.
//
// What bounds it: the samples, 4 x the planes, come from the L2 into the SMs in phase A (about 40 bytes per
// cycle and SM; 8-byte loads of that pattern reach 46 - 55), and phase B, during which nothing is loaded.
// Pairs of columns instead of pairs of planes halve the loads, and what counts as much, the loads are kept in
// program order 24 samples ahead of their use (SplitLoad): 4,096 planes of 128 x 128 209 -> 145 us, 12,288 of
// 118 x 118 602 -> 440, 4,096 of 97 x 101 (4-byte loads) 201 -> 145, 12 planes of 128 x 128 33 -> 18 us.  16 and
// 32 samples ahead: 150 and 145 us, 434 and 457.  Tried and not kept: the compiler's own order of the loads (181 us,
// 435 for 97 x 101); teams of 8 warps for A and B with half a tile between them (200 us: fewer loads in flight); four
// planes per item, stored in rows of 16 bytes (390 us); a tile's four items one after the other in one CTA (280 us).
#pragma once

#include "fft_big.cuh"

namespace fc {

struct SplitGeom {
    static constexpr int N = 128, M = 64, NC = 65, G = 8, T = 512, CLASSES = 4;
    static constexpr int CP = N / 2;                     // pairs of columns in a row
    static constexpr int RP = CP;                        // 16-byte units per row: (re, re', im, im') of a pair of columns
    static constexpr int PP = 16 * RP + 1;               // per plane; odd: lanes that run over the planes are conflict-free
    static constexpr size_t MID = (size_t)G * PP * 16;
    static constexpr size_t STAGE = (size_t)2 * 2 * N * 8 * G * 4;
    static constexpr size_t BUF = ((MID > STAGE ? MID : STAGE) + 127) / 128 * 128;
    static constexpr size_t NY = (size_t)2 * N * G * 4;
    static constexpr size_t SMEM = BUF + NY;
};

// Last step of a row: E and O, the transforms of the even and the odd columns, are the two halves of a packed
// value; X_q = E + w_N^q O and X_{q + N/2} = E - w_N^q O, w = (c, -s).
__device__ __forceinline__ void split_last(F2 re, F2 im, float c, float s, float& ar, float& ai, float& br, float& bi) {
    float er, orr, ei, oi;
    f2_unpack(re, er, orr);
    f2_unpack(im, ei, oi);
    ar = vfma(s, oi, vfma(c, orr, er));
    ai = vfma(-s, orr, vfma(c, oi, ei));
    br = vfma(2.0f, er, -ar);
    bi = vfma(2.0f, ei, -ai);
}

__device__ __forceinline__ void fk_tma_store_5d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];"
        ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

// The samples of two adjacent columns, row by row: one 8-byte load where the pair is so aligned, two of 4
// bytes else; rows and columns past the plane are zeros.  The loads are volatile, so that they are issued in
// program order, well ahead of their use (split_column): left to itself the compiler puts each load right
// before its use and a thread has a few in flight.
template <bool PAIR>
struct SplitLoad {
    const float* s0;
    int pitch;                      // bytes from row to row
    int rows, rows2;                // rows that exist in the first and in the second column
    template <int r>
    __device__ __forceinline__ F2 get() const {
        const char* q = reinterpret_cast<const char*>(s0) + (long long)pitch * r;
        if constexpr (PAIR) {
            F2 v;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\tmov.b64 %0, 0;\n\t@p ld.global.nc.b64 %0, [%1];\n\t}"
                         : "=l"(v.b) : "l"(q), "r"(rows), "n"(r));
            return v;
        } else {
            float u, v;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.b32 %0, [%1];\n\t}"
                         : "=f"(u) : "l"(q), "r"(rows), "n"(r));
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.b32 %0, [%1+4];\n\t}"
                         : "=f"(v) : "l"(q), "r"(rows2), "n"(r));
            return f2_pack(u, v);
        }
    }
};

// Phase A of class R: first butterflies of a column, twiddles, 16-point FFT; put(row, re, im) with row = 8 *
// (second residue) + hi; release() comes before the first put.  The samples of the next AHEAD butterflies are on
// their way.
template <int R, bool PAIR, class Release>
__device__ __forceinline__ void split_column(const SplitLoad<PAIR>& x, ulonglong2* dst, Release&& release) {
    constexpr int AHEAD = 3;
    auto put = [&](auto K, F2 re, F2 im) __attribute__((always_inline)) { dst[decltype(K)::value * SplitGeom::RP] = make_ulonglong2(re.b, im.b); };
    F2 ring[AHEAD][8];
    auto fetch = [&](auto J) __attribute__((always_inline)) {
        constexpr int j = decltype(J)::value;
        static_for<8>([&](auto V) __attribute__((always_inline)) { ring[j % AHEAD][decltype(V)::value] = x.template get<j + 16 * decltype(V)::value>(); });
    };
    static_for<AHEAD>(fetch);
    F2 ar[R == 0 ? 32 : 16], ai[16];
    static_for<16>([&](auto J) __attribute__((always_inline)) {
        constexpr int j = decltype(J)::value;
        const F2 (&v)[8] = ring[j % AHEAD];
        if constexpr (R == 0) {
            ar[j] = (v[0] + v[4]) + (v[2] + v[6]);
            ar[j + 16] = (v[1] + v[5]) + (v[3] + v[7]);
        } else {
            F2 re, im;                                      // sum_v x_v w_8^{R v}
            if constexpr (R == 2) {
                re = (v[0] + v[4]) - (v[2] + v[6]);
                im = (v[3] + v[7]) - (v[1] + v[5]);
            } else {
                constexpr float s = Tw<8, 1>::c;
                const F2 d0 = v[0] - v[4], d1 = v[1] - v[5], d3 = v[3] - v[7];
                if constexpr (R == 1) {
                    re = vfma(s, d1 - d3, d0);
                    im = vfma(-s, d1 + d3, v[6] - v[2]);
                } else {
                    re = vfma(s, d3 - d1, d0);
                    im = vfma(-s, d1 + d3, v[2] - v[6]);
                }
            }
            if constexpr (j == 0) {
                ar[0] = re; ai[0] = im;
            } else {
                constexpr float c = Tw<128, R * j>::c, sn = Tw<128, R * j>::s;
                ar[j] = vfma(sn, im, vmul(c, re));
                ai[j] = vfma(-sn, re, vmul(c, im));
            }
        }
        if constexpr (j + AHEAD < 16) fetch(std::integral_constant<int, j + AHEAD>{});
    });
    if constexpr (R == 0) {
        F2 Xr[17], Xi[17];
        rfft<32>(ar, Xr, Xi);                               // X[k] = row ky = 4k
        release();
        put(std::integral_constant<int, 0>{}, Xr[0], Xr[16]);
        static_for<15>([&](auto K) __attribute__((always_inline)) {
            constexpr int k = decltype(K)::value + 1;
            put(std::integral_constant<int, (k & 1) * 8 + k / 2>{}, Xr[k], Xi[k]);
        });
    } else {
        cfft<16, false>(ar, ai);                            // row ky = 8m + R
        release();
        static_for<16>([&](auto Mm) __attribute__((always_inline)) {
            constexpr int m = decltype(Mm)::value;
            if constexpr (m < 8) put(std::integral_constant<int, m>{}, ar[m], ai[m]);
            else put(std::integral_constant<int, 8 + 15 - m>{}, ar[m], -ai[m]);
        });
    }
}
template <bool PAIR, class Release>
__device__ __forceinline__ void split_class(int cls, const SplitLoad<PAIR>& x, ulonglong2* dst, Release&& release) {
    if (cls == 0)      split_column<0>(x, dst, release);
    else if (cls == 1) split_column<1>(x, dst, release);
    else if (cls == 2) split_column<2>(x, dst, release);
    else               split_column<3>(x, dst, release);
}

// Requests an item's share (two planes) of its tile's samples into the L2.
__device__ __forceinline__ void split_prefetch(int item, int items0, const FftParams& p0, const FftParams& p1) {
    using Gm = SplitGeom;
    const bool second = item >= items0;
    const FftParams& p = second ? p1 : p0;
    const int it = second ? item - items0 : item;
    const int tile = it / Gm::CLASSES, cls = it - tile * Gm::CLASSES;
    const int row = tile / p.tiles_per_row, c0 = (tile - row * p.tiles_per_row) * Gm::G;
    constexpr int PART = Gm::G / Gm::CLASSES;
    const int planes = min(PART, p.C - c0 - cls * PART);
    if (planes <= 0) return;
    const uintptr_t a = reinterpret_cast<uintptr_t>(p.real_in + ((size_t)row * p.C + c0 + cls * PART) * (size_t)(p.h * p.w));
    const uintptr_t lo = (a + 15) & ~(uintptr_t)15, hi = (a + (size_t)planes * p.h * p.w * 4) & ~(uintptr_t)15;
    if (hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo)) : "memory");
}

__global__ void __launch_bounds__(SplitGeom::T, 1)
r2c_split_kernel(const __grid_constant__ CUtensorMap tmS0, const __grid_constant__ CUtensorMap tmNy0,
                 const __grid_constant__ CUtensorMap tmS1, const __grid_constant__ CUtensorMap tmNy1,
                 const __grid_constant__ FftParams p0, const __grid_constant__ FftParams p1) {
    using Gm = SplitGeom;
    constexpr int N = Gm::N, M = Gm::M, G = Gm::G, CP = Gm::CP, RP = Gm::RP, PP = Gm::PP, T = Gm::T;
    extern __shared__ __align__(128) unsigned char fc_smem[];
    ulonglong2* sMid = reinterpret_cast<ulonglong2*>(fc_smem);
    float* sStage = reinterpret_cast<float*>(fc_smem);
    float* sNy = reinterpret_cast<float*>(fc_smem + Gm::BUF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gA = tid / CP, cA = 2 * (tid - gA * CP);      // A: plane, first of two columns
    const int t = warp & 7, rg0 = warp >> 3;                // B: part of the row, group of four rows
    ulonglong2* rowp = sMid + (lane & 7) * PP + (rg0 * 4 + (lane >> 3)) * RP;
    const int items0 = Gm::CLASSES * p0.num_tiles, items = items0 + Gm::CLASSES * p1.num_tiles;

    dep_trigger();
    dep_wait();                     // no global access above this line

    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const bool second = item >= items0;
        const FftParams& p = second ? p1 : p0;
        const int it = second ? item - items0 : item;
        const int tile = it / Gm::CLASSES, cls = it - tile * Gm::CLASSES;
        const int row = tile / p.tiles_per_row, c0 = (tile - row * p.tiles_per_row) * G;
        const int h = p.h, w = p.w;
        if (tid == 32 && item + (int)gridDim.x < items) split_prefetch(item + gridDim.x, items0, p0, p1);

        // ---- A: columns; a pair of columns past the plane reads no sample and writes zeros ----
        {
            const float* planes = p.real_in + ((size_t)row * p.C + c0) * (size_t)(h * w);
            const bool live = gA < p.C - c0 && cA < w;
            const float* s0 = planes + (live ? gA * (h * w) + cA : 0);
            const int rows = live ? h : 0, rows2 = live && cA + 1 < w ? h : 0;
            ulonglong2* dst = sMid + gA * PP + (cA >> 1);
            auto release = [&]() __attribute__((always_inline)) {  // the previous item's store has read the buffer
                if (tid == 0) fk_bulk_wait_read();
                __syncthreads();
            };
            if (((w & 1) | ((int)(reinterpret_cast<uintptr_t>(planes) >> 2) & 1)) == 0)
                split_class(cls, SplitLoad<true>{s0, 4 * w, rows, rows2}, dst, release);
            else
                split_class(cls, SplitLoad<false>{s0, 4 * w, rows, rows2}, dst, release);
        }
        __syncthreads();

        // ---- B: rows; lanes run over the planes, then over four adjacent rows hi.  Eight threads per row of 64
        // pairs: 8 points, twiddle, an exchange in place (the slots a thread writes are the slots it has read),
        // 8 points; a warp takes two groups of four rows ----
        F2 zr[2][8], zi[2][8];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            ulonglong2* rp = rowp + b * 8 * RP;
            static_for<8>([&](auto U) {
                const ulonglong2 v = rp[t + 8 * decltype(U)::value];
                zr[b][decltype(U)::value].b = v.x; zi[b][decltype(U)::value].b = v.y;
            });
            cfft<8, false>(zr[b], zi[b]);
            static_for<8>([&](auto K) {
                constexpr int k = decltype(K)::value;
                if constexpr (k > 0) big_rotate(zr[b][k], zi[b][k], c_big_tw.c[t][k], c_big_tw.s[t][k]);
                rp[8 * k + t] = make_ulonglong2(zr[b][k].b, zi[b][k].b);
            });
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            ulonglong2* rp = rowp + b * 8 * RP;
            static_for<8>([&](auto U) {
                const ulonglong2 v = rp[8 * t + decltype(U)::value];
                zr[b][decltype(U)::value].b = v.x; zi[b][decltype(U)::value].b = v.y;
            });
            cfft<8, false>(zr[b], zi[b]);                   // E, O at q = t + 8r
        }
        __syncthreads();                                    // the rows are in registers: the buffer becomes the staging tile
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            float* o = sStage + ((size_t)(b * 2 * N) + t) * (8 * G) + rg0 * 32 + lane;
            static_for<8>([&](auto Rr) {
                constexpr int r = decltype(Rr)::value;
                float ar, ai, br, bi;
                split_last(zr[b][r], zi[b][r], c_big_tw.ec[t][r], c_big_tw.es[t][r], ar, ai, br, bi);
                o[(8 * r) * (8 * G)] = ar;           o[(N + 8 * r) * (8 * G)] = ai;
                o[(M + 8 * r) * (8 * G)] = br;       o[(N + M + 8 * r) * (8 * G)] = bi;
            });
        }
        if (cls == 0) {
            // row ky = 0 of every plane holds Z = FFT(X_0 + i X_{N/2}):
            // X_0[k] = (Z_k + conj Z_{-k}) / 2,  X_{N/2}[k] = (Z_k - conj Z_{-k}) / (2i)
            __syncthreads();
            for (int i = tid; i < G * (M + 1); i += T) {
                const int j = i & (G - 1), k = i / G, kp = (N - k) & (N - 1);
                constexpr int PITCH = 8 * G;
                float* a = sStage + j;
                const float fr = a[k * PITCH], fi = a[(N + k) * PITCH], gr = a[kp * PITCH], gi = a[(N + kp) * PITCH];
                const float x0r = 0.5f * (fr + gr), x0i = 0.5f * (fi - gi);
                const float xnr = 0.5f * (fi + gi), xni = 0.5f * (gr - fr);
                a[k * PITCH] = x0r;   a[(N + k) * PITCH] = x0i;
                a[kp * PITCH] = x0r;  a[(N + kp) * PITCH] = kp != k ? -x0i : x0i;
                float* b = sNy + j;
                b[k * G] = xnr;       b[(N + k) * G] = xni;
                b[kp * G] = xnr;      b[(N + kp) * G] = kp != k ? -xni : xni;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            const CUtensorMap* tm = second ? &tmS1 : &tmS0;
            const uint32_t src = fk_smem_u32(sStage);
            fk_tma_store_5d(tm, src, c0, row, cls, 0, 0);
            fk_tma_store_5d(tm, src + (uint32_t)(Gm::STAGE / 2), c0, row, cls == 0 ? 4 : 8 - cls, 0, 0);
            if (cls == 0) fk_tma_store_4d(second ? &tmNy1 : &tmNy0, fk_smem_u32(sNy), c0, row, M, 0);
            fk_bulk_commit();
        }
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Forward transform of one operand, or of two in one launch (pb may be null).
static cudaError_t launch_r2c_split(FftParams pa, const FftParams* pb_in, cudaStream_t st) {
    using Gm = SplitGeom;
    FftParams pb{};
    CUtensorMap m[4];
    memset(m, 0, sizeof(m));
    if (!fill_tiling<Gm::G>(pa)) return cudaErrorInvalidValue;
    if (!big_make_class_map<8>(&m[0], pa.spec_out, pa) || !big_make_map<128>(&m[1], pa.spec_out, pa, 1)) return cudaErrorInvalidValue;
    if (pb_in) {
        pb = *pb_in;
        if (!fill_tiling<Gm::G>(pb)) return cudaErrorInvalidValue;
        if (!big_make_class_map<8>(&m[2], pb.spec_out, pb) || !big_make_map<128>(&m[3], pb.spec_out, pb, 1)) return cudaErrorInvalidValue;
    }
    const long long items = (long long)Gm::CLASSES * ((long long)pa.num_tiles + pb.num_tiles);
    if (items > 0x3fffffffLL) return cudaErrorInvalidValue;
    int grid = 0;
    const cudaError_t e = persistent_grid(reinterpret_cast<const void*>(r2c_split_kernel), Gm::T, Gm::SMEM, items, &grid);
    if (e != cudaSuccess) return e;
    return dep_launch(false, r2c_split_kernel, dim3(grid), dim3(Gm::T), Gm::SMEM, st, m[0], m[1], m[2], m[3], pa, pb);
}

}  // namespace fc
