// Forward 2-D R2C transform at n = 64 and 128 with the rows ky split over work items.
//
// 8 planes are the least that give the frequency-major rows the 32 bytes the memory system needs, and the half
// spectrum of 8 planes does not fit shared memory at n = 128 (528 KB) and leaves room for one CTA at n = 64 (132 KB).
// So a work item is a tile of 8 planes and 16 of the rows ky: those congruent to +-r modulo n/16 for class r = 0 .. n/32 - 1.
// Every item reads all samples of its planes -- the items of a tile run next to each other, so that the samples
// come from HBM once and from the L2 after that -- but computes only its own rows: the first butterflies of a
// decimation in frequency leave 16 of the n points of a column, one 16-point transform yields the rows
// ky = (n/16) m + r, m < 16, and those above n/2 are the conjugates of the rows congruent to -r (Section 5.2:
// Hermitian symmetry).  No work is done twice, except loads, and nothing passes through a scratch area between the
// two 1-D passes.
//
// Per item, packed fp32 pairs (f32x2.cuh) of two adjacent columns, 512 threads at n = 128, 256 and two CTAs per SM at 64:
//   A. thread = (plane, pair of columns): coalesced loads straight into the first butterflies, 16-point FFT,
//      16 rows to shared memory ([plane][row][pair], 16 bytes per element);
//   B. rows of n/2 pairs: eight threads each at n = 128 (8 points, twiddle, an exchange in shared memory, 8 points), two
//      at n = 64 (one butterfly on the loads, 16 points).  The halves of a pair are then the transforms of the even
//      and the odd columns and one last butterfly between them completes the row.
//      Results form the staging tile [lo][part * n + kx][hi][plane], which overlays the rows;
//   C. one TMA store per residue lo of the rows (ky = (n/16) hi + lo): boxes of 8 planes x 8 hi x 2n.
// Row ky = 0 carries ky = n/2 as (re, im) and is taken apart in the staging tile.  The store of an
// item overlaps phase A of the next, whose samples are requested into the L2 one item ahead.
//
// What bounds it, n = 128: the samples, 4 x the planes, come from the L2 into the SMs in phase A (about 40 bytes per
// cycle and SM; 8-byte loads of that pattern reach 46 - 55), and phase B, during which nothing is loaded.
// Pairs of columns instead of pairs of planes halve the loads, and what counts as much, the loads are kept in
// program order 24 samples ahead of their use (SplitLoad): 4,096 planes of 128 x 128 209 -> 145 us, 12,288 of
// 118 x 118 602 -> 440, 4,096 of 97 x 101 (4-byte loads) 201 -> 145, 12 planes of 128 x 128 33 -> 18 us.  16 and
// 32 samples ahead: 150 and 145 us, 434 and 457.  Tried and not kept: the compiler's own order of the loads (181 us,
// 435 for 97 x 101); teams of 8 warps for A and B with half a tile between them (200 us: fewer loads in flight); four
// planes per item, stored in rows of 16 bytes (390 us); a tile's four items one after the other in one CTA (280 us).
// n = 64: 8,192 planes of 64 x 64 78 -> 58 us (4.7 TB/s; its stores alone take 31), of 57 x 57 78 -> 59, 32 planes
// 14.7 -> 8.7, against tiles of 4 + 4 planes in one CTA per SM with whole columns and rows per thread.  Three CTAs of 80
// registers spill (84 - 90 us); teams for A and B that share a tile through shared memory, samples by bulk copies: 73 - 81.
#pragma once

#include "fft_big.cuh"

namespace fc {

template <int N_>
struct SplitGeom {
    static constexpr int N = N_, M = N / 2, NC = M + 1, G = 8;
    static constexpr int CP = N / 2;                     // pairs of columns in a row
    static constexpr int T = G * CP;                     // threads
    static constexpr int L = N / 16, CLASSES = L / 2;    // rows ky = L hi + lo, hi < 8; class r: lo = r and L - r (0 and L / 2)
    static constexpr int MINB = N == 64 ? 2 : 1;
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
// before its use and a thread has a few in flight.  The output is written before the address is read
// (early-clobber constraint).
// LOW (windows): the rows below `low` do not exist either.
template <bool PAIR, bool LOW>
struct SplitLoad {
    const float* s0;
    int pitch;                      // bytes from row to row
    int rows, rows2;                // rows that exist in the first and in the second column
    int low;
    template <int r>
    __device__ __forceinline__ F2 get() const {
        const char* q = reinterpret_cast<const char*>(s0) + (long long)pitch * r;
        const unsigned at = LOW ? (unsigned)(r - low) : (unsigned)r;
        if constexpr (PAIR) {
            F2 v;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.u32 p, %2, %3;\n\tmov.b64 %0, 0;\n\t@p ld.global.nc.b64 %0, [%1];\n\t}"
                         : "=&l"(v.b) : "l"(q), "r"(rows), "r"(at));
            return v;
        } else {
            float u, v;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.u32 p, %2, %3;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.b32 %0, [%1];\n\t}"
                         : "=&f"(u) : "l"(q), "r"(rows), "r"(at));
            asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.u32 p, %2, %3;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.b32 %0, [%1+4];\n\t}"
                         : "=&f"(v) : "l"(q), "r"(rows2), "r"(at));
            return f2_pack(u, v);
        }
    }
};

// Phase A of class R: first butterflies of a column, twiddles, 16-point FFT; put(row, re, im) with row = 8 *
// (second residue) + hi; release() comes before the first put.  The samples of the next AHEAD butterflies are on
// their way.
template <int N, int R, class Load, class Release>
__device__ __forceinline__ void split_column(const Load& x, ulonglong2* dst, Release&& release) {
    constexpr int V = N / 16, AHEAD = 24 / V;
    auto put = [&](auto K, F2 re, F2 im) __attribute__((always_inline)) { dst[decltype(K)::value * SplitGeom<N>::RP] = make_ulonglong2(re.b, im.b); };
    F2 ring[AHEAD][V];
    auto fetch = [&](auto J) __attribute__((always_inline)) {
        constexpr int j = decltype(J)::value;
        static_for<V>([&](auto W) __attribute__((always_inline)) { ring[j % AHEAD][decltype(W)::value] = x.template get<j + 16 * decltype(W)::value>(); });
    };
    static_for<AHEAD>(fetch);
    F2 ar[R == 0 ? 32 : 16], ai[16];
    static_for<16>([&](auto J) __attribute__((always_inline)) {
        constexpr int j = decltype(J)::value;
        const F2 (&v)[V] = ring[j % AHEAD];
        if constexpr (R == 0) {
            if constexpr (N == 64) {
                ar[j] = v[0] + v[2];
                ar[j + 16] = v[1] + v[3];
            } else {
                ar[j] = (v[0] + v[4]) + (v[2] + v[6]);
                ar[j + 16] = (v[1] + v[5]) + (v[3] + v[7]);
            }
        } else {
            F2 re, im;                                      // sum_v x_v w_V^{R v}
            if constexpr (N == 64) {
                re = v[0] - v[2];
                im = v[3] - v[1];
            } else if constexpr (R == 2) {
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
                constexpr float c = Tw<N, R * j>::c, sn = Tw<N, R * j>::s;
                ar[j] = vfma(sn, im, vmul(c, re));
                ai[j] = vfma(-sn, re, vmul(c, im));
            }
        }
        if constexpr (j + AHEAD < 16) fetch(std::integral_constant<int, j + AHEAD>{});
    });
    if constexpr (R == 0) {
        F2 Xr[17], Xi[17];
        rfft<32>(ar, Xr, Xi);                               // X[k] = row ky = k N / 32
        release();
        put(std::integral_constant<int, 0>{}, Xr[0], Xr[16]);
        static_for<15>([&](auto K) __attribute__((always_inline)) {
            constexpr int k = decltype(K)::value + 1;
            put(std::integral_constant<int, (k & 1) * 8 + k / 2>{}, Xr[k], Xi[k]);
        });
    } else {
        cfft<16, false>(ar, ai);                            // row ky = L m + R
        release();
        static_for<16>([&](auto Mm) __attribute__((always_inline)) {
            constexpr int m = decltype(Mm)::value;
            if constexpr (m < 8) put(std::integral_constant<int, m>{}, ar[m], ai[m]);
            else put(std::integral_constant<int, 8 + 15 - m>{}, ar[m], -ai[m]);
        });
    }
}
template <int N, class Load, class Release>
__device__ __forceinline__ void split_class(int cls, const Load& x, ulonglong2* dst, Release&& release) {
    if (cls == 0)                 split_column<N, 0>(x, dst, release);
    else if (N == 64 || cls == 1) split_column<N, 1>(x, dst, release);
    else if constexpr (N == 128) {
        if (cls == 2) split_column<N, 2>(x, dst, release);
        else          split_column<N, 3>(x, dst, release);
    }
}

// Requests an item's share of its tile's samples into the L2.
template <int N>
__device__ __forceinline__ void split_prefetch(int item, int items0, const FftParams& p0, const FftParams& p1) {
    using Gm = SplitGeom<N>;
    const bool second = item >= items0;
    const FftParams& p = second ? p1 : p0;
    if (p.win) return;              // the windows of a plane share its samples, which are in the L2 already for the most part
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

template <int N, bool WIN>
__global__ void __launch_bounds__(SplitGeom<N>::T, SplitGeom<N>::MINB)
r2c_split_kernel(const __grid_constant__ CUtensorMap tmS0, const __grid_constant__ CUtensorMap tmNy0,
                 const __grid_constant__ CUtensorMap tmS1, const __grid_constant__ CUtensorMap tmNy1,
                 const __grid_constant__ FftParams p0, const __grid_constant__ FftParams p1, const int in_step) {
    using Gm = SplitGeom<N>;
    constexpr int M = Gm::M, G = Gm::G, CP = Gm::CP, RP = Gm::RP, PP = Gm::PP, T = Gm::T;
    extern __shared__ __align__(128) unsigned char fc_smem[];
    ulonglong2* sMid = reinterpret_cast<ulonglong2*>(fc_smem);
    float* sStage = reinterpret_cast<float*>(fc_smem);
    float* sNy = reinterpret_cast<float*>(fc_smem + Gm::BUF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gA = tid / CP, cA = 2 * (tid - gA * CP);      // A: plane, first of two columns
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
        if (tid == 32 && item + (int)gridDim.x < items) split_prefetch<N>(item + gridDim.x, items0, p0, p1);

        if (N == 64 && in_step) {                   // the CTAs of a cluster begin each item together
            asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        }

        // ---- A: columns; a pair of columns past the plane reads no sample and writes zeros ----
        {
            // a window of a larger plane: its origin (y0, x0) may lie outside, samples there read as zero
            int pitch = w, size = h * w, s = row, y0 = 0, x0 = 0, low = 0, high = h, left = 0, right = w;
            if (WIN && p.win) {
                const int nt = p.nty * p.ntx;
                s = row / nt;
                const int t = row - s * nt, ty = t / p.ntx, tx = t - ty * p.ntx;
                pitch = p.W; size = p.H * p.W;
                y0 = ty * p.step_y + p.oy; x0 = tx * p.step_x + p.ox;
                low = max(0, -y0); high = min(h, p.H - y0);
                left = max(0, -x0); right = min(w, p.W - x0);
            }
            const float* planes = p.real_in + ((size_t)s * p.C + c0) * (size_t)size;
            const bool plane = gA < p.C - c0 && high > low;
            const bool live = plane && cA >= left && cA < right, live2 = plane && cA + 1 >= left && cA + 1 < right;
            const float* s0 = planes + (plane ? gA * size + y0 * pitch + x0 + cA : 0);
            const int rows = live ? high - low : 0, rows2 = live2 ? high - low : 0;
            ulonglong2* dst = sMid + gA * PP + (cA >> 1);
            auto release = [&]() __attribute__((always_inline)) {  // the previous item's store has read the buffer
                if (tid == 0) fk_bulk_wait_read();
                __syncthreads();
            };
            // pairs that start at multiples of 8 bytes are inside or outside as a whole
            if (((w | pitch | x0 | (int)(reinterpret_cast<uintptr_t>(planes) >> 2)) & 1) == 0)
                split_class<N>(cls, SplitLoad<true, WIN>{s0, 4 * pitch, rows, rows2, low}, dst, release);
            else
                split_class<N>(cls, SplitLoad<false, WIN>{s0, 4 * pitch, rows, rows2, low}, dst, release);
        }
        __syncthreads();

        // ---- B: rows; lanes run over the planes, then over four adjacent rows hi ----
        ulonglong2* rowp = sMid + (lane & 7) * PP + (lane >> 3) * RP;
        if constexpr (N == 128) {
            // Eight threads per row of 64 pairs: 8 points, twiddle, an exchange in place (the slots a thread writes are
            // the slots it has read), 8 points; a warp takes two groups of four rows.
            const int t = warp & 7, rg0 = warp >> 3;
            rowp += rg0 * 4 * RP;
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
                cfft<8, false>(zr[b], zi[b]);               // E, O at q = t + 8r
            }
            __syncthreads();                                // the rows are in registers: the buffer becomes the staging tile
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
        } else {
            // Two threads per row of 32 pairs: one decimation-in-frequency step on the loads, 16 points.
            const int rg = warp >> 1;
            const ulonglong2* rp = rowp + rg * 4 * RP;
            float* o = sStage + (size_t)((rg >> 1) * 2 * N) * (8 * G) + (rg & 1) * 32 + lane;
            F2 zr[16], zi[16];
            auto load = [&](auto Q) __attribute__((always_inline)) {
                constexpr int q = decltype(Q)::value;
                static_for<16>([&](auto J) __attribute__((always_inline)) {
                    constexpr int j = decltype(J)::value;
                    const ulonglong2 a = rp[j], b = rp[j + 16];
                    if constexpr (q == 0) {
                        zr[j] = F2{a.x} + F2{b.x}; zi[j] = F2{a.y} + F2{b.y};
                    } else {
                        const F2 dr = F2{a.x} - F2{b.x}, di = F2{a.y} - F2{b.y};
                        if constexpr (j == 0) {
                            zr[j] = dr; zi[j] = di;
                        } else if constexpr (j == 8) {
                            zr[j] = di; zi[j] = -dr;
                        } else {
                            constexpr float c = Tw<32, j>::c, sn = Tw<32, j>::s;
                            zr[j] = vfma(sn, di, vmul(c, dr));
                            zi[j] = vfma(-sn, dr, vmul(c, di));
                        }
                    }
                });
            };
            auto store = [&](auto Q) __attribute__((always_inline)) {
                static_for<16>([&](auto K) __attribute__((always_inline)) {
                    constexpr int k = decltype(K)::value, kx = 2 * k + decltype(Q)::value;
                    float ar, ai, br, bi;
                    split_last(zr[k], zi[k], Tw<64, kx>::c, Tw<64, kx>::s, ar, ai, br, bi);
                    o[kx * (8 * G)] = ar;        o[(N + kx) * (8 * G)] = ai;
                    o[(M + kx) * (8 * G)] = br;  o[(N + M + kx) * (8 * G)] = bi;
                });
            };
            constexpr std::integral_constant<int, 0> even{};
            constexpr std::integral_constant<int, 1> odd{};
            if ((warp & 1) == 0) load(even);
            else                 load(odd);
            __syncthreads();                                // the rows are in registers: the buffer becomes the staging tile
            cfft<16, false>(zr, zi);                        // E, O at 2k + q
            if ((warp & 1) == 0) store(even);
            else                 store(odd);
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
            fk_tma_store_5d(tm, src + (uint32_t)(Gm::STAGE / 2), c0, row, cls == 0 ? Gm::L / 2 : Gm::L - cls, 0, 0);
            if (cls == 0) fk_tma_store_4d(second ? &tmNy1 : &tmNy0, fk_smem_u32(sNy), c0, row, M, 0);
            fk_bulk_commit();
        }
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// At n = 64 (without windows) the plain kernel, whose tiles are 4 planes, is the better one where no tile is more than half full: 300 rows of
// 4 planes 20.9 -> 18.8 us (25 x 25), of 6 planes 18.8 against 26.9.
// Spectra whose rows are no whole sectors (ld = 4 mod 8), from about the size of the L2 on.  Every other row starts in the
// middle of a sector, so a tile shares its sectors with the tiles before and after it, and parts of a sector that SMs
// of different dies write cost more than everything else.
// * The plain kernel's tiles share sectors in pairs (2j, 2j + 1), which adjacent CTAs write, if the tiles of every matrix and
//   those launched before it come in even numbers: SECTORS_PLAIN.  Plain / this kernel in single CTAs (passes, planes of 50 x 50):
//   1,332 rows of 9 planes 389 / 570 us, 1,000 of 12 298 / 371, 1,332 of 18 496 / 700, 352 of 34 209 / 236, 240 of 50 187 / 200, 134 of
//   178 323 / 406.  With odd numbers the plain kernel is the one that loses (353 of 34 288 / 230, 135 of 178 608 / 418; 160 rows of
//   90 filters behind 115 tiles 351 / 252, behind 92 210 / 249), and where rows of planes start off a 16-byte boundary it waits for
//   the odd samples of every tile (298 rows of 134 planes of 49 x 49 759 / 298).
// * Otherwise SECTORS_NEAR: clusters of eight CTAs, which share a die, take four adjacent tiles and begin their items together.  Single
//   CTAs / clusters (transform alone): 3,333 rows of 12 planes of 62 x 62 1064 / 586 us, 1,176 of 34 737 / 528, 800 of 50 planes
//   of 49 x 49 612 / 474; clusters of four 769, 647, 565.
// Smaller spectra are better off in single CTAs (160 rows of 50 89 / 93), longer rows turn over later (666 of 12 134 / 119 at
// 135 MB; plain / single CTAs 160 of 50 147 / 144 at 135 MB, 52 of 201 225 / 203 at 176).
enum { SECTORS_WHOLE = 0, SECTORS_NEAR = 1, SECTORS_PLAIN = 2 };
static inline int split_sectors(const FftParams& pa, const FftParams* pb) {
    const FftParams* ops[2] = {&pa, pb};
    double bytes[2] = {0, 0}, partial = 0;
    int widest = 0;
    long long before = 0;
    bool pairs = true;
    for (int i = 0; i < (pb ? 2 : 1); ++i) bytes[i] = 8.0 * 64 * 33 * (double)ops[i]->R * ops[i]->C;
    const double total = bytes[0] + bytes[1];
    for (int i = 0; i < (pb ? 2 : 1); ++i) {
        const FftParams& p = *ops[i];
        const long long tiles = (long long)p.R * ((p.C + 3) / 4);
        if (10 * bytes[i] > total) {
            const bool rows_aligned = (reinterpret_cast<uintptr_t>(p.real_in) & 15) == 0 && (long long)p.C * p.h * p.w % 4 == 0;
            pairs = pairs && rows_aligned && before % 2 == 0 && tiles % 2 == 0;
            if (p.ld % 8 != 0) {
                partial += bytes[i];
                if (p.C > widest) widest = p.C;
            }
        }
        before += tiles;
    }
    if (3 * partial <= total || total <= 120e6 + 450e3 * widest) return SECTORS_WHOLE;
    return pairs ? SECTORS_PLAIN : SECTORS_NEAR;
}
static inline bool split_pays(int n, const FftParams& pa, const FftParams* pb) {
    if (n != 64) return false;
    if (pa.win || (pb && pb->win)) return true;
    if (split_sectors(pa, pb) == SECTORS_PLAIN) return false;
    return 2 * pa.C > SplitGeom<64>::G || (pb && 2 * pb->C > SplitGeom<64>::G);
}

// Forward transform of one operand, or of two in one launch (pb may be null).
template <int N>
static cudaError_t launch_r2c_split(FftParams pa, const FftParams* pb_in, cudaStream_t st) {
    using Gm = SplitGeom<N>;
    FftParams pb{};
    CUtensorMap m[4];
    memset(m, 0, sizeof(m));
    if (!fill_tiling<Gm::G>(pa)) return cudaErrorInvalidValue;
    if (!big_make_class_map<N, Gm::L>(&m[0], pa.spec_out, pa) || !big_make_map<N>(&m[1], pa.spec_out, pa, 1)) return cudaErrorInvalidValue;
    if (pb_in) {
        pb = *pb_in;
        if (!fill_tiling<Gm::G>(pb)) return cudaErrorInvalidValue;
        if (!big_make_class_map<N, Gm::L>(&m[2], pb.spec_out, pb) || !big_make_map<N>(&m[3], pb.spec_out, pb, 1)) return cudaErrorInvalidValue;
    }
    const long long items = (long long)Gm::CLASSES * ((long long)pa.num_tiles + pb.num_tiles);
    if (items > 0x3fffffffLL) return cudaErrorInvalidValue;
    int grid = 0;
    // the windowed variant is an instantiation of its own, so that the plain one carries none of its tests
    auto kern = N == 64 && (pa.win || pb.win) ? r2c_split_kernel<N, N == 64> : r2c_split_kernel<N, false>;
    if (N != 64 && (pa.win || pb.win)) return cudaErrorInvalidValue;
    const cudaError_t e = persistent_grid(reinterpret_cast<const void*>(kern), Gm::T, Gm::SMEM, items, &grid);
    if (e != cudaSuccess) return e;
    // n = 64: the CTAs of a launch drift apart, and in a long one the second of a tile's two items no longer finds the samples in
    // the L2 (40,200 planes of 62 x 62: 764 MB read from memory instead of 618).  From about 400 MB of spectra on the two
    // are a cluster whose CTAs begin each item together: 40,000 planes of 62 x 62 373 -> 311 us, 49 x 49 300 -> 278; 24,000
    // 172 / 173 and 170 / 166, 8,000 60 / 64.
    int cluster = 1;
    if (N == 64 && !pa.win && !pb.win && items > grid)
        cluster = split_sectors(pa, pb_in ? &pb : nullptr) == SECTORS_NEAR ? 8 : (items >= 8000 ? 2 : 1);
    if (cluster > 1) {
        const int fit = cluster * resident_clusters(reinterpret_cast<const void*>(kern), Gm::T, Gm::SMEM, cluster);
        const int together = (fit < grid ? fit : grid) / cluster * cluster;
        if (together > 0) grid = together;
        else cluster = 1;           // (a part of a GPU that holds no such cluster)
    }
    // One round of items: no L1 is of use, and the filters' transform, launched early behind this one, finds the SMs divided as it
    // needs them (S9 f58 f'6 36 x 44 k9 43.9 -> 37.7 us, S17 f34 f'6 50 x 57 k13 38.1 -> 34.3).
    return dep_launch({false, cluster, items <= grid ? 100 : -1}, kern, dim3(grid), dim3(Gm::T), Gm::SMEM, st, m[0], m[1], m[2], m[3], pa, pb, cluster > 1 ? 1 : 0);
}

}  // namespace fc
