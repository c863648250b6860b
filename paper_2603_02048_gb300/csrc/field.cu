// Refractive-index volume from density (Sec. 3.3.1 of arXiv 2603.02048):
// Gladstone-Dale dn = n - 1 = K rho (Eq. 12) and g = grad n = K grad rho
// (Eq. 13) by finite differences: central inside, one-sided on the first and
// last voxel of each axis. Packed per voxel as {dn, gx, gy, gz}:
//   FP32: float4, 16 B/voxel (one pass: read rho, write the volume);
//   FP16: four halves, 8 B/voxel, dn / s_n and g / s_g with per-volume scales
//         s = the smallest power of two with max|.| / s <= 16384 (pass 1
//         reduces the maxima, pass 2 recomputes the differences and quantises
//         with exact multiplications by 1 / s; rho is read twice, nothing else
//         stored).
// The packed volume is written in the volume's layout (ZPAIR with its halo of
// edge copies for volumes the march reads, LINEAR for the allocation-free
// build's caller buffer). The ZPAIR FP32 stores are marked evict-first: the
// volume outgrows L2 anyway, and this keeps the density, which the kernel is
// still reading, resident in L2 instead.
// ZPAIR builds also leave the volume's free-corner mask (the march skips the
// eight loads of a sample whose corners are all zero): the store pass records
// which voxels are nonzero (ballots, no atomics), and free_mask_kernel turns
// those into one bit per element, set when the eight voxels of the cell it is
// the first corner of are all zero.
#include "hh_internal.h"

namespace hh {
namespace {

// Scale of a channel group from the bit pattern of its maximum |value| m:
// the smallest power of two s with m / s <= HH_FP16_CODE_MAX (the largest code
// lies in (HH_FP16_CODE_MAX / 2, HH_FP16_CODE_MAX]); 1 for an all-zero group.
// A power of two makes value / s exact, a multiplication by 1 / s.
__device__ __forceinline__ float scale_of(unsigned bits) {
    const float m = __uint_as_float(bits);
    if (!(m > 0.0f)) return 1.0f;
    unsigned b = __float_as_uint(m * (1.0f / HH_FP16_CODE_MAX));  // exact: a power of two
    if (b < 0x00800000u) return __uint_as_float(0x00800000u);    // below FLT_MIN: FLT_MIN
    if (b & 0x007FFFFFu) b = (b & 0xFF800000u) + 0x00800000u;     // round up to a power of two
    return __uint_as_float(b);
}

// 32 bytes to an aligned address in one store, evict-first in L2.
__device__ __forceinline__ void store32(void* p, uint4 a, uint4 b) {
    asm volatile("st.global.L2::evict_first.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z),
                 "r"(b.w)
                 : "memory");
}

// One voxel's {dn, gx, gy, gz}, as stored: FP32, or halves of value / s (the
// nearest half; the products are exact as s is a power of two).
struct Voxel {
    float dn, gx, gy, gz;
};
__device__ __forceinline__ uint4 pack32(const Voxel& v) {
    return make_uint4(__float_as_uint(v.dn), __float_as_uint(v.gx), __float_as_uint(v.gy),
                      __float_as_uint(v.gz));
}
__device__ __forceinline__ uint2 pack16(const Voxel& v, float rs_n, float rs_g) {
    const __half2 lo = __floats2half2_rn(v.dn * rs_n, v.gx * rs_g);
    const __half2 hi = __floats2half2_rn(v.gy * rs_g, v.gz * rs_g);
    return make_uint2(*reinterpret_cast<const unsigned*>(&lo),
                      *reinterpret_cast<const unsigned*>(&hi));
}

// A thread owns grid column i of a pair of padded rows J = 2 jj, 2 jj + 1 and
// walks `run` pairs of padded slices K = 2 kk, 2 kk + 1: four voxels an iteration.
// A row's two are consecutive in the ZPAIR layout, so a warp stores 1 KiB (FP32)
// or 512 B (FP16) in one piece per row. K rho of the two rows stays in registers
// from slice to slice and each row is the other's y neighbour: a slice of the
// pair costs eight loads (two centres, two outer rows, four x neighbours),
// where a thread per column needs ten. H = 1 (ZPAIR): padded coordinates are
// grid coordinates + 1 and the halo repeats the nearest grid voxel (in x, the
// first and last column store twice); H = 0 (LINEAR, and
// the max pass, which stores nothing): they are the grid's. A
// one-sided difference is the central one with the missing neighbour replaced
// by the voxel itself and the factor 1 instead of 1/2. Threads of the padding
// compute a clamped voxel, which does not change a maximum and is not stored.
// What bounds it: DRAM and its latency. 256^3 FP32: 58 us for the 285 MB it
// moves (74 with a thread per column and 16-byte stores), FP16: maxima 31, store
// 46 us (38 and 66). 5 resident blocks (48 registers) against 4 take 4 % off a
// 512^3 FP16 build.
constexpr int field_blocks(int mode) { return mode == 1 ? 4 : 5; }

template <int MODE, int H>  // 0: FP32 store, 1: FP16 max pass, 2: FP16 store
__global__ void __launch_bounds__(256, field_blocks(MODE))
    field_kernel(const float* __restrict__ rho, int nx, int ny, int nz, float K, int run,
                 unsigned row, unsigned pair, void* __restrict__ out,
                 unsigned* __restrict__ nz_bits, unsigned* __restrict__ sparse,
                 unsigned* __restrict__ max_bits, float* __restrict__ scales) {
    await_previous();
    rho = after_wait(rho);
    max_bits = after_wait(max_bits);
    release_next();
    // warps go along x, then to the next pair of rows
    const unsigned lane = threadIdx.x & 31, nz_words = (static_cast<unsigned>(nx) + 31u) / 32u;
    const unsigned warp = blockIdx.x * 8 + (threadIdx.x >> 5);
    const unsigned jj = warp / nz_words, word = warp - jj * nz_words;
    const unsigned I = word * 32 + lane;  // grid column
    const int row_pairs = (ny + 2 * H + 1) / 2, slice_pairs = (nz + 2 * H + 1) / 2;
    const int kk0 = blockIdx.y * run, kk1 = min(kk0 + run, slice_pairs);
    const bool valid = static_cast<int>(jj) < row_pairs && static_cast<int>(I) < nx;
    float s_n = 1.0f, s_g = 1.0f;
    if (MODE == 2) {
        s_n = scale_of(max_bits[0]);
        s_g = scale_of(max_bits[1]);
    }
    const float rs_n = 1.0f / s_n, rs_g = 1.0f / s_g;  // exact: powers of two
    if (MODE != 1 && threadIdx.x == 0 && blockIdx.x + blockIdx.y == 0) {
        scales[0] = s_n;
        scales[1] = s_g;
        if (H) *sparse = 0;  // free_mask_kernel, the next launch, may set it
    }
    // this warp's row pair of nonzero words: lane l < 4 owns row l & 1, slice l >> 1
    unsigned* const nz_at =
        H ? nz_bits + (static_cast<size_t>(2 * kk0 + (lane >> 1)) * (2 * row_pairs) + 2 * jj +
                       (lane & 1)) * nz_words + word
          : nullptr;
    const size_t nz_step = static_cast<size_t>(4 * row_pairs) * nz_words;
    const int i = min(static_cast<int>(I), nx - 1);
    const int J0 = min(2 * static_cast<int>(jj), 2 * row_pairs - 2) - H, J1 = J0 + 1;
    const int j0 = min(max(J0, 0), ny - 1), j1 = min(J1, ny - 1);
    const size_t sz = static_cast<size_t>(nx) * ny;
    const float* r0 = rho + static_cast<size_t>(j0) * nx + i;
    const float* r1 = rho + static_cast<size_t>(j1) * nx + i;
    const float* ra = rho + static_cast<size_t>(max(j0 - 1, 0)) * nx + i;
    const float* rd = rho + static_cast<size_t>(min(j1 + 1, ny - 1)) * nx + i;
    const int xl = i > 0 ? -1 : 0, xh = i < nx - 1 ? 1 : 0;
    const float fx = xl && xh ? 0.5f : 1.0f;
    const float fy0 = j0 > 0 && j0 < ny - 1 ? 0.5f : 1.0f;
    const float fy1 = j1 > 0 && j1 < ny - 1 ? 0.5f : 1.0f;
    const bool first_row = J0 < 0, last_row = J1 >= ny;
    // dn = K rho, rounded by itself (an FMA with the difference that uses it would
    // give a gradient that is not the stored dn's)
    auto dn_of = [K](const float* p) { return __fmul_rn(K, __ldg(p)); };
    auto at = [&](const float* p, int k) { return dn_of(p + static_cast<size_t>(k) * sz); };
    // rows 0 and 1: p at slice s0 - 1, a at s0, b at s1, n at s1 + 1
    float p0, p1, a0, a1;
    {
        const int k = max(2 * kk0 - H, 0);
        p0 = at(r0, max(k - 1, 0));
        p1 = at(r1, max(k - 1, 0));
        a0 = at(r0, min(k, nz - 1));
        a1 = at(r1, min(k, nz - 1));
    }
    float mn = 0.0f, mg = 0.0f;
    // the max pass scales the largest x and y differences once, at the end (max and
    // the multiplication by 1/2 commute), and walks two pairs at once: 256^3 FP16
    // build 183.7 against 181.5 us, 512^3 1564 against 1557
    float mx = 0.0f, my0 = 0.0f, my1 = 0.0f;
    const float kx = MODE == 1 ? 1.0f : fx;
    const float ky0 = MODE == 1 ? 1.0f : fy0, ky1 = MODE == 1 ? 1.0f : fy1;
#pragma unroll(MODE == 1 ? 2 : 1)
    for (int kk = kk0; kk < kk1; ++kk) {
        const int K0 = 2 * kk - H, K1 = K0 + 1;  // grid slices of the pair
        const int s0 = min(max(K0, 0), nz - 1), s1 = min(K1, nz - 1), sn = min(K1 + 1, nz - 1);
        if (K0 >= nz) {  // the halo slice alone: again slice nz - 1, whose neighbour is nz - 2
            p0 = at(r0, nz - 2);
            p1 = at(r1, nz - 2);
        }
        const float b0 = at(r0, s1), b1 = at(r1, s1);
        const float n0 = at(r0, sn), n1 = at(r1, sn);
        const float fz0 = s0 > 0 && s0 < nz - 1 ? 0.5f : 1.0f;
        const float fz1 = s1 > 0 && s1 < nz - 1 ? 0.5f : 1.0f;
        Voxel v00, v10, v01, v11;  // [row][slice]
        v00.dn = a0;
        v10.dn = a1;
        v01.dn = b0;
        v11.dn = b1;
        // K0 < 0: the halo slice below slice 0, both of the pair are slice 0;
        // K1 >= nz: both are slice nz - 1
        v00.gz = ((K0 < 0 ? n0 : b0) - p0) * fz0;
        v10.gz = ((K0 < 0 ? n1 : b1) - p1) * fz0;
        v01.gz = (n0 - (K1 >= nz ? p0 : a0)) * fz1;
        v11.gz = (n1 - (K1 >= nz ? p1 : a1)) * fz1;
        {
            const size_t z = static_cast<size_t>(s0) * sz;
            const float oa = dn_of(ra + z), od = dn_of(rd + z);
            v00.gx = (dn_of(r0 + z + xh) - dn_of(r0 + z + xl)) * kx;
            v10.gx = (dn_of(r1 + z + xh) - dn_of(r1 + z + xl)) * kx;
            v00.gy = ((first_row ? od : a1) - oa) * ky0;
            v10.gy = (od - (last_row ? oa : a0)) * ky1;
        }
        {
            const size_t z = static_cast<size_t>(s1) * sz;
            const float oa = dn_of(ra + z), od = dn_of(rd + z);
            v01.gx = (dn_of(r0 + z + xh) - dn_of(r0 + z + xl)) * kx;
            v11.gx = (dn_of(r1 + z + xh) - dn_of(r1 + z + xl)) * kx;
            v01.gy = ((first_row ? od : b1) - oa) * ky0;
            v11.gy = (od - (last_row ? oa : b0)) * ky1;
        }
        if (MODE == 1) {
            auto peak = [](float m, float a, float b) {
                return fmaxf(m, fmaxf(fabsf(a), fabsf(b)));
            };
            mn = peak(peak(mn, a0, a1), b0, b1);
            mx = peak(peak(mx, v00.gx, v10.gx), v01.gx, v11.gx);
            my0 = peak(my0, v00.gy, v01.gy);
            my1 = peak(my1, v10.gy, v11.gy);
            mg = peak(peak(mg, v00.gz, v10.gz), v01.gz, v11.gz);
        } else if (H == 0) {
            if (valid) {
                const size_t o = (static_cast<size_t>(K0) * ny + J0) * nx + i;
                uint4* to = static_cast<uint4*>(out) + o;
                __stcs(to, pack32(v00));
                if (J1 < ny) __stcs(to + nx, pack32(v10));
                if (K1 < nz) __stcs(to + sz, pack32(v01));
                if (J1 < ny && K1 < nz) __stcs(to + sz + nx, pack32(v11));
            }
        } else {
            const unsigned J = 2 * jj;
            const bool valid1 = valid && static_cast<int>(J) + 1 < ny + 2;
            // element of (I = i + 1, J, 2 kk); the halo columns are the first
            // and the last thread's second stores
            const size_t o = static_cast<size_t>(kk) * pair + J * row + 2 * (I + 1);
            bool z00, z10, z01, z11;  // holds only +-0
            if (MODE == 0) {
                const uint4 w00 = pack32(v00), w01 = pack32(v01);
                const uint4 w10 = pack32(v10), w11 = pack32(v11);
                auto zero = [](uint4 w) { return ((w.x | w.y | w.z | w.w) & 0x7FFFFFFFu) == 0u; };
                z00 = zero(w00);
                z01 = zero(w01);
                z10 = zero(w10);
                z11 = zero(w11);
                uint4* to = static_cast<uint4*>(out) + o;
                auto put = [&](int d) {
                    if (valid) store32(to + d, w00, w01);
                    if (valid1) store32(to + static_cast<int>(row) + d, w10, w11);
                };
                put(0);
                if (xl == 0) put(-2);
                if (xh == 0) put(2);
            } else {
                const uint2 w00 = pack16(v00, rs_n, rs_g), w01 = pack16(v01, rs_n, rs_g);
                const uint2 w10 = pack16(v10, rs_n, rs_g), w11 = pack16(v11, rs_n, rs_g);
                auto zero = [](uint2 w) { return ((w.x | w.y) & 0x7FFF7FFFu) == 0u; };
                z00 = zero(w00);
                z01 = zero(w01);
                z10 = zero(w10);
                z11 = zero(w11);
                uint2* to = static_cast<uint2*>(out) + o;
                auto put = [&](int d) {
                    if (valid)
                        __stcs(reinterpret_cast<uint4*>(to + d),
                               make_uint4(w00.x, w00.y, w01.x, w01.y));
                    if (valid1)
                        __stcs(reinterpret_cast<uint4*>(to + static_cast<int>(row) + d),
                               make_uint4(w10.x, w10.y, w11.x, w11.y));
                };
                put(0);
                if (xl == 0) put(-2);
                if (xh == 0) put(2);
            }
            // nonzero bits, a word per row and slice
            const unsigned n00 = __ballot_sync(0xffffffffu, valid && !z00);
            const unsigned n10 = __ballot_sync(0xffffffffu, valid1 && !z10);
            const unsigned n01 = __ballot_sync(0xffffffffu, valid && !z01);
            const unsigned n11 = __ballot_sync(0xffffffffu, valid1 && !z11);
            if (lane < 4 && static_cast<int>(jj) < row_pairs)
                nz_at[(kk - kk0) * nz_step] =
                    lane & 2 ? (lane & 1 ? n11 : n01) : (lane & 1 ? n10 : n00);
        }
        p0 = b0;
        p1 = b1;
        a0 = n0;
        a1 = n1;
    }
    if (MODE == 1) {  // block maximum, then one atomic per block
        mg = fmaxf(fmaxf(mg, mx * fx), fmaxf(my0 * fy0, my1 * fy1));
        for (int d = 16; d > 0; d >>= 1) {
            mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, d));
            mg = fmaxf(mg, __shfl_xor_sync(0xffffffffu, mg, d));
        }
        __shared__ float sn[8], sg[8];
        if ((threadIdx.x & 31) == 0) {
            sn[threadIdx.x >> 5] = mn;
            sg[threadIdx.x >> 5] = mg;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) {
                mn = fmaxf(mn, sn[w]);
                mg = fmaxf(mg, sg[w]);
            }
            atomicMax(max_bits + 0, __float_as_uint(mn));
            atomicMax(max_bits + 1, __float_as_uint(mg));
        }
    }
}

// A warp's stretch of the mask (1024 elements) with at least this many free
// ones makes the volume sparse: marches then ask the mask, RK4 at every sample,
// Eq. 16 after a sample with dn = 0. In a volume without empty space the question
// costs Eq. 16 little and RK4 a load's latency a sample, for nothing (720p views of
// a 192x160x224 turbulence volume, asked and not: Eq. 16 at theta 1e-5 178 and 175
// us, RK4 595 and 558, RK4 at half a voxel 1205 and 1070; a 64^3 128x128 RK4 view
// 203 and 171). So the line is low, one stretch an eighth of which is free, and a
// volume with a hole of that size only is marched as a sparse one.
constexpr unsigned kSparseFree = 128;

// The free-corner mask from the store pass's nonzero bits, a word (32
// consecutive elements: 16 columns of a row of a pair of slices, or the end of
// one row and the start of the next) per thread; blockIdx.y is the pair of
// slices the word starts in. Column I of row J, slice K is free when none of
// columns I, I + 1 of rows J, J + 1 of slices K, K + 1 holds a nonzero value; the
// halo columns hold what the first and the last grid column do. What it says of
// cells beyond the last sampled column, row and slice is not read.
// 256^3 (537,000 words): 13 us, latency and issue; with a window per row, slice
// and neighbour and the words' places from integer divisions it took 17.
__global__ void __launch_bounds__(256)
    free_mask_kernel(const unsigned* __restrict__ nz, unsigned nz_words, int nx, int ny,
                     unsigned pairs, unsigned row, unsigned pair, float per_row,
                     unsigned* __restrict__ fr, unsigned* __restrict__ sparse) {
    await_previous();
    nz = after_wait(nz);
    const unsigned rows = (static_cast<unsigned>(ny) + 3u) / 2u * 2u;
    const size_t slice = static_cast<size_t>(rows) * nz_words;  // words
    unsigned kk = blockIdx.y;
    const unsigned g = (kk * pair + 31u) / 32u + blockIdx.x * blockDim.x + threadIdx.x;
    unsigned at = 32u * g - kk * pair;  // element of the pair; even
    unsigned sampled_free = 0;
    if (at < pair) {
        unsigned word = 0;
        for (unsigned done = 0; done < 32u && kk < pairs;) {
            // at / row, off by one at most
            unsigned J = static_cast<unsigned>(__uint2float_rz(at) * per_row);
            if (J * row > at) --J;
            if ((J + 1u) * row <= at) ++J;
            const unsigned e = at - J * row, n = min(32u - done, min(row - e, pair - at));
            // columns I = c, c + 1, .. hold grid columns c - 1, c, ..: a window of
            // the rows' bits from c - 1 on, ORed with itself one column on. The
            // words left of the first and right of the last are another row's.
            const int c = static_cast<int>(e >> 1), i = (c - 1) >> 5;
            const unsigned in_lo = i >= 0 ? 0xFFFFFFFFu : 0u;
            const unsigned in_hi = i + 1 < static_cast<int>(nz_words) ? 0xFFFFFFFFu : 0u;
            const unsigned* w = nz + 2u * kk * slice + static_cast<size_t>(J) * nz_words + i;
            unsigned lo[3], hi[3];  // per slice, rows J and J + 1
#pragma unroll
            for (int z = 0; z < 3; ++z, w += slice) {
                lo[z] = __ldg(w) | __ldg(w + nz_words);
                hi[z] = __ldg(w + 1) | __ldg(w + nz_words + 1);
            }
            auto busy = [&](unsigned l, unsigned h) {  // of 16 columns, to the even bits
                unsigned x = __funnelshift_r(l & in_lo, h & in_hi, static_cast<unsigned>(c - 1));
                x = (x | (x >> 1)) & 0xFFFFu;
                x = (x | (x << 8)) & 0x00FF00FFu;
                x = (x | (x << 4)) & 0x0F0F0F0Fu;
                x = (x | (x << 2)) & 0x33333333u;
                return (x | (x << 1)) & 0x55555555u;
            };
            const unsigned b = busy(lo[0] | lo[1], hi[0] | hi[1]) |
                               (busy(lo[1] | lo[2], hi[1] | hi[2]) << 1);
            const unsigned f = ~b & (0xFFFFFFFFu >> (32u - n));
            word |= f << done;
            // the sampled cells among them: columns up to nx of rows up to ny
            const int cells = J <= static_cast<unsigned>(ny) ? nx + 1 - c : 0;
            if (cells > 0) sampled_free += __popc(cells >= 16 ? f : f & ((1u << (2 * cells)) - 1u));
            done += n;
            at += n;
            if (at == pair) {
                at = 0;
                ++kk;
            }
        }
        fr[g] = word;
    }
    const unsigned free_here = __reduce_add_sync(0xffffffffu, sampled_free);
    if (free_here >= kSparseFree && (threadIdx.x & 31) == 0) *sparse = 1;
    // at the end: blocks of a march placed earlier would gather on the SMs that
    // empty first (64x80x72 FP16 frame of 640x480 pixels 49.4 against 48.5 us)
    release_next();
}

__global__ void export_kernel(const void* __restrict__ data, int storage, unsigned row,
                              unsigned pair, int nx, int ny, const float* __restrict__ scales,
                              float4* __restrict__ dst) {
    const int i = blockIdx.x * 32 + threadIdx.x;
    const int j = blockIdx.y * 8 + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= nx || j >= ny) return;
    const size_t v = (static_cast<size_t>(k) * ny + j) * nx + i;
    const unsigned Kp = k + 1;
    const size_t src = static_cast<size_t>(Kp >> 1) * pair + static_cast<size_t>(j + 1) * row +
                       2u * (i + 1) + (Kp & 1u);
    if (storage == HH_STORE_FP32) {
        dst[v] = reinterpret_cast<const float4*>(data)[src];
    } else {
        const ushort4 q = reinterpret_cast<const ushort4*>(data)[src];
        const float s_n = scales[0], s_g = scales[1];
        dst[v] = make_float4(__half2float(__ushort_as_half(q.x)) * s_n,
                             __half2float(__ushort_as_half(q.y)) * s_g,
                             __half2float(__ushort_as_half(q.z)) * s_g,
                             __half2float(__ushort_as_half(q.w)) * s_g);
    }
}

}  // namespace

cudaError_t launch_field(const float* rho, int nx, int ny, int nz, float K, hh_volume_s* vol,
                         bool max_clear, cudaStream_t s) {
    // eight warps of 32 columns a block, rows padded to whole warps; blockIdx.y
    // picks the run of slice pairs: eight, or fewer where that leaves the chip's
    // 152 SMs with less than four blocks each
    const bool halo = vol->layout == HH_LAYOUT_ZPAIR;
    const dim3 block(256);
    auto grid_of = [&](int h, int& run) {
        const unsigned row_pairs = (ny + 2 * h + 1) / 2, pairs = (nz + 2 * h + 1) / 2;
        const unsigned blocks = (row_pairs * ((nx + 31) / 32) + 7) / 8;
        run = 8;
        while (run > 1 && blocks * ((pairs + run - 1) / run) < 608) run /= 2;
        return dim3(blocks, (pairs + run - 1) / run);
    };
    int run = 0;
    const dim3 grid = grid_of(halo ? 1 : 0, run);
    if (vol->storage == HH_STORE_FP32) {
        launch_next(halo ? field_kernel<0, 1> : field_kernel<0, 0>, grid, block, s, rho, nx, ny, nz,
                    K, run, vol->row, vol->pair, vol->data, vol->nz_dev, vol->sparse_dev, nullptr,
                    vol->scales_dev);
        count_launch();
    } else {
        if (!max_clear) {
            const cudaError_t e = cudaMemsetAsync(vol->max_dev, 0, 2 * sizeof(unsigned), s);
            if (e != cudaSuccess) return e;
        }
        int max_run = 0;
        const dim3 max_grid = grid_of(0, max_run);
        launch_next(field_kernel<1, 0>, max_grid, block, s, rho, nx, ny, nz, K, max_run, 0, 0,
                    nullptr, nullptr, nullptr, vol->max_dev, vol->scales_dev);
        launch_next(field_kernel<2, 1>, grid, block, s, rho, nx, ny, nz, K, run, vol->row,
                    vol->pair, vol->data, vol->nz_dev, vol->sparse_dev, vol->max_dev,
                    vol->scales_dev);
        count_launch(2);
    }
    if (halo) {
        const unsigned pairs = (nz + 3) / 2;
        const dim3 mgrid((vol->pair / 32 + 1 + 255) / 256, pairs);
        launch_next(free_mask_kernel, mgrid, block, s, vol->nz_dev, vol->nz_words, nx, ny, pairs,
                    vol->row, vol->pair, 1.0f / static_cast<float>(vol->row), vol->free_dev,
                    vol->sparse_dev);
        count_launch();
    }
    return cudaGetLastError();
}

cudaError_t launch_export(const hh_volume_s* vol, float4* dst, cudaStream_t s) {
    if (vol->layout != HH_LAYOUT_ZPAIR) return cudaErrorInvalidValue;
    const dim3 block(32, 8);
    const dim3 grid((vol->nx + 31) / 32, (vol->ny + 7) / 8, vol->nz);
    export_kernel<<<grid, block, 0, s>>>(vol->data, vol->storage, vol->row, vol->pair, vol->nx,
                                         vol->ny, vol->scales_dev, dst);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hh
