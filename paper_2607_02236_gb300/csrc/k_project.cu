// Push conversion into band-limited block coefficients (the compressed staging form).
//
// The energies of a stream cover a band of beta = (E_max - E_min) dt / h cycles per frame, usually a
// small part of the +-1/2 a frame interval resolves.  Seen through those energies a block of B
// consecutive frames has only about beta B + 8 degrees of freedom, so instead of B frames the staging
// area takes the block's R < B coefficients on an orthonormal basis of that band (discrete prolate
// spheroidal sequences v_q, real, even or odd about the block's centre):
//
//   z[b, q] = sum_u v_q[u] m[t] (psi[t] - mu_hat),   t = b B + u,   m[t] = w_t exp(-2 pi i f_c (u - (B-1)/2))
//
// with the window and the shift to the band's centre f_c in m.  The contraction then runs over
// coefficients as it runs over frames (32 staged slots to a block of its rows, its own twiddle table),
// with R / B of the work, and the staged rows are R / B as long.  k_tables.cu holds the expansion, and
// tacaw_band.cu chooses R at plan creation for a reconstruction error of 1e-7 (kBandTol).
//
// One thread per row (probe, ROI pixel); a CTA takes groups of 128 rows of the push, all blocks of a group
// one after another, with the frames of the next stages (4 or 8 frames each) in flight into each warp's ring
// in shared memory: cp.async keeps them out of the registers that hold the R coefficients, and no
// warp waits for another.  Control flow depends on the CTA alone, so that addresses and loop state sit in
// uniform registers.  Frames u and B-1-u share a basis row: s = x[u] + x[B-1-u] feeds
// the even half of the basis, d = x[u] - x[B-1-u] the odd half, R real x complex products a pair as
// packed FMAs on two coefficients at a time, weights from shared memory (one broadcast 16-byte load for
// four coefficients).  Bound: the frames read once and the coefficients written once, (8 + 8 R / B)
// bytes a (row, frame) against 16 for the staged frames of the dense form; about R + 12 FP32
// operations a (row, frame).  Pushes that end inside a block leave its frames (psi - mu_hat, FP32) in
// the carry [B][M_pad], read back by the push that completes the block.
#include <math_constants.h>

#include "tacaw_internal.cuh"

namespace tacaw {

// A stage of a warp's ring: this many pairs of frames; all slots but one in flight while one is multiplied.
// The weights come from the kernel's parameters (constant bank: no shared-memory wavefronts) on the split
// path, from shared memory on the FP32 path, whose 128-frame blocks have a basis too large for the
// constant cache.  Measured on 64-frame pushes of 2^19 rows (B 64, R 24): 2.63 ps a (row, frame) with
// 2-pair stages and parameters, 2.79 with shared memory, 2.99 with 4-pair stages and parameters; FP32
// (B 128, R 36) 2.40 with 4-pair stages and shared memory, 2.98 with 2-pair stages, 3.12 with parameters.
template <bool SPLIT>
struct ProjRing {
    static constexpr int kPairs = SPLIT ? 2 : 4, kStages = SPLIT ? 6 : 4;
};

// Element offset of row m in a pushed frame.
__device__ __forceinline__ int64_t proj_row(const FrameGeom &g, uint32_t m) {
    const uint32_t npix = (uint32_t)g.npix, kx = (uint32_t)g.kx;   // rows fit 32 bits (checked at plan creation)
    const uint32_t p = m / npix, pix = m - p * npix, y = pix / kx, x = pix - y * kx;
    return (int64_t)p * g.pitch_probe + (int64_t)(g.roi_y0 + (int)y) * g.pitch_row + (g.roi_x0 + (int)x);
}

// 8-byte asynchronous copy global -> shared; zeros when bytes is 0 (the address is not read).
__device__ __forceinline__ void proj_copy(float2 *dst, const float2 *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes)
                 : "memory");
}

// tot + rest += part, the rounding of tot kept in rest (Knuth's two-sum).  The residual sums behind the exact
// mean round no more than those of plain frames, which go to FP64 after 8 frames (FP32 path) or 32 (split path).
// With frames of size a and unit rounding u: on the FP32 path sums of 16 frames from four sums of four (68 a u, two sums
// of eight one by one 70) are added this way; FP64 adds would be two additions and two conversions each, on a pipe with
// a 64th of the FP32 rate.  On the split path a block's sums of four frames are added in FP32: 668 a u for 64 frames,
// two sums of 32 one by one 1054.  Cost: the FP32 scan (blocks of 128 frames, R 36) 6.14 ms instead of 6.08.
__device__ __forceinline__ void add_partial(float2 &tot, float2 &rest, float2 part) {
    const float2 t = __fadd2_rn(tot, part);
    const float2 b = __fadd2_rn(t, make_float2(-tot.x, -tot.y));       // the part as it went in
    const float2 a = __fadd2_rn(t, make_float2(-b.x, -b.y));           // tot as it went in
    rest = __fadd2_rn(rest, __fadd2_rn(__fadd2_rn(tot, make_float2(-a.x, -a.y)),
                                       __fadd2_rn(part, make_float2(-b.x, -b.y))));
    tot = t;
}
// (one lane alone adds to a row in a launch: the sum's order is fixed)
__device__ __forceinline__ void add_residual(double2 *sum_res, float2 tot) {
    atomicAdd(&sum_res->x, (double)tot.x);
    atomicAdd(&sum_res->y, (double)tot.y);
}
__device__ __forceinline__ void add_residual(double2 *sum_res, float2 tot, float2 rest) {
    atomicAdd(&sum_res->x, (double)tot.x + (double)rest.x);
    atomicAdd(&sum_res->y, (double)tot.y + (double)rest.y);
}

// (re, im) of a scaled coefficient as fp16 hi + lo (22 bits), re in the low half.
__device__ __forceinline__ void proj_split_f16(float2 r, uint32_t &hi, uint32_t &lo) {
    const __half2 h = __float22half2_rn(r);
    const float2 b = __half22float2(h);
    const __half2 l = __float22half2_rn(__fadd2_rn(r, make_float2(-b.x, -b.y)));
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
__device__ __forceinline__ uint32_t scale_f16x2(uint32_t v, float f) {
    const float x = __half2float(__ushort_as_half((unsigned short)(v & 0xffffu))) * f;
    const float y = __half2float(__ushort_as_half((unsigned short)(v >> 16))) * f;
    return (uint32_t)__half_as_ushort(__float2half_rn(x)) | ((uint32_t)__half_as_ushort(__float2half_rn(y)) << 16);
}

// Multiplies the staged coefficients [0, slots) of this lane's row by f (a power of two; 1: left alone):
// rows whose coefficients outgrow the range their scale was chosen for.  All lanes of the warp call it and
// share each row's chunks, whole 128-byte lines at a time (one lane to a row walks its chunks one after
// another, and rows outgrow their scales at different blocks, so the lanes of a warp wait for one another).
__device__ __noinline__ void rescale_rows(const ProjEntry &e, int64_t m, int slots, float f) {
    const int lane = threadIdx.x & 31;
    for (unsigned todo = __ballot_sync(0xffffffffu, f != 1.f); todo; todo &= todo - 1) {
        const int r = __ffs(todo) - 1;
        const float g = __shfl_sync(0xffffffffu, f, r);
        const int64_t row = m - lane + r;
        for (int h = 0; h < 2; ++h) {
            uint4 *out = reinterpret_cast<uint4 *>(h ? e.A_lo : e.A_hi);
            for (int ch = lane; ch < slots / 4; ch += 32) {
                uint4 *q = out + ((size_t)(ch >> 3) * e.M_pad + row) * 8 + ((ch & 7) ^ (int)(row & 7));
                uint4 v = *q;
                v.x = scale_f16x2(v.x, g);
                v.y = scale_f16x2(v.y, g);
                v.z = scale_f16x2(v.z, g);
                v.w = scale_f16x2(v.w, g);
                *q = v;
            }
        }
    }
}

// Exponent of the scale of a row whose first nonzero block has largest component zmax, where the window
// grows by 2^growth from that block to its largest in the ring: the ring's largest coefficient to about
// 2^6, so that it may outgrow the window 500-fold before the row is rescaled (the range ends at 2^15), but the
// block itself no lower than 2^-4, 20 bits above the smallest fp16 step.  Scales from the first block alone
// had nearly every row rescaled under Blackman-Harris, which grows by more than 2^14: a segment of 16 200 rows x
// 6681 frames took 5.89 ms and takes 1.00 (plain frames 1.20), the scan of 2^20 rows x 2048 frames 15.1 and 9.96.
__device__ __forceinline__ float row_scale_for(float zmax, int growth) {
    const int x = max(6 - growth, -4) - ilogbf(zmax);
    return exp2f((float)max(-120, min(120, x)));
}

// Shared memory of a CTA of four warps: the basis, then per warp ring, modulation, transposition tile.
template <int B, int R, bool SPLIT>
struct ProjSmem {
    static constexpr int kPairs = ProjRing<SPLIT>::kPairs, kStages = ProjRing<SPLIT>::kStages;
    static constexpr int kBasis = SPLIT ? 0 : B / 2 * R * 4;
    static constexpr int kRing = kStages * 2 * kPairs * 32 * 8;
    static constexpr int kMod = B * 8;
    static constexpr int kTile = SPLIT ? 32 * (R / 4) * 16 : 0;
    static constexpr int kWarp = kRing + kMod + kTile;
    static constexpr int kBytes = (kBasis + 15) / 16 * 16 + 4 * kWarp;
    // resident CTAs: by registers (2 R sums and about 54 or 80 more a thread) and by shared memory
    static constexpr int kRegs = 2 * R + (SPLIT ? 54 : 80);
    static constexpr int kByRegs = 65536 / (128 * ((kRegs + 7) / 8 * 8));
    static constexpr int kBySmem = 227 * 1024 / (kBytes + 1024);
    static constexpr int kCtas = kByRegs < kBySmem ? kByRegs : kBySmem;
};

// SPLIT: fp16 hi/lo rows of 32 slots, pre-swizzled (chunk c of row m at c ^ (m mod 8)); else FP32
// [slot][M_pad].  fp16 pieces carry 22 bits against 16 of bf16 pieces, which the few coefficients of
// a block need (a tone sits in two or three of them, so their roundings average over fewer terms
// than those of its B frames: bf16 pieces of them measured 1.4e-6 of the intensities on the scan of
// 2048 frames, bf16 pieces of the frames 0.5e-6); the fp16 range is met by a power-of-two scale per
// row, taken from the ring's first nonzero block and the window (row_scale_for) and undone in the
// contraction's epilogue.  A row that outgrows it has its staged coefficients rescaled.
// CHECK: frame components beyond 65504 / e.f16_scale set DEVERR_FP16_RANGE (split-FP16 plans): 1: of the frames less
// their provisional mean, as those of plain frames; 2: of the frames as they are (a kept mean stays in plain frames).
// ONE: a launch of one entry, whose fields then are constants of the launch and not loads by index.
template <int B, int R, bool SPLIT, int CHECK, bool ONE>
__global__ void __launch_bounds__(128, ProjSmem<B, R, SPLIT>::kCtas)
    project_group_kernel(const __grid_constant__ ProjGroup pg) {
    using SM = ProjSmem<B, R, SPLIT>;
    constexpr int KP = SM::kPairs, NS = SM::kStages;
    constexpr int H = B / 2, NC = R / 4, RH = R / 2, RP = R / 4;   // RP: coefficient pairs of a parity
    extern __shared__ __align__(16) unsigned char proj_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *sv = reinterpret_cast<float *>(proj_smem);
    unsigned char *mine = proj_smem + (SM::kBasis + 15) / 16 * 16 + warp * SM::kWarp;
    float2 *ring = reinterpret_cast<float2 *>(mine) + lane;                  // [stage][2 KP][32]
    float4 *sm = reinterpret_cast<float4 *>(mine + SM::kRing);               // [H] (m[u], m[B-1-u])
    uint4 *tile = reinterpret_cast<uint4 *>(mine + SM::kRing + SM::kMod);    // [32][NC]
    if (!SPLIT) {
        for (int i = threadIdx.x; i < H * R; i += 128) sv[i] = pg.basis[i];
        __syncthreads();
    }

    const int total = (int)pg.groups, step = (int)gridDim.x, first_group = (int)blockIdx.x;
    auto entry_of = [&](int rg) {
        int i = 0;
        while (!ONE && i + 1 < pg.n && rg >= pg.e[i + 1].group_begin) ++i;
        return i;
    };
    // The next stage to copy: block pk, stage pst of row group prg (entry pe); groups without a whole
    // block have nothing to copy.
    int prg = first_group, pe = 0, pk = 0, pst = 0;
    const float2 *pa = nullptr, *pb = nullptr;    // this thread's row in frames KP pst and B-1 - KP pst of the block
    uint32_t pm = 0;
    int pbytes = 0;                               // 8, or 0 for a padding row
    float2 mu_next = make_float2(0.f, 0.f);
    auto open_copy = [&]() {
        for (; prg < total; prg += step) {
            pe = entry_of(prg);
            if (pg.e[ONE ? 0 : pe].nblk > 0) break;
        }
        if (prg < total) {
            const ProjEntry &e = pg.e[ONE ? 0 : pe];
            pm = (uint32_t)(prg - (int)e.group_begin) * 128u + threadIdx.x;
            const bool valid = (int64_t)pm < e.g.M;
            pbytes = valid ? 8 : 0;
            pa = e.g.base + (valid ? proj_row(e.g, pm) : 0) - (int64_t)e.c0 * e.g.pitch_frame;
            pb = pa + (int64_t)(B - 1) * e.g.pitch_frame;
            mu_next = valid ? e.mu_hat[pm] : make_float2(0.f, 0.f);
            pk = pst = 0;
        }
    };
    int put = 0;
    auto copy_stage = [&]() {
        if (prg < total) {
            const ProjEntry &e = pg.e[ONE ? 0 : pe];
            const int f0 = pk * B - e.c0;
            const int64_t pitch = e.g.pitch_frame;
            float2 *dst = ring + put * (2 * KP * 32);
            if (f0 >= 0 && f0 + B <= e.n) {
#pragma unroll
                for (int i = 0; i < KP; ++i) {
                    proj_copy(dst + i * 32, pa, pbytes);
                    proj_copy(dst + (KP + i) * 32, pb, pbytes);
                    pa += pitch;
                    pb -= pitch;
                }
            } else {
                // frames before the push are in the carry; frames past the segment's end are zero, as padding
                // rows are, whose carry nobody writes
#pragma unroll
                for (int i = 0; i < KP; ++i) {
                    const int u = KP * pst + i, v = B - 1 - u, f = f0 + u, g = f0 + v;
                    proj_copy(dst + i * 32, f < 0 ? e.carry + (int64_t)u * e.M_pad + pm : pa, f < e.n ? pbytes : 0);
                    proj_copy(dst + (KP + i) * 32, g < 0 ? e.carry + (int64_t)v * e.M_pad + pm : pb, g < e.n ? pbytes : 0);
                    pa += pitch;
                    pb -= pitch;
                }
            }
            if (++pst == H / KP) {
                pst = 0;
                pa += (int64_t)H * pitch;         // from u = B/2 to the next block's u = 0
                pb += (int64_t)(B + H) * pitch;   // from u = B/2 - 1 to the next block's u = B - 1
                if (++pk == e.nblk) {
                    prg += step;
                    open_copy();
                }
            }
        }
        put = (put + 1) % NS;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    open_copy();
#pragma unroll 1
    for (int i = 0; i < NS - 1; ++i) copy_stage();

    int get = 0;
    const float2 *mod_now = nullptr;
#pragma unroll 1
    for (int rg = first_group; rg < total; rg += step) {
        const ProjEntry &e = pg.e[ONE ? 0 : entry_of(rg)];
        const uint32_t m = (uint32_t)(rg - (int)e.group_begin) * 128u + threadIdx.x;
        // (a block has more stages than the ring, so the copies are in this group: mu_next is its mean)
        const float2 mu = e.nblk > 0 ? mu_next : ((int64_t)m < e.g.M ? e.mu_hat[m] : make_float2(0.f, 0.f));
        float amax = 0.f;
        float sc = SPLIT && e.nblk > 0 && e.slot0 > 0 ? e.row_scale[m] : 0.f;
#pragma unroll 1
        for (int k = 0; k < e.nblk; ++k) {
            const int f0 = k * B - e.c0;          // pushed frame at the block's u = 0 (negative: in the carry)
            const float2 *mod = e.mod + e.t_block + k * B;
            if (mod != mod_now) {
                __syncwarp();
                for (int u = lane; u < H; u += 32) {
                    const float2 a = mod[u], b = mod[B - 1 - u];
                    sm[u] = make_float4(a.x, a.y, b.x, b.y);
                }
                __syncwarp();
                mod_now = mod;
            }
            const bool whole = f0 >= 0 && f0 + B <= e.n;
            // coefficient pairs (2 i, 2 i + 1) of the even and the odd half
            float2 er[RP], ei[RP], dr[RP], di[RP];
            float2 tot = make_float2(0.f, 0.f), rest = tot, part = tot;   // sum of the residuals (rest: add_partial's)
#pragma unroll
            for (int i = 0; i < RP; ++i) er[i] = ei[i] = dr[i] = di[i] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int st = 0; st < H / KP; ++st) {
                asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
                float2 y[2 * KP];
#pragma unroll
                for (int i = 0; i < 2 * KP; ++i) y[i] = ring[(get * 2 * KP + i) * 32];
                get = (get + 1) % NS;
                copy_stage();                     // into the slot read one stage ago
                const float2 nmu = make_float2(-mu.x, -mu.y);
                if (CHECK == 2) {                 // (carried frames were checked when they came)
#pragma unroll
                    for (int i = 0; i < 2 * KP; ++i) {
                        const int f = f0 + (i < KP ? KP * st + i : B - 1 - KP * st - (i - KP));
                        if (f >= 0) amax = fmaxf(amax, fmaxf(fabsf(y[i].x), fabsf(y[i].y)));
                    }
                }
                float2 s0 = make_float2(0.f, 0.f), s1 = s0;   // residuals of the block's front and back frames
                if (whole) {
#pragma unroll
                    for (int i = 0; i < 2 * KP; ++i) {
                        y[i] = __fadd2_rn(y[i], nmu);
                        float2 &s = i < KP ? s0 : s1;
                        s = i % KP == 0 ? y[i] : __fadd2_rn(s, y[i]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 2 * KP; ++i) {
                        const int f = f0 + (i < KP ? KP * st + i : B - 1 - KP * st - (i - KP));
                        if (f >= 0 && f < e.n) {   // (carried frames are residuals, already counted)
                            y[i] = __fadd2_rn(y[i], nmu);
                            float2 &s = i < KP ? s0 : s1;
                            s = __fadd2_rn(s, y[i]);
                        }
                    }
                }
                if (SPLIT) {
                    tot = __fadd2_rn(tot, __fadd2_rn(s0, s1));
                } else {
                    part = __fadd2_rn(part, __fadd2_rn(s0, s1));
                    if (st & 1) {
                        add_partial(tot, rest, part);
                        part = make_float2(0.f, 0.f);
                    }
                }
                if (CHECK == 1) {
#pragma unroll
                    for (int i = 0; i < 2 * KP; ++i) amax = fmaxf(amax, fmaxf(fabsf(y[i].x), fabsf(y[i].y)));
                }
#pragma unroll
                for (int i = 0; i < KP; ++i) {
                    const int u = KP * st + i;
                    const float4 mm = sm[u];
                    const float2 a = y[i], b = y[KP + i];
                    const float2 xa = make_float2(a.x * mm.x - a.y * mm.y, a.x * mm.y + a.y * mm.x);
                    const float2 xb = make_float2(b.x * mm.z - b.y * mm.w, b.x * mm.w + b.y * mm.z);
                    const float2 s = __fadd2_rn(xa, xb), d = make_float2(xa.x - xb.x, xa.y - xb.y);
                    const float2 sr = make_float2(s.x, s.x), si = make_float2(s.y, s.y);
                    const float2 tr = make_float2(d.x, d.x), ti = make_float2(d.y, d.y);
                    const float *v = SPLIT ? pg.basis + u * R : sv + u * R;
#pragma unroll
                    for (int q = 0; q < RP; q += 2) {
                        // (RH = 2 RP weights a half: 16-byte loads where RP is even, 8-byte else)
                        float2 w0, w1, o0, o1;
                        if (RP % 2 == 0) {
                            const float4 x = *reinterpret_cast<const float4 *>(v + 2 * q);
                            const float4 z = *reinterpret_cast<const float4 *>(v + RH + 2 * q);
                            w0 = make_float2(x.x, x.y);
                            w1 = make_float2(x.z, x.w);
                            o0 = make_float2(z.x, z.y);
                            o1 = make_float2(z.z, z.w);
                        } else {
                            w0 = *reinterpret_cast<const float2 *>(v + 2 * q);
                            o0 = *reinterpret_cast<const float2 *>(v + RH + 2 * q);
                            w1 = q + 1 < RP ? *reinterpret_cast<const float2 *>(v + 2 * q + 2) : w0;
                            o1 = q + 1 < RP ? *reinterpret_cast<const float2 *>(v + RH + 2 * q + 2) : o0;
                        }
                        er[q] = __ffma2_rn(w0, sr, er[q]);
                        ei[q] = __ffma2_rn(w0, si, ei[q]);
                        dr[q] = __ffma2_rn(o0, tr, dr[q]);
                        di[q] = __ffma2_rn(o0, ti, di[q]);
                        if (q + 1 < RP) {
                            er[q + 1] = __ffma2_rn(w1, sr, er[q + 1]);
                            ei[q + 1] = __ffma2_rn(w1, si, ei[q + 1]);
                            dr[q + 1] = __ffma2_rn(o1, tr, dr[q + 1]);
                            di[q + 1] = __ffma2_rn(o1, ti, di[q + 1]);
                        }
                    }
                }
            }
            if ((int64_t)m < e.g.M) {
                if (SPLIT) add_residual(&e.sum_res[m], tot);
                else add_residual(&e.sum_res[m], tot, rest);
            }
            // coefficient q of the block: even half first
            auto z = [&](int q) {
                const int i = (q % RH) >> 1;
                const float2 re = q < RH ? er[i] : dr[i], im = q < RH ? ei[i] : di[i];
                return (q & 1) ? make_float2(re.y, im.y) : make_float2(re.x, im.x);
            };
            const int slot = e.slot0 + k * R;
            if (SPLIT) {
                float zmax = 0.f;
#pragma unroll
                for (int q = 0; q < R; ++q) zmax = fmaxf(zmax, fmaxf(fabsf(z(q).x), fabsf(z(q).y)));
                const bool fresh = (sc == 0.f ? zmax > 0.f : zmax * sc > 32768.f) && zmax < CUDART_INF_F;
                if (__any_sync(0xffffffffu, fresh)) {
                    const float ns = fresh ? row_scale_for(zmax, e.growth[k]) : sc;
                    rescale_rows(e, m, slot, fresh && sc != 0.f ? ns / sc : 1.f);
                    sc = ns;
                }
                const float s = sc == 0.f ? 1.f : sc;
                const int c0 = slot / 4;
                // a tail after the ring's last block: zero chunks up to the end of the 32-slot row
                const int zc = k == e.nblk - 1 ? e.zero_slots / 4 : 0;
                const int64_t m0 = (int64_t)m - lane;
                uint32_t hi[R], lo[R];
#pragma unroll
                for (int q = 0; q < R; ++q) proj_split_f16(__fmul2_rn(z(q), make_float2(s, s)), hi[q], lo[q]);
                // rows transposed through the warp's tile, so that consecutive lanes store consecutive
                // 16-byte chunks of a row; hi pieces first, then lo
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t *p = h ? lo : hi;
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        tile[lane * NC + (c + lane) % NC] = make_uint4(p[4 * c], p[4 * c + 1], p[4 * c + 2], p[4 * c + 3]);
                    __syncwarp();
                    uint4 *out = reinterpret_cast<uint4 *>(h ? e.A_lo : e.A_hi);
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const int i = j * 32 + lane, rr = i / NC, c = i - rr * NC, ch = c0 + c;
                        out[((size_t)(ch >> 3) * e.M_pad + m0 + rr) * 8 + ((ch & 7) ^ (rr & 7))] =
                            tile[rr * NC + (c + rr) % NC];
                    }
                    for (int c = 0; c < zc; ++c) {
                        const int ch = c0 + NC + c;
                        out[((size_t)(ch >> 3) * e.M_pad + m) * 8 + ((ch & 7) ^ (lane & 7))] = make_uint4(0, 0, 0, 0);
                    }
                }
                // the rescaling of a later block reads what other lanes stored for this row
                __syncwarp();
            } else {
                float2 *out = e.A32 + (size_t)slot * e.M_pad + m;
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    *out = z(q);
                    out += e.M_pad;
                }
            }
        }
        if (SPLIT && e.nblk > 0) e.row_scale[m] = sc;
        // frames past the last whole block wait in the carry
        const int done = e.nblk * B - e.c0;       // pushed frames used by the blocks above
        const int first = done > 0 ? done : 0;
        if (first < e.n) {
            const bool valid = (int64_t)m < e.g.M;
            const float2 *src = e.g.base + (valid ? proj_row(e.g, m) : 0);
            float2 *carry = e.carry + m;
            const int base = e.nblk > 0 ? -done : e.c0;   // carry slot of pushed frame f: base + f
#pragma unroll 1
            for (int f = first; f < e.n; f += 8) {
                float2 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    v[i] = valid && f + i < e.n ? __ldcs(src + (int64_t)(f + i) * e.g.pitch_frame) : mu;
                float2 sum = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (f + i < e.n) {
                        const float2 y = make_float2(v[i].x - mu.x, v[i].y - mu.y);
                        sum = __fadd2_rn(sum, y);
                        if (CHECK) {
                            const float2 c = CHECK == 2 ? v[i] : y;
                            amax = fmaxf(amax, fmaxf(fabsf(c.x), fabsf(c.y)));
                        }
                        carry[(int64_t)(base + f + i) * e.M_pad] = y;
                    }
                if (valid) add_residual(&e.sum_res[m], sum);
            }
        }
        if (CHECK && amax * e.f16_scale > 65504.f) atomicOr(e.err, DEVERR_FP16_RANGE);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Pushes that complete no block: their frames' residuals go to the carry, 8 bytes read and 8 written a
// (row, frame) at full occupancy; their sums to FP64 every 32 frames (SPLIT) or 16 (by fours), straight to memory: kept in
// registers over the push (add_partial) the longer code cost more than the atomics (16-frame pushes of 10^4 rows
// x 2048 frames, FP32: 1.47 ms a segment against 1.29).  CTA b: rows 128 (b - group_begin) .. of its entry.
template <int CHECK, bool SPLIT>
__global__ void __launch_bounds__(128, 8) carry_group_kernel(const __grid_constant__ ProjGroup pg) {
    int i = 0;
    while (i + 1 < pg.n && (int64_t)blockIdx.x >= pg.e[i + 1].group_begin) ++i;
    const ProjEntry &e = pg.e[i];
    const uint32_t m = (uint32_t)((int64_t)blockIdx.x - e.group_begin) * 128u + threadIdx.x;
    if ((int64_t)m >= e.g.M) return;
    const int64_t pitch = e.g.pitch_frame;
    const float2 *src = e.g.base + proj_row(e.g, m);
    float2 *carry = e.carry + m + (int64_t)e.c0 * e.M_pad;
    const float2 mu = e.mu_hat[m];
    float2 sum = make_float2(0.f, 0.f);
    float amax = 0.f;
    for (int f0 = 0; f0 < e.n; f0 += 16) {
        float2 v[16], four[4] = {};
#pragma unroll
        for (int f = 0; f < 16; ++f) v[f] = f0 + f < e.n ? __ldcs(src + (int64_t)(f0 + f) * pitch) : mu;
#pragma unroll
        for (int f = 0; f < 16; ++f)
            if (f0 + f < e.n) {
                const float2 y = make_float2(v[f].x - mu.x, v[f].y - mu.y);
                float2 &s = SPLIT ? sum : four[f / 4];
                s.x += y.x;
                s.y += y.y;
                if (CHECK) {
                    const float2 c = CHECK == 2 ? v[f] : y;
                    amax = fmaxf(amax, fmaxf(fabsf(c.x), fabsf(c.y)));
                }
                carry[(int64_t)(f0 + f) * e.M_pad] = y;
            }
        if (!SPLIT) sum = __fadd2_rn(__fadd2_rn(four[0], four[1]), __fadd2_rn(four[2], four[3]));
        if (!SPLIT || (f0 & 16)) {
            add_residual(&e.sum_res[m], sum);
            sum = make_float2(0.f, 0.f);
        }
    }
    if (SPLIT) add_residual(&e.sum_res[m], sum);
    if (CHECK && amax * e.f16_scale > 65504.f) atomicOr(e.err, DEVERR_FP16_RANGE);
}

template <int B, int R, bool SPLIT, int CHECK>
static cudaError_t launch_project_kernel(const ProjGroup &pg, cudaStream_t st) {
    using SM = ProjSmem<B, R, SPLIT>;
    auto *kern = pg.n == 1 ? project_group_kernel<B, R, SPLIT, CHECK, true> : project_group_kernel<B, R, SPLIT, CHECK, false>;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && SM::kBytes > 48 * 1024)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SM::kBytes);
    if (e != cudaSuccess) return e;
    // one wave of CTAs walks the row groups
    const int64_t wave = (int64_t)sms * SM::kCtas;
    kern<<<(unsigned)(pg.groups < wave ? pg.groups : wave), 128, SM::kBytes, st>>>(pg);
    return cudaGetLastError();
}

template <int B, int R>
static cudaError_t launch_project_shape(const ProjGroup &pg, bool split, cudaStream_t st) {
    if constexpr (B == 32 || (B == 64 && R <= 36)) {
        if (split && pg.check == 2) return launch_project_kernel<B, R, true, 2>(pg, st);
        if (split && pg.check == 1) return launch_project_kernel<B, R, true, 1>(pg, st);
        if (split) return launch_project_kernel<B, R, true, 0>(pg, st);
    }
    if constexpr (B >= 64) return launch_project_kernel<B, R, false, 0>(pg, st);
    return cudaErrorInvalidValue;
}

// Split staging takes blocks of 32 or 64 frames (128 pays only where a push holds them whole and then
// about what 64 does) with up to 24 or 36 coefficients (beyond, the contraction saves too little);
// FP32 staging, whose contraction costs ten times as much a coefficient, 64 or 128.
bool project_shape_ok(int B, int R, bool split) {
    if (R % 4 || R < 8) return false;
    return split ? (B == 32 && R <= 24) || (B == 64 && R <= 36) : (B == 64 || B == 128) && R <= 48;
}

cudaError_t launch_project_group(ProjGroup &pg, int B, int R, bool split, cudaStream_t st) {
    if (pg.n < 1 || pg.n > kConvGroupMax || !project_shape_ok(B, R, split)) return cudaErrorInvalidValue;
    pg.groups = 0;
    for (int i = 0; i < pg.n; ++i) {
        // (entries of one launch share the basis: the same band, B and R)
        if (pg.e[i].M_pad % 128) return cudaErrorInvalidValue;
        pg.e[i].group_begin = pg.groups;
        pg.groups += pg.e[i].M_pad / 128;
    }
    if (pg.groups < 1 || pg.groups > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    bool blocks = false;
    for (int i = 0; i < pg.n; ++i) blocks = blocks || pg.e[i].nblk > 0;
    if (!blocks) {
        void (*kern)(ProjGroup) = !split            ? carry_group_kernel<0, false>
                                  : pg.check == 2   ? carry_group_kernel<2, true>
                                  : pg.check == 1   ? carry_group_kernel<1, true>
                                                    : carry_group_kernel<0, true>;
        kern<<<(unsigned)pg.groups, 128, 0, st>>>(pg);
        return cudaGetLastError();
    }
#define TACAW_PROJ(b, r) \
    if (B == b && R == r) return launch_project_shape<b, r>(pg, split, st);
    TACAW_PROJ(32, 8) TACAW_PROJ(32, 12) TACAW_PROJ(32, 16) TACAW_PROJ(32, 20) TACAW_PROJ(32, 24)
    TACAW_PROJ(64, 8) TACAW_PROJ(64, 12) TACAW_PROJ(64, 16) TACAW_PROJ(64, 20) TACAW_PROJ(64, 24) TACAW_PROJ(64, 28)
    TACAW_PROJ(64, 32) TACAW_PROJ(64, 36) TACAW_PROJ(64, 40) TACAW_PROJ(64, 44) TACAW_PROJ(64, 48)
    TACAW_PROJ(128, 8) TACAW_PROJ(128, 12) TACAW_PROJ(128, 16) TACAW_PROJ(128, 20) TACAW_PROJ(128, 24)
    TACAW_PROJ(128, 28) TACAW_PROJ(128, 32) TACAW_PROJ(128, 36) TACAW_PROJ(128, 40) TACAW_PROJ(128, 44)
    TACAW_PROJ(128, 48)
#undef TACAW_PROJ
    return cudaErrorInvalidValue;
}

}  // namespace tacaw
