// Initial microstructure: Algorithm 1, "Initialization" (Sec. 2.1.3; the
// tessellation input of Sec. 3.1).
//
//   k_labels        power-diagram label of each cell: argmin_i |x - s_i|^2 - w_i
//                   with minimum-image displacements, lowest id on ties.  The
//                   seeds are binned on a uniform grid; a CTA takes a tile of
//                   cells and collects once the seeds that can hold one of them,
//                   its cells compare those in FP32, and candidates within a safe
//                   margin of the minimum are decided in FP64 with explicitly
//                   rounded operations, so the integer result does not depend on
//                   FMA contraction or on the search order.
//   k_label_faces   grains whose cells touch across a face (bit matrix); per
//                   grain, min/max of the integer minimum-image offsets of its
//                   cells from its rounded seed.
//   k_init_boxes    box = that bbox grown by the halo (full axis if it reaches N).
//   k_sdf           phi_i(x) = clamp(min_{j in Nb(i)} signed distance of x to the
//                   power bisector of (i, j), -eps, eps) and the minimising j.
#include <cfloat>
#include <climits>

#include "lsgg_internal.cuh"

namespace lsgg {

// Minimum image d - n * rint(d / n) for |d| < n (cells and seeds in [0, n)):
// rint(d / n) is +1 exactly when d > n / 2 and -1 when d < -n / 2 (n / 2 is
// exact; a double d within half an ulp of 0.5 n is n / 2 itself, whose
// quotient 0.5 rounds to 0), so the division is replaced by comparisons.
// Seeds outside [0, n) take the general form.
__device__ __forceinline__ double min_image(double d, double n) {
    const double h = 0.5 * n;
    if (fabs(d) < n) return d > h ? __dsub_rn(d, n) : (d < -h ? __dadd_rn(d, n) : d);
    return __dsub_rn(d, __dmul_rn(n, rint(__ddiv_rn(d, n))));
}

__device__ __forceinline__ float wrap_half(float d, float n) {
    return d > 0.5f * n ? d - n : (d < -0.5f * n ? d + n : d);
}

// A bin index within one period of [0, nb) (the reach never exceeds a period).
__device__ __forceinline__ int wrap_bin(int i, int nb) { return i < 0 ? i + nb : (i >= nb ? i - nb : i); }

// Bins of one axis to visit around bin c at reach k: [lo, lo + cnt) cyclically.
__device__ __forceinline__ void bin_range(int c, int k, int nb, int& lo, int& cnt) {
    if (2 * k + 1 >= nb) { lo = 0; cnt = nb; }
    else { lo = c - k; cnt = 2 * k + 1; }
}

// Visit every seed in the bin block around (cx, cy, cz) of reach (kx, ky, kz).
template <class F>
__device__ __forceinline__ void for_block(const SeedBins& S, int cx, int cy, int cz, int kx, int ky, int kz, F f) {
    int lx, nx_, ly, ny_, lz, nz_;
    bin_range(cx, kx, S.nb[0], lx, nx_);
    bin_range(cy, ky, S.nb[1], ly, ny_);
    bin_range(cz, kz, S.nb[2], lz, nz_);
    for (int iz = 0; iz < nz_; ++iz) {
        const int bz = wrap_bin(lz + iz, S.nb[2]);
        for (int iy = 0; iy < ny_; ++iy) {
            const int by = wrap_bin(ly + iy, S.nb[1]);
            const int row = (bz * S.nb[1] + by) * S.nb[0];
            for (int ix = 0; ix < nx_; ++ix) {
                const int bin = row + wrap_bin(lx + ix, S.nb[0]);
                for (int q = S.start[bin]; q < S.start[bin + 1]; ++q) f(q);
            }
        }
    }
}

// Visit every seed in the bins that meet [x - r, x + r] on each axis (cyclic;
// a range of a period or more visits the whole axis once).
template <class F>
__device__ __forceinline__ void for_reach(const SeedBins& S, float fx, float fy, float fz, float r, F f) {
    const float c[3] = {fx, fy, fz};
    int lo[3], cnt[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (2.0f * r + 2.0f * S.size[a] >= (float)S.nb[a] * S.size[a]) { lo[a] = 0; cnt[a] = S.nb[a]; continue; }
        const int l = (int)floorf((c[a] - r) / S.size[a]);
        const int h = (int)floorf((c[a] + r) / S.size[a]);
        cnt[a] = h - l + 1;
        lo[a] = l;
        if (cnt[a] >= S.nb[a]) { lo[a] = 0; cnt[a] = S.nb[a]; }
        else { lo[a] %= S.nb[a]; if (lo[a] < 0) lo[a] += S.nb[a]; }
    }
    for (int iz = 0; iz < cnt[2]; ++iz) {
        const int bz = wrap_bin(lo[2] + iz, S.nb[2]);
        for (int iy = 0; iy < cnt[1]; ++iy) {
            const int by = wrap_bin(lo[1] + iy, S.nb[1]);
            const int row = (bz * S.nb[1] + by) * S.nb[0];
            for (int ix = 0; ix < cnt[0]; ++ix) {
                const int bin = row + wrap_bin(lo[0] + ix, S.nb[0]);
                for (int q = S.start[bin]; q < S.start[bin + 1]; ++q) f(q);
            }
        }
    }
}

// The label of one cell (see k_labels).
__device__ __forceinline__ int label_cell(const Domain& D, const SeedBins& S, const double* __restrict__ seeds,
                                          const double* __restrict__ weights, long long cell) {
    const int x = (int)(cell % D.nx);
    const int y = (int)((cell / D.nx) % D.ny);
    const int z = (int)(cell / ((long long)D.nx * D.ny));
    const float fx = (float)x, fy = (float)y, fz = (float)z;
    const float fnx = (float)D.nx, fny = (float)D.ny, fnz = (float)D.nz;
    const int cx = min(S.nb[0] - 1, (int)(fx / S.size[0]));
    const int cy = min(S.nb[1] - 1, (int)(fy / S.size[1]));
    const int cz = min(S.nb[2] - 1, (int)(fz / S.size[2]));
    auto d32 = [&](int q) {
        const float4 p = S.pts[q];
        const float dx = wrap_half(fx - p.x, fnx), dy = wrap_half(fy - p.y, fny), dz = wrap_half(fz - p.z, fnz);
        return dx * dx + dy * dy + dz * dz - p.w;
    };
    // an upper bound from the neighbouring bins, then every seed that can beat it
    float bound = FLT_MAX;
    for_block(S, cx, cy, cz, 1, 1, 1, [&](int q) { bound = fminf(bound, d32(q)); });
    const float nmax = fmaxf(fnx, fmaxf(fny, fnz));
    // margin covering FP32 rounding of |d|^2 <= 3 N^2, of the seeds and of the weights
    auto margin = [&](float v) { return 0.5f + 4e-6f * nmax * nmax + 1e-5f * fabsf(v); };
    // every seed within the margin of the minimum lies within r of the cell
    const float r = bound < FLT_MAX ? sqrtf(fmaxf(0.0f, bound + margin(bound) + S.wmax)) + 1.0f   // + 1: bin-edge rounding
                                    : FLT_MAX;
    // one pass: the FP32 minimum and the seeds within the margin of the running
    // minimum (a superset of those within the margin of the final one); a
    // full candidate list falls back to a second pass
    constexpr int kCand = 8;
    int cand[kCand];
    float cand_d[kCand];
    int n_cand = 0;
    bool rescan = false;
    float best32 = FLT_MAX;
    for_reach(S, fx, fy, fz, r, [&](int q) {
        const float d = d32(q);
        best32 = fminf(best32, d);
        if (d <= best32 + margin(best32)) {
            if (n_cand < kCand) { cand[n_cand] = q; cand_d[n_cand] = d; ++n_cand; }
            else rescan = true;
        }
    });
    const float lim = best32 + margin(best32);
    double best = DBL_MAX;
    int arg = -1;
    auto exact = [&](int q) {
        const int i = S.ids[q];
        const double ex = min_image(__dsub_rn((double)x, seeds[3 * i]), (double)D.nx);
        const double ey = min_image(__dsub_rn((double)y, seeds[3 * i + 1]), (double)D.ny);
        const double ez = min_image(__dsub_rn((double)z, seeds[3 * i + 2]), (double)D.nz);
        double rr = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
        if (weights) rr = __dsub_rn(rr, weights[i]);
        if (rr < best || (rr == best && i < arg)) { best = rr; arg = i; }
    };
    if (!rescan) {
        for (int c = 0; c < n_cand; ++c)
            if (cand_d[c] <= lim) exact(cand[c]);
    } else {
        for_reach(S, fx, fy, fz, r, [&](int q) {
            if (d32(q) <= lim) exact(q);
        });
    }
    return arg;
}

// The labels, a CTA per tile of kLabelCells cells (8 x 8 x 8, in 2D 32 x 16).
// A cell-by-cell search reads every bin within its reach again for every cell,
// and with weights the reach is that of the largest weight (some thousand
// seeds a cell): 440 ms at 512^3 / 40 000 weighted seeds, 4.6 ms at 256^3 /
// 5000 on GB300, against 5.1 and 0.52 ms per tile, bound by the FP32 compares
// (about eight instructions a cell and candidate).  Per tile the search runs once: an upper bound of the power
// distance that some seed keeps over the whole tile (from the bins around its
// centre) leaves the seeds whose smallest distance to the tile does not exceed
// it, typically 20-60, staged in shared memory with FP32 displacements from the
// tile's centre (rounded from FP64, so that the FP32 error is that of the
// displacement and not of the domain's size).  Each cell keeps the smallest
// and second smallest value; unless they are closer than twice the FP32 error
// bound the smallest one's seed is the label, otherwise FP64 decides among the
// candidates within it.  A tile with more than kLabelCand candidates (seeds
// nearly as dense as cells) takes the cell-by-cell search.
constexpr int kLabelCells = 512;
constexpr int kLabelThreads = 256;
constexpr int kLabelCand = 768;

__global__ void __launch_bounds__(kLabelThreads)
k_labels(Domain D, int G, SeedBins S, const double* __restrict__ seeds, const double* __restrict__ weights,
         int* __restrict__ labels, int tx, int ty, int tz, int ntx, int nty) {
    __shared__ float4 s_c[kLabelCand];               // displacement from the tile's centre, weight
    __shared__ int s_q[kLabelCand];                  // sorted seed index
    __shared__ float s_red[kLabelThreads / 32];
    __shared__ float s_far;                          // largest squared reach of a candidate
    __shared__ int s_n, s_wrap;
    const int t = threadIdx.x;
    const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
    const int o[3] = {bx * tx, by * ty, bz * tz};
    const int N[3] = {D.nx, D.ny, D.nz};
    const float fN[3] = {(float)D.nx, (float)D.ny, (float)D.nz};
    const int e[3] = {min(tx, D.nx - o[0]), min(ty, D.ny - o[1]), min(tz, D.nz - o[2])};
    float c[3], h[3];                                // centre and half extent over the cells' points
    int cb[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c[a] = (float)o[a] + 0.5f * (float)(e[a] - 1);
        h[a] = 0.5f * (float)(e[a] - 1);
        cb[a] = min(S.nb[a] - 1, (int)(c[a] / S.size[a]));
    }
    // squared power distances of a seed to the tile: smallest and largest over its cells
    auto range = [&](const float4 p, float& near, float& far) {
        const float q[3] = {p.x, p.y, p.z};
        near = far = -p.w;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float d = fabsf(wrap_half(c[a] - q[a], fN[a]));
            const float n0 = fmaxf(d - h[a], 0.0f), f0 = fminf(d + h[a], 0.5f * fN[a]);
            near = fmaf(n0, n0, near);
            far = fmaf(f0, f0, far);
        }
    };
    // the bins [lo, lo + cnt) per axis (cyclic), spread over the threads
    auto for_bins = [&](const int (&lo)[3], const int (&cnt)[3], auto f) {
        const int nbin = cnt[0] * cnt[1] * cnt[2];
        for (int k = t; k < nbin; k += kLabelThreads) {
            const int ix = k % cnt[0], iy = (k / cnt[0]) % cnt[1], iz = k / (cnt[0] * cnt[1]);
            const int bin = (wrap_bin(lo[2] + iz, S.nb[2]) * S.nb[1] + wrap_bin(lo[1] + iy, S.nb[1])) * S.nb[0] +
                            wrap_bin(lo[0] + ix, S.nb[0]);
            for (int q = S.start[bin]; q < S.start[bin + 1]; ++q) f(q);
        }
    };
    auto block_min = [&](float v) {
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, k));
        __syncthreads();
        if ((t & 31) == 0) s_red[t >> 5] = v;
        __syncthreads();
        v = s_red[0];
#pragma unroll
        for (int k = 1; k < kLabelThreads / 32; ++k) v = fminf(v, s_red[k]);
        return v;
    };
    // an upper bound that one seed keeps over the tile, from the bins around the centre
    float bound = FLT_MAX;
    int lo[3], cnt[3];
    for (int k = 1; bound == FLT_MAX; k *= 2) {
        bool whole = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            bin_range(cb[a], k, S.nb[a], lo[a], cnt[a]);
            whole = whole && cnt[a] == S.nb[a];
        }
        float m = FLT_MAX;
        for_bins(lo, cnt, [&](int q) {
            float near, far;
            range(S.pts[q], near, far);
            m = fminf(m, far);
        });
        bound = block_min(m);
        if (whole) break;
    }
    const float nmax = fmaxf(fN[0], fmaxf(fN[1], fN[2]));
    // margin covering FP32 rounding of |d|^2 <= 3 N^2, of the seeds and of the weights
    bound += 0.5f + 4e-6f * nmax * nmax + 1e-5f * fabsf(bound);
    // the seeds that can hold a cell lie within r of the tile on every axis
    const float r = sqrtf(fmaxf(0.0f, bound + S.wmax)) + 1.0f;   // + 1: bin-edge rounding
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float ra = r + h[a];
        lo[a] = 0;
        cnt[a] = S.nb[a];
        if (2.0f * ra + 2.0f * S.size[a] < (float)S.nb[a] * S.size[a]) {
            const int l = (int)floorf((c[a] - ra) / S.size[a]), u = (int)floorf((c[a] + ra) / S.size[a]);
            if (u - l + 1 < S.nb[a]) {
                cnt[a] = u - l + 1;
                lo[a] = l % S.nb[a];
                if (lo[a] < 0) lo[a] += S.nb[a];
            }
        }
    }
    if (t == 0) { s_n = 0; s_wrap = 0; s_far = 0.0f; }
    __syncthreads();
    for_bins(lo, cnt, [&](int q) {
        const float4 p = S.pts[q];
        float near, far;
        range(p, near, far);
        if (near > bound) return;
        const int k = atomicAdd(&s_n, 1);
        if (k >= kLabelCand) return;
        const int i = S.ids[q];
        float d[3], r2 = 0.0f;
        bool wrap = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            d[a] = (float)min_image(__dsub_rn(seeds[3 * i + a], (double)c[a]), (double)N[a]);
            const float u = fabsf(d[a]) + h[a];
            wrap = wrap || (N[a] > 1 && u > 0.5f * fN[a] - 0.01f);
            r2 = fmaf(u, u, r2);
        }
        s_c[k] = make_float4(d[0], d[1], d[2], p.w);
        s_q[k] = q;
        if (wrap) s_wrap = 1;
        atomicMax(reinterpret_cast<int*>(&s_far), __float_as_int(r2 + fabsf(p.w)));   // non-negative floats
    });
    __syncthreads();
    const int n = s_n;
    const bool wrap = s_wrap != 0;
    // twice the FP32 error of a candidate's value: displacements and squares
    // (5e-7 of the squared reach), the weight's rounding and the difference's
    const float margin = 4e-6f * s_far + 1e-4f;
    for (int k = t; k < e[0] * e[1] * e[2]; k += kLabelThreads) {
        const int x = k % e[0], y = (k / e[0]) % e[1], z = k / (e[0] * e[1]);
        const int g[3] = {o[0] + x, o[1] + y, o[2] + z};
        const long long cell = ((long long)g[2] * D.ny + g[1]) * D.nx + g[0];
        if (n > kLabelCand) {
            labels[cell] = label_cell(D, S, seeds, weights, cell);
            continue;
        }
        const float p[3] = {(float)x - h[0], (float)y - h[1], (float)z - h[2]};
        auto value = [&](int q) {
            const float4 s = s_c[q];
            float dx = p[0] - s.x, dy = p[1] - s.y, dz = p[2] - s.z;
            if (wrap) {
                dx = wrap_half(dx, fN[0]);
                dy = wrap_half(dy, fN[1]);
                dz = wrap_half(dz, fN[2]);
            }
            return fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, -s.w)));
        };
        float v1 = FLT_MAX, v2 = FLT_MAX;
        int k1 = 0;
        for (int q = 0; q < n; ++q) {
            const float v = value(q);
            k1 = v < v1 ? q : k1;
            v2 = fminf(v2, fmaxf(v1, v));
            v1 = fminf(v1, v);
        }
        int arg;
        if (v2 > v1 + margin) {
            arg = S.ids[s_q[k1]];
        } else {
            double best = DBL_MAX;
            arg = -1;
            for (int q = 0; q < n; ++q) {
                if (value(q) > v1 + margin) continue;
                const int i = S.ids[s_q[q]];
                const double ex = min_image(__dsub_rn((double)g[0], seeds[3 * i]), (double)D.nx);
                const double ey = min_image(__dsub_rn((double)g[1], seeds[3 * i + 1]), (double)D.ny);
                const double ez = min_image(__dsub_rn((double)g[2], seeds[3 * i + 2]), (double)D.nz);
                double rr = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
                if (weights) rr = __dsub_rn(rr, weights[i]);
                if (rr < best || (rr == best && i < arg)) { best = rr; arg = i; }
            }
        }
        labels[cell] = arg;
    }
}

__device__ __forceinline__ int offset_from(int x, int r, int n) {
    int e = pmod(x - r, n);
    return e > n / 2 ? e - n : e;
}

// Per grain: its rounded seed's cell, and empty offset bounds.
__global__ void k_bbox_init(Domain D, int G, const double* __restrict__ seeds, int* bb, int* seed_cell) {
    const int N[3] = {D.nx, D.ny, D.nz};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G; i += gridDim.x * blockDim.x) {
        for (int a = 0; a < 3; ++a) {
            bb[6 * i + a] = INT_MAX;
            bb[6 * i + 3 + a] = INT_MIN;
            seed_cell[3 * i + a] = pmod((int)rint(seeds[3 * i + a]), N[a]);
        }
    }
}

__device__ __forceinline__ void set_pair_bit(unsigned* bits, long long words_per_row, int a, int b) {
    unsigned* w = bits + (long long)a * words_per_row + (b >> 5);
    const unsigned m = 1u << (b & 31);
    if (!(*(volatile unsigned*)w & m)) atomicOr(w, m);
}

// A thread per cell and its next cell on every axis (periodic).  Different
// labels: the two grains touch, and only such a cell can be the last of its
// grain on the axis and the next one the first of its own; equal labels count
// only across the cut of the grain's offsets (half a period from its seed).
// Taking every cell's offsets took 6 atomics a cell: 14.9 ms with the pairs at
// 512^3 on GB300, against 2.2 ms.
__global__ void __launch_bounds__(256)
k_label_faces(Domain D, const int* __restrict__ labels, const int* __restrict__ seed_cell,
              unsigned* __restrict__ bits, long long words_per_row, int* __restrict__ bb) {
    const long long ncell = (long long)D.nx * D.ny * D.nz;
    const int N[3] = {D.nx, D.ny, D.nz};
    const long long st[3] = {1, D.nx, (long long)D.nx * D.ny};
    for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < ncell;
         cell += (long long)gridDim.x * blockDim.x) {
        const int c[3] = {(int)(cell % D.nx), (int)((cell / D.nx) % D.ny), (int)(cell / ((long long)D.nx * D.ny))};
        const int a = labels[cell];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (N[k] == 1) continue;
            const int nx = c[k] + 1 < N[k] ? c[k] + 1 : 0;
            const int b = labels[cell + (long long)(nx - c[k]) * st[k]];
            const int ra = seed_cell[3 * a + k];
            if (b != a) {
                set_pair_bit(bits, words_per_row, a, b);
                set_pair_bit(bits, words_per_row, b, a);
                atomicMax(&bb[6 * a + 3 + k], offset_from(c[k], ra, N[k]));
                atomicMin(&bb[6 * b + k], offset_from(nx, seed_cell[3 * b + k], N[k]));
            } else {
                int cut = ra + N[k] / 2 + 1;          // the first cell past half a period
                if (cut >= N[k]) cut -= N[k];
                if (nx == cut) {
                    atomicMax(&bb[6 * a + 3 + k], offset_from(c[k], ra, N[k]));
                    atomicMin(&bb[6 * a + k], offset_from(nx, ra, N[k]));
                }
            }
        }
    }
}

__global__ void k_init_boxes(Domain D, int G, const int* __restrict__ bb, const double* __restrict__ seeds,
                             Box* __restrict__ cur) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G; i += gridDim.x * blockDim.x) {
        Box b{};
        if (bb[6 * i] > bb[6 * i + 3]) {       // no cell: extinct from the start
            cur[i] = b;
            continue;
        }
        int N[3] = {D.nx, D.ny, D.nz};
        int o[3], n[3];
        for (int a = 0; a < 3; ++a) {
            if (N[a] == 1) { o[a] = 0; n[a] = 1; continue; }
            int r = pmod((int)rint(seeds[3 * i + a]), N[a]);
            int lo = bb[6 * i + a], hi = bb[6 * i + 3 + a];
            int ext = hi - lo + 1 + 2 * D.halo;
            n[a] = ext < N[a] ? ext : N[a];
            o[a] = pmod(r + lo - D.halo, N[a]);
        }
        b.ox = o[0]; b.oy = o[1]; b.oz = o[2];
        b.nx = n[0]; b.ny = n[1]; b.nz = n[2];
        cur[i] = b;
    }
}

// neighbours of a grain the initial functions take (more: refused)
constexpr int kSdfNb = 512;

__device__ __forceinline__ double power_dist(const double* p, const double* s, double w, const double* N,
                                             double& e0, double& e1, double& e2) {
    e0 = min_image(__dsub_rn(p[0], s[0]), N[0]);
    e1 = min_image(__dsub_rn(p[1], s[1]), N[1]);
    e2 = min_image(__dsub_rn(p[2], s[2]), N[2]);
    return __dsub_rn(__dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)), __dmul_rn(e2, e2)), w);
}

// For cell p with displacement a = p - s_i (minimum image) and neighbour j
// with D = s_i - s_j (minimum image), p - s_j = a + D up to one period per
// axis; with d = (p - s_j) - a the bisector distance is
// (d . (d + 2a) - (w_j - w_i)) / (2 |d|).  Where p - s_j needs no other
// period than D's (every cell of a box small against the domain), d = D and
// the distance is affine in a: n . a + c with n = D / |D| and
// c = |D| / 2 - (w_j - w_i) / (2 |D|), both per pair, computed once per grain
// in FP64.  An FP32 pass over the neighbours (3 FMAs each) finds the
// candidates within a bound of its rounding error of the minimum; those are
// evaluated in FP64 (3 FMAs): the definition's value
// ((p - s_j)^2 - w_j - (p - s_i)^2 + w_i) / (2 |d|) up to FP64 rounding, far
// below the FP32 result's half unit.  Cells where the image of s_j or of s_i
// is too close to call in FP32 take the general form with a per-cell image.
struct SdfPair {
    double n0, n1, n2, c;
};

__device__ __forceinline__ float two_sum_f(float a, float b, float& e) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

constexpr int kSdfThreads = 256;

// A CTA per item (box, first of `groups` groups of four cells along x).  One
// CTA a box leaves a large grain's box (hundreds of neighbours, 10^6 cells) on
// one SM: 130 ms of a 160^3 lognormal start on GB300, 176 ms at 512^3; the
// items below take 3.6 and 15.5 ms, bound by the screening's issue slots.
//
// Where every cell of the box sees the seed and every neighbour through one
// image (any box small against the domain) the values are affine throughout
// (`fast`): a thread screens a group of four cells at once, the two smallest
// FP32 values of each kept in registers (six instructions a cell and neighbour).
// With the smallest one clear of the other by twice the FP32 error bound E, its
// value is taken in double-float arithmetic (pairs of FP32, about 2^-47 of the
// terms' size), and it is the FP64 value's FP32 rounding unless a rounding
// boundary lies within that error; then, and where E does not separate the two,
// the cell takes the general FP64 form (`slow_cell`), as every cell of a box
// without `fast` does.  FP64 for every cell's winner kept the FP64 pipe busy:
// 9.6 ms at 256^3 / 5000 grains, against 2.00 ms.
__global__ void __launch_bounds__(kSdfThreads)
k_sdf(Domain D, const int2* __restrict__ items, int groups, const Box* __restrict__ boxes,
      const double* __restrict__ seeds, const double* __restrict__ weights, const unsigned* __restrict__ bits,
      long long words_per_row, float* __restrict__ X, int* __restrict__ IDF, int* __restrict__ status) {
    __shared__ int s_nb[kSdfNb];
    __shared__ float4 s_d[kSdfNb];          // D = s_i - s_j (minimum image), w_j - w_i
    __shared__ float4 s_f[kSdfNb];          // n and c in FP32
    __shared__ float4 s_l[kSdfNb];          // what FP32 leaves of them
    __shared__ SdfPair s_p[kSdfNb];         // n and c in FP64
    __shared__ int s_warp[kSdfThreads / 32];
    __shared__ float s_cmax;
    const int i = items[blockIdx.x].x;
    const Box b = boxes[i];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // the neighbours in ascending order: a word of the bit row per thread, its
    // bits placed by a block-wide prefix of the counts
    int cnt = 0;
    for (long long w0 = 0; w0 < words_per_row; w0 += kSdfThreads) {
        unsigned m = w0 + t < words_per_row ? bits[(long long)i * words_per_row + w0 + t] : 0u;
        const int own = __popc(m);
        int pre = own;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, pre, k);
            if (lane >= k) pre += v;
        }
        if (lane == 31) s_warp[warp] = pre;
        __syncthreads();
        int at = cnt + pre - own, total = 0;
#pragma unroll
        for (int k = 0; k < kSdfThreads / 32; ++k) {
            if (k < warp) at += s_warp[k];
            total += s_warp[k];
        }
        for (; m; m &= m - 1, ++at)
            if (at < kSdfNb) s_nb[at] = (int)((w0 + t) * 32 + __ffs(m) - 1);
        cnt += total;
        __syncthreads();
    }
    if (cnt > kSdfNb) {
        if (t == 0) atomicExch(status, -8);
        cnt = kSdfNb;
    }
    if (t == 0) s_cmax = 0.0f;
    __syncthreads();
    const double si[3] = {seeds[3 * i], seeds[3 * i + 1], seeds[3 * i + 2]};
    const double wi = weights ? weights[i] : 0.0;
    const double Nd[3] = {(double)D.nx, (double)D.ny, (double)D.nz};
    const float Nf[3] = {(float)D.nx, (float)D.ny, (float)D.nz};
    const int Ni[3] = {D.nx, D.ny, D.nz};
    const int o[3] = {b.ox, b.oy, b.oz};
    const int bn[3] = {b.nx, b.ny, b.nz};
    // the box's cells as consecutive integers q = shift + l whose displacement
    // q - s_i stays within half a period (fast), its first and last values
    int shift[3];
    double first[3], last[3];
    float asum = 0.0f, ssum = 0.0f;
    bool fast = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        shift[a] = o[a];
        const double d0 = (double)o[a] - si[a];
        if (d0 > 0.5 * Nd[a]) shift[a] -= Ni[a];
        else if (d0 < -0.5 * Nd[a]) shift[a] += Ni[a];
        first[a] = (double)shift[a] - si[a];
        last[a] = first[a] + (double)(bn[a] - 1);
        fast = fast && first[a] > -0.5 * Nd[a] + 2e-2 && last[a] < 0.5 * Nd[a] - 2e-2 && Ni[a] < (1 << 22);
        asum += (float)fmax(fabs(first[a]), fabs(last[a]));
        ssum += fabsf((float)si[a]);
    }
    for (int k = t; k < cnt; k += kSdfThreads) {
        const int j = s_nb[k];
        const double wj = weights ? weights[j] : 0.0;
        const double d0 = min_image(si[0] - seeds[3 * j], Nd[0]), d1 = min_image(si[1] - seeds[3 * j + 1], Nd[1]),
                     d2 = min_image(si[2] - seeds[3 * j + 2], Nd[2]);
        const double dd[3] = {d0, d1, d2};
        s_d[k] = make_float4((float)d0, (float)d1, (float)d2, (float)(wj - wi));
        const double len = sqrt(fma(d0, d0, fma(d1, d1, d2 * d2)));
        SdfPair q;
        q.n0 = d0 / len;
        q.n1 = d1 / len;
        q.n2 = d2 / len;
        q.c = 0.5 * len - 0.5 * (wj - wi) / len;
        s_p[k] = q;
        const float4 f = make_float4((float)q.n0, (float)q.n1, (float)q.n2, (float)q.c);
        s_f[k] = f;
        s_l[k] = make_float4((float)(q.n0 - (double)f.x), (float)(q.n1 - (double)f.y), (float)(q.n2 - (double)f.z),
                             (float)(q.c - (double)f.w));
        // one image of the neighbour's seed for every cell of the box
#pragma unroll
        for (int a = 0; a < 3; ++a)
            fast = fast && fabs(first[a] + dd[a]) < 0.5 * Nd[a] - 2e-2 && fabs(last[a] + dd[a]) < 0.5 * Nd[a] - 2e-2;
        fast = fast && fabsf(f.w) < 1e6f;
        atomicMax(reinterpret_cast<int*>(&s_cmax), __float_as_int(fabsf(f.w)));
    }
    fast = __syncthreads_and(fast);
    const float sif[3] = {(float)si[0], (float)si[1], (float)si[2]};
    const float nmax = fmaxf(Nf[0], fmaxf(Nf[1], Nf[2]));
    const int ps = plane_stride(b.nx, b.ny);
    const double eps = (double)D.eps;

    // the general form at the box's cell l (local coordinates): value and neighbour
    auto slow_cell = [&](const int (&l)[3], int& arg) {
        // the cell's global coordinates g and its displacement from s_i: the
        // image decided in FP32 (g - (float)s_i is exact), FP64 only for the value
        int g[3], sh[3];
        float af[3];
        bool amb = false;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            int gc = o[c] + l[c];
            if (gc >= Ni[c]) gc -= Ni[c];
            g[c] = gc;
            const float raw = (float)gc - sif[c];
            const float h = 0.5f * Nf[c];
            amb |= fabsf(fabsf(raw) - h) < 1e-2f;
            sh[c] = raw > h ? -Ni[c] : (raw < -h ? Ni[c] : 0);
            af[c] = raw + (float)sh[c];
        }
        double a0, a1, a2;
        if (amb) {
            const double p[3] = {(double)g[0], (double)g[1], (double)g[2]};
            power_dist(p, si, wi, Nd, a0, a1, a2);
            af[0] = (float)a0;
            af[1] = (float)a1;
            af[2] = (float)a2;
        } else {
            a0 = __dsub_rn((double)(g[0] + sh[0]), si[0]);
            a1 = __dsub_rn((double)(g[1] + sh[1]), si[1]);
            a2 = __dsub_rn((double)(g[2] + sh[2]), si[2]);
        }
        const float as = fabsf(af[0]) + fabsf(af[1]) + fabsf(af[2]);
        // whether neighbour k's image for this cell is D's (then the affine form
        // holds); near half a period the general form decides
        auto affine = [&](const float4& dk) {
            bool ok = !amb;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float v = af[c] + (c == 0 ? dk.x : (c == 1 ? dk.y : dk.z));
                ok &= fabsf(v) < 0.5f * Nf[c] - 1e-2f;
            }
            return ok;
        };
        auto screen = [&](int k, float& v, float& err) {
            const float4 dk = s_d[k];
            if (affine(dk)) {
                const float4 f = s_f[k];
                v = fmaf(f.x, af[0], fmaf(f.y, af[1], fmaf(f.z, af[2], f.w)));
                // rounding of s_i, n and c to FP32 and of the three FMAs
                err = 2.4e-7f * (3.0f * nmax + 2.0f * as + 2.0f * fabsf(f.w) + 4.0f);
                return;
            }
            const float dd[3] = {dk.x, dk.y, dk.z};
            float num = -dk.w, den = 0.0f;
            bool near_half = false;                            // image choice too close to call in FP32
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float u = af[c] + dd[c];                 // p - s_j before wrapping
                near_half |= fabsf(fabsf(u) - 0.5f * Nf[c]) < 1e-2f;
                const float dc = u > 0.5f * Nf[c] ? dd[c] - Nf[c] : (u < -0.5f * Nf[c] ? dd[c] + Nf[c] : dd[c]);
                num = fmaf(dc, fmaf(2.0f, af[c], dc), num);
                den = fmaf(dc, dc, den);
            }
            const float rinv = rsqrtf(den);
            v = 0.5f * num * rinv;
            // about 64 FP32 ulps of every term of num / (2 |d|), and of v
            err = near_half || amb ? FLT_MAX
                                   : 4e-6f * (0.5f * den * rinv + as + 0.5f * fabsf(dk.w) * rinv + fabsf(v) + 1.0f);
        };
        // the screening's upper bound U of the minimum, then the exact
        // evaluation of the neighbours that may be it, in neighbour order (which
        // decides ties, as in the definition)
        float U = FLT_MAX;
        for (int k = 0; k < cnt; ++k) {
            float v, err;
            screen(k, v, err);
            U = fminf(U, v + err);
        }
        double best = DBL_MAX;
        arg = -1;
        for (int k = 0; k < cnt; ++k) {
            float v, err;
            screen(k, v, err);
            if (!(v - err <= U)) continue;
            const int j = s_nb[k];
            double ve;
            if (affine(s_d[k])) {
                const SdfPair q = s_p[k];
                ve = fma(q.n0, a0, fma(q.n1, a1, fma(q.n2, a2, q.c)));
            } else {
                const double p[3] = {(double)g[0], (double)g[1], (double)g[2]};
                const double* sj = seeds + 3 * j;
                const double d0 = __dsub_rn(min_image(__dsub_rn(p[0], sj[0]), Nd[0]), a0);
                const double d1 = __dsub_rn(min_image(__dsub_rn(p[1], sj[1]), Nd[1]), a1);
                const double d2 = __dsub_rn(min_image(__dsub_rn(p[2], sj[2]), Nd[2]), a2);
                double num = fma(d0, fma(2.0, a0, d0), fma(d1, fma(2.0, a1, d1), d2 * fma(2.0, a2, d2)));
                if (weights) num -= weights[j] - wi;
                ve = num * (0.5 * rsqrt(fma(d0, d0, fma(d1, d1, d2 * d2))));
            }
            if (ve < best) { best = ve; arg = j; }
        }
        return (float)(best == DBL_MAX ? eps : (best < -eps ? -eps : (best > eps ? eps : best)));
    };

    // Error bounds, with A = asum >= |n . a|, S = ssum = the sum of |s_i|, C =
    // s_cmax >= |c| and u = 2^-24 (half an FP32 ulp, relative).
    // Screening: n, a and c rounded (u (2 A + C)), three FMAs (3 u (A + C)); E
    // is twice that.  a is the displacement from the FP64 seed, rounded once:
    // from the seed rounded to FP32, as u S alone exceeds E in wide domains.
    // Double-float, in u^2: s_i beyond 48 bits and its low part's difference
    // (A + 2 S), n and c beyond 48 bits (A + C), the product of the low parts
    // (A), the products' rests (each u |n a|) added up (2 A), six FMAs on at most
    // 3 u A (18 A), the sums' rests added up (5 A + C), c's low part added (3 A
    // + 2 C) and the total (6 A + 2 C), the test's own rest + edd (A + C), and
    // the FP64 form's roundings (below A / 4 + C / 8): 39 A + 2 S + 8 C.
    const float E = 1.2e-7f * (5.0f * asum + 4.0f * s_cmax + 1.0f);
    const float edd = 3.6e-15f * (39.0f * asum + 2.0f * ssum + 8.0f * s_cmax);
    float s_hi[3], s_lo[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        s_hi[a] = (float)si[a];
        s_lo[a] = (float)(si[a] - (double)s_hi[a]);
    }
    const int ngx = (b.nx + 3) >> 2;
    const int per_plane = ngx * b.ny;
    const int g0 = items[blockIdx.x].y, g1 = min(per_plane * b.nz, g0 + groups);
    for (int q = g0 + t; q < g1; q += kSdfThreads) {
        const int z = q / per_plane, rem = q - z * per_plane;
        const int y = rem / ngx, x0 = 4 * (rem - y * ngx);
        const long long off = b.off + (long long)z * ps + (long long)y * b.nx + x0;
        if (!fast) {
            for (int u = 0; u < min(4, b.nx - x0); ++u) {
                const int l[3] = {x0 + u, y, z};
                int arg;
                X[off + u] = slow_cell(l, arg);
                if (IDF) IDF[off + u] = arg;
            }
            continue;
        }
        // displacements a = (shift + l) - s_i as pairs (the y and z ones shared)
        float ah[3], al[3], a0h[4], a0l[4];
#pragma unroll
        for (int a = 1; a < 3; ++a) {
            float e;
            const float d = two_sum_f((float)(shift[a] + (a == 1 ? y : z)), -s_hi[a], e);
            ah[a] = two_sum_f(d, e - s_lo[a], al[a]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float e;
            const float d = two_sum_f((float)(shift[0] + x0 + u), -s_hi[0], e);
            a0h[u] = two_sum_f(d, e - s_lo[0], a0l[u]);
        }
        float v1[4], v2[4];
        int k1[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { v1[u] = v2[u] = FLT_MAX; k1[u] = 0; }
        for (int k = 0; k < cnt; ++k) {
            const float4 f = s_f[k];
            const float row = fmaf(f.y, ah[1], fmaf(f.z, ah[2], f.w));
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float v = fmaf(f.x, a0h[u], row);
                k1[u] = v < v1[u] ? k : k1[u];
                v2[u] = fminf(v2[u], fmaxf(v1[u], v));
                v1[u] = fminf(v1[u], v);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (x0 + u >= b.nx) break;
            float out = D.eps;
            int arg = -1;
            if (cnt > 0) {
                const float4 f = s_f[k1[u]], lo = s_l[k1[u]];
                // n . a + c: products exact as pairs, their sum by two-sums
                const float p0 = f.x * a0h[u], p1 = f.y * ah[1], p2 = f.z * ah[2];
                float e = fmaf(f.x, a0h[u], -p0) + fmaf(f.y, ah[1], -p1) + fmaf(f.z, ah[2], -p2);
                e = fmaf(f.x, a0l[u], fmaf(lo.x, a0h[u], e));
                e = fmaf(f.y, al[1], fmaf(lo.y, ah[1], e));
                e = fmaf(f.z, al[2], fmaf(lo.z, ah[2], e));
                float r0, r1, r2;
                float sum = two_sum_f(p0, p1, r0);
                sum = two_sum_f(sum, p2, r1);
                sum = two_sum_f(sum, f.w, r2);
                e += lo.w + (r0 + r1 + r2);
                float rest;
                const float hi = two_sum_f(sum, e, rest);
                // the nearest FP32 number of every value within edd
                const bool sure = v2[u] > v1[u] + 2.0f * E && __fadd_rn(hi, rest + edd) == hi &&
                                  __fadd_rn(hi, rest - edd) == hi;
                if (sure) {
                    out = fminf(fmaxf(hi, -D.eps), D.eps);
                    arg = s_nb[k1[u]];
                } else {
                    const int l[3] = {x0 + u, y, z};
                    out = slow_cell(l, arg);
                }
            }
            X[off + u] = out;
            if (IDF) IDF[off + u] = arg;
        }
    }
}

cudaError_t launch_init(const Domain& D, int G, const SeedBins& bins, const double* d_seeds, const double* d_weights,
                        int* d_labels, unsigned* d_bits, long long words_per_row, int* d_bb, int* d_seed_cell,
                        Box* d_cur, cudaStream_t s) {
    const long long ncell = (long long)D.nx * D.ny * D.nz;
    const int tx = D.dim == 3 ? 8 : 32, ty = D.dim == 3 ? 8 : 16, tz = D.dim == 3 ? 8 : 1;
    const int ntx = (D.nx + tx - 1) / tx, nty = (D.ny + ty - 1) / ty, ntz = (D.nz + tz - 1) / tz;
    k_labels<<<ntx * nty * ntz, kLabelThreads, 0, s>>>(D, G, bins, d_seeds, d_weights, d_labels, tx, ty, tz, ntx, nty);
    cudaError_t e = cudaMemsetAsync(d_bits, 0, (size_t)G * words_per_row * 4, s);
    if (e != cudaSuccess) return e;
    long long gs = (ncell + 255) / 256;
    if (gs > 65535 * 8) gs = 65535 * 8;
    k_bbox_init<<<(G + 255) / 256, 256, 0, s>>>(D, G, d_seeds, d_bb, d_seed_cell);
    k_label_faces<<<(int)gs, 256, 0, s>>>(D, d_labels, d_seed_cell, d_bits, words_per_row, d_bb);
    k_init_boxes<<<(G + 255) / 256, 256, 0, s>>>(D, G, d_bb, d_seeds, d_cur);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// initialisation from a label field
// ---------------------------------------------------------------------------
// Per grain and axis, the positions holding one of its cells, as bits
// (words of 32 positions per (grain, axis)).
__global__ void k_label_occupancy(Domain D, const int* __restrict__ labels, unsigned* __restrict__ occ, int words) {
    const long long ncell = (long long)D.nx * D.ny * D.nz;
    const int N[3] = {D.nx, D.ny, D.nz};
    for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < ncell;
         cell += (long long)gridDim.x * blockDim.x) {
        const int c[3] = {(int)(cell % D.nx), (int)((cell / D.nx) % D.ny), (int)(cell / ((long long)D.nx * D.ny))};
        const long long i = labels[cell];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (N[a] > 1) atomicOr(&occ[(i * 3 + a) * words + (c[a] >> 5)], 1u << (c[a] & 31));
    }
}

// Grain i's box from its label cells: per axis the shortest cyclic interval
// holding every occupied position -- the complement of the longest run of
// empty positions, the first such run (smallest start) on ties -- grown by
// the halo and capped at the axis; no cell: extinct.
// A warp per grain: its lanes look for the starts of empty runs and follow
// them word by word (one thread per grain, bit by bit, took 0.6 ms on a
// 149 x 97 x 61 domain on GB300).
__global__ void __launch_bounds__(128)
k_label_boxes(Domain D, int G, const unsigned* __restrict__ occ, int words, Box* __restrict__ cur) {
    const int N[3] = {D.nx, D.ny, D.nz};
    const int lane = threadIdx.x & 31;
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= G) return;                                       // uniform across the warp
    const unsigned* ox = occ + ((long long)i * 3) * words;
    bool any = false;
    for (int w = lane; w < words; w += 32) any = any || ox[w] != 0u;
    Box b{};
    if (!__any_sync(0xffffffffu, any)) {
        if (lane == 0) cur[i] = b;
        return;
    }
    int o[3], n[3];
    for (int a = 0; a < 3; ++a) {
        const int na = N[a];
        if (na == 1) { o[a] = 0; n[a] = 1; continue; }
        const unsigned* bits = occ + ((long long)i * 3 + a) * words;
        auto at = [&](int p) { return (bits[p >> 5] >> (p & 31)) & 1u; };
        // the longest run, the smallest start on ties, as one key
        unsigned long long best = 0;
        for (int p = lane; p < na; p += 32) {
            if (at(p) || !at(p == 0 ? na - 1 : p - 1)) continue;   // not the first empty position of a run
            int len = 0;
            for (int q = p; len < na;) {                      // empty positions from p on, a word at a time
                const int room = min(32 - (q & 31), na - q);  // positions of this word
                unsigned m = bits[q >> 5] >> (q & 31);
                if (room < 32) m |= 1u << room;               // ends the search at the word's (axis') end
                const int free_ = m ? __ffs(m) - 1 : 32;
                len += free_;
                if (free_ < room) break;
                q = q + room >= na ? 0 : q + room;
            }
            len = min(len, na);
            const unsigned long long key = ((unsigned long long)len << 32) | (0xffffffffu - (unsigned)p);
            best = key > best ? key : best;
        }
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, k);
            best = v > best ? v : best;
        }
        int start = 0, length = na;                           // every position held
        if (best) {
            const int best_len = (int)(best >> 32), best_start = (int)(0xffffffffu - (unsigned)(best & 0xffffffffu));
            start = (best_start + best_len) % na;
            length = na - best_len;
        }
        n[a] = length + 2 * D.halo < na ? length + 2 * D.halo : na;
        o[a] = pmod(start - D.halo, na);
    }
    b.ox = o[0]; b.oy = o[1]; b.oz = o[2];
    b.nx = n[0]; b.ny = n[1]; b.nz = n[2];
    if (lane == 0) cur[i] = b;
}

// The starting function before the re-initialisation: +1/2 on the grain's
// label cells and -1/2 on the other cells of its box (`cur` layout, FP32).
__global__ void k_label_phi(Domain D, const Box* __restrict__ cur, const int* __restrict__ labels,
                            float* __restrict__ Z) {
    const int i = blockIdx.x;
    const Box b = cur[i];
    if (b.nx <= 0) return;
    const int ps = plane_stride(b.nx, b.ny);
    const int A = b.nx * b.ny;
    const long long n = (long long)A * b.nz;
    for (long long k = blockIdx.y * blockDim.x + threadIdx.x; k < n; k += gridDim.y * blockDim.x) {
        const int z = (int)(k / A), rem = (int)(k - (long long)z * A);
        const int y = rem / b.nx, x = rem - y * b.nx;
        const long long g = ((long long)pmod(b.oz + z, D.nz) * D.ny + pmod(b.oy + y, D.ny)) * D.nx + pmod(b.ox + x, D.nx);
        Z[b.off + (long long)z * ps + rem] = labels[g] == i ? 0.5f : -0.5f;
    }
}

cudaError_t launch_label_boxes(const Domain& D, int G, const int* d_labels, unsigned* d_occ, int words, Box* d_cur,
                               cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(d_occ, 0, (size_t)G * 3 * words * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const long long ncell = (long long)D.nx * D.ny * D.nz;
    long long gs = (ncell + 255) / 256;
    if (gs > 65535 * 8) gs = 65535 * 8;
    k_label_occupancy<<<(int)gs, 256, 0, s>>>(D, d_labels, d_occ, words);
    k_label_boxes<<<(G + 3) / 4, 128, 0, s>>>(D, G, d_occ, words, d_cur);
    return cudaGetLastError();
}

cudaError_t launch_label_phi(const Domain& D, int G, const Box* d_cur, const int* d_labels, float* Z, cudaStream_t s) {
    k_label_phi<<<dim3(G, 8), 256, 0, s>>>(D, d_cur, d_labels, Z);
    return cudaGetLastError();
}

cudaError_t launch_sdf(const Domain& D, const int2* d_items, int n_items, int groups, const Box* d_cur,
                       const double* d_seeds, const double* d_weights, const unsigned* d_bits, long long words_per_row,
                       float* X, int* IDF, int* d_status, cudaStream_t s) {
    if (n_items > 0)
        k_sdf<<<n_items, kSdfThreads, 0, s>>>(D, d_items, groups, d_cur, d_seeds, d_weights, d_bits, words_per_row, X,
                                              IDF, d_status);
    return cudaGetLastError();
}

}  // namespace lsgg
