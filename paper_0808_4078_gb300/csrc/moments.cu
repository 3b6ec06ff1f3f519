// moments.cu -- coarse-grained moment recorder: the inputs and label parts of the learned
// collision closure, per coarse cell (bx x by transverse cells x the whole z extent).
//
// The paper closes by conjecturing that the collisional drag on the return current could be
// written through the local plasma state; the quantities recorded here are the reading of that
// closure's inputs and label (rows in pic.h: densities, mean u_z, momentum variances of beam and
// background, electrostatic fluctuation energy W_ES, and the background's mean particle force
// against the force of the coarse-grained fields).
//
// Two passes over the particles: the first sums w and w u per coarse cell and species, the
// second the centred second moments w (u - <u>)^2 (variances of a cold beam are ~1e-6 of <u>^2,
// far below what <u^2> - <u>^2 resolves) and the background's force and velocity sums.  Sums are
// int64 fixed point (2^36 per unit; a coarse cell's sum of |w u| must stay below 2^27),
// accumulated per CTA and added with one atomic per quantity, so they do not depend on the order
// of the particles; the field column sums are FP64 in a fixed order.  The record is bitwise
// reproducible.
#include "pic_internal.cuh"

namespace pic {

// psum rows: pass 1 per species w, w ux, w uy, w uz (rows 4 s + 0..3); pass 2 per species
// w (ux - <ux>)^2, w (uy - <uy>)^2, w (uz - <uz>)^2 (rows 8 + 3 s + 0..2), then the background's
// w Fz, w vx, w vy, w vz (rows 14..17).
constexpr int MOM_PSUMS = 18;
constexpr int MOM_COLS = 4;                 // per column: W_ES mean, mean Ez, mean Bx, mean By
constexpr double MOM_FIX = 68719476736.0;   // 2^36

namespace {

constexpr int NT = 256;

struct MomArgs {
    Args a;
    int run;
    int bx, by;        // coarse block in cells
    int zc;            // z layers per CTA
    int ncx, ncy;      // coarse cells per axis
    float q_bg;        // background charge
    float nu_bg;       // background Krook rate
    long long* psum;   // [MOM_PSUMS][nc]
    float* meanbuf;    // [nc][12]: coarse means of pass 1 as FP32 pairs
    double* col;       // [MOM_COLS][nx * ny]
    float* out;        // [PIC_MOM_ROWS][nc]
};

__device__ __forceinline__ int wrap1(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// 2D: component c of E (c < 3) or B at the particle, CIC on its Yee lattice.
__device__ __forceinline__ float gather_comp(const RunDev& R, int c, int cx, int cy, float ox, float oy) {
    // half-shifted axes of each component: Ex x, Ey y, Bx y, By x, Bz x and y (bit c set: component c
    // is half-shifted along the axis; c = Ex Ey Ez Bx By Bz)
    const bool hx = (0x31 >> c) & 1, hy = (0x2A >> c) & 1;
    const float* F = c < 3 ? R.E[c] : R.B[c - 3];
    const float xs = hx ? ox - 0.5f : ox, ys = hy ? oy - 0.5f : oy;
    const int i0 = xs < 0.f ? -1 : 0, j0 = ys < 0.f ? -1 : 0;
    const float ax = xs - (float)i0, ay = ys - (float)j0;
    float v = 0.f;
    for (int dj = 0; dj < 2; ++dj)
        for (int di = 0; di < 2; ++di) {
            // neighbours within one cell of the particle's: one conditional wrap
            const int gi = wrap1(cx + i0 + di, R.nx), gj = wrap1(cy + j0 + dj, R.ny);
            v += (di ? ax : 1.f - ax) * (dj ? ay : 1.f - ay) * F[(size_t)gj * R.nx + gi];
        }
    return v;
}

// 3D: Ez, Bx, By at the particle, CIC on their Yee lattices (Ez half-shifted in z, Bx in y and z, By in
// x and z), by interpolation along x, y, z in turn with explicit roundings: particles in slots and
// spilled ones, whose fields come from shared and from global memory, get the same bits (which
// particles spill depends on the order of atomics).  at(c, i, j, k): Ez (c = 0), Bx or By of the cell
// (i, j, k) away from the particle's.
template <class At>
__device__ __forceinline__ void gather_force3(const At& at, const float o[3], float f[3]) {
    // per axis: weight of the upper point on the nodes and on the half-shifted lattice, whose lower
    // point is at offset bh
    float wh[3];
    int bh[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float h = __fsub_rn(o[d], 0.5f);
        bh[d] = h < 0.f ? -1 : 0;
        wh[d] = h < 0.f ? __fadd_rn(h, 1.f) : h;
    }
    auto lerp = [](float t, float lo, float hi) { return __fmaf_rn(t, hi, __fmul_rn(__fsub_rn(1.f, t), lo)); };
    auto interp = [&](int c, int i, int j, int k, float tx, float ty, float tz) {
        const float a00 = lerp(tx, at(c, i, j, k), at(c, i + 1, j, k));
        const float a10 = lerp(tx, at(c, i, j + 1, k), at(c, i + 1, j + 1, k));
        const float a01 = lerp(tx, at(c, i, j, k + 1), at(c, i + 1, j, k + 1));
        const float a11 = lerp(tx, at(c, i, j + 1, k + 1), at(c, i + 1, j + 1, k + 1));
        return lerp(tz, lerp(ty, a00, a10), lerp(ty, a01, a11));
    };
    f[0] = interp(0, 0, 0, bh[2], o[0], o[1], wh[2]);
    f[1] = interp(1, 0, bh[1], bh[2], o[0], wh[1], wh[2]);
    f[2] = interp(2, bh[0], 0, bh[2], wh[0], o[1], wh[2]);
}

// Pass-2 terms of a background particle of weight w in fields f = Ez, Bx, By: w Fz, w vx, w vy, w vz.
__device__ __forceinline__ void force_terms(float w, float q_bg, const float f[3], const float u[3], float t[4]) {
    const float ig = __fdiv_rn(1.0f, __fsqrt_rn(__fmaf_rn(u[2], u[2], __fmaf_rn(u[1], u[1], __fmaf_rn(u[0], u[0], 1.0f)))));
    const float vx = __fmul_rn(u[0], ig), vy = __fmul_rn(u[1], ig), vz = __fmul_rn(u[2], ig);
    t[0] = __fmul_rn(w, __fmul_rn(q_bg, __fmaf_rn(-vy, f[1], __fmaf_rn(vx, f[2], f[0]))));
    t[1] = __fmul_rn(w, vx);
    t[2] = __fmul_rn(w, vy);
    t[3] = __fmul_rn(w, vz);
}

// v 2^36 rounded to the nearest int64 (ties to even) through 32-bit conversions only: the 64-bit
// ones run on the FP64 unit, which this part has little of.  With a = |v| 2^36 (an exact
// scaling), hi = floor(a 2^-32) and a - hi 2^32 are exact in FP32 (either hi = 0 or
// ulp(a) >= 2^9), so hi 2^32 + rint(a - hi 2^32) = rint(a); valid for |v| 2^36 < 2^62.
__device__ __forceinline__ long long fx(float v) {
    const float a = fabsf(v) * 68719476736.0f;
    const float hi = floorf(a * 2.3283064365386963e-10f);
    const unsigned lo = __float2uint_rn(a - hi * 4294967296.0f);
    const long long r = (long long)__float2uint_rz(hi) * 4294967296LL + (long long)lo;
    return v < 0.0f ? -r : r;
}

// Mean of a coarse cell as an unevaluated FP32 sum hi + lo, so that u - mean keeps FP32
// relative accuracy for the small deviations of a cold beam: u - hi is exact when u is within a
// factor 2 of hi (Sterbenz), then lo is subtracted.
struct Mean2 { float hi[2][3], lo[2][3]; };

// Add one particle to the thread's sums (FP32 arithmetic, exact fixed-point sums): pass 1 first
// moments, pass 2 centred second moments about its coarse cell's mean and the background force
// and velocity.
// Rows of each pass: pass 1 rows [0, 8), pass 2 rows [8, 18); acc holds the pass's rows only.
template <int PASS> struct PassRows;
template <> struct PassRows<1> { static constexpr int base = 0, n = 8; };
template <> struct PassRows<2> { static constexpr int base = 8, n = 10; };

template <int PASS, bool D3>
__device__ __forceinline__ void add_particle(const MomArgs& m, const RunDev& R, int s, float w,
                                             const Mean2& mean, int cx, int cy, int cz, float ox,
                                             float oy, float oz, float ux, float uy, float uz,
                                             long long* acc) {
    const float du[3] = {ux, uy, uz};
    if (PASS == 1) {
        acc[4 * s] += fx(w);
#pragma unroll
        for (int d = 0; d < 3; ++d) acc[4 * s + 1 + d] += fx(__fmul_rn(w, du[d]));
        return;
    }
    acc -= 8;   // pass-2 rows are numbered from 8
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float e = __fsub_rn(__fsub_rn(du[d], mean.hi[s][d]), mean.lo[s][d]);
        acc[8 + 3 * s + d] += fx(__fmul_rn(w, __fmul_rn(e, e)));
    }
    if (s == 1) {
        float f[3], t[4];
        if (D3) {
            const float o[3] = {ox, oy, oz};
            auto at = [&](int c, int i, int j, int k) {
                const float* F = c == 0 ? R.E[2] : R.B[c - 1];
                return F[((size_t)wrap1(cz + k, R.nz) * R.ny + wrap1(cy + j, R.ny)) * R.nx + wrap1(cx + i, R.nx)];
            };
            gather_force3(at, o, f);
        } else {
            for (int c = 0; c < 3; ++c) f[c] = gather_comp(R, 2 + c, cx, cy, ox, oy);
        }
        force_terms(w, m.q_bg, f, du, t);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[14 + k] += fx(t[k]);
    }
}

// Means <u> per species of each coarse cell from the pass-1 sums, computed once (FP64 divisions
// are costly on this part) and stored as FP32 pairs for pass 2: meanbuf[cc] = hi[6], lo[6].
__global__ void __launch_bounds__(NT) mom_means(const MomArgs m) {
    const long long nc = (long long)m.ncx * m.ncy;
    for (long long cc = blockIdx.x * (long long)NT + threadIdx.x; cc < nc; cc += (long long)gridDim.x * NT) {
        float* o = m.meanbuf + (size_t)cc * 12;
        for (int s = 0; s < 2; ++s) {
            const double sw = (double)m.psum[(size_t)(4 * s) * nc + cc];
            for (int d = 0; d < 3; ++d) {
                const double mu = sw > 0 ? (double)m.psum[(size_t)(4 * s + 1 + d) * nc + cc] / sw : 0.0;
                const float hi = (float)mu;
                o[3 * s + d] = hi;
                o[6 + 3 * s + d] = (float)(mu - (double)hi);
            }
        }
    }
}

__device__ __forceinline__ void coarse_means(const MomArgs& m, long long cc, Mean2& mean) {
    const float* o = m.meanbuf + (size_t)cc * 12;
    for (int s = 0; s < 2; ++s)
        for (int d = 0; d < 3; ++d) {
            mean.hi[s][d] = o[3 * s + d];
            mean.lo[s][d] = o[6 + 3 * s + d];
        }
}

// 2D (particles binned by cell): one CTA per (coarse cell, z chunk): a thread per fine cell, all its particles; one kernel per
// pass, each holding only its own sums (pass 2 with its field gathers runs 2 CTAs per SM without
// spilling, measured faster than 3 with spills).
template <int PASS>
__global__ void __launch_bounds__(NT, PASS == 1 ? 3 : 2) mom_particles(const MomArgs m) {
    constexpr int B = PassRows<PASS>::base, NR = PassRows<PASS>::n;
    __shared__ long long red[NT / 32][NR];
    const Args& a = m.a;
    const RunDev& R = a.runs[m.run];
    const int cc = blockIdx.x;
    Mean2 mean{};
    if (PASS == 2) coarse_means(m, cc, mean);
    const int X0 = (cc % m.ncx) * m.bx, Y0 = (cc / m.ncx) * m.by;
    const int per = m.bx * m.by;
    long long acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = 0;
    const int par = a.ctl->parity;
    for (int t = threadIdx.x; t < per * m.zc; t += NT) {
        const int col = t % per, lz = t / per;
        const int cx = X0 + col % m.bx, cy = Y0 + col / m.bx;
        const int cz = blockIdx.y * m.zc + lz;
        if (cz >= R.nz) continue;
        const long long g = R.cell_off + ((long long)cz * R.ny + cy) * R.nx + cx;
        for (int s = 0; s < a.nspecies && s < 2; ++s) {
            if (!R.sp[s].active) continue;
            const Slots& S = a.slot[s][par];
            const CellRange cr = cell_range(S, a.cap[s], a.cap_stay[s], g);
            const float w = R.sp[s].w;
            for (int k = 0; k < cr.n; ++k) {
                const size_t q = slot_elt(S, (long long)slot_of(g, a.cap[s], a.cap_stay[s], cr.ns, k));
                add_particle<PASS, false>(m, R, s, w, mean, cx, cy, cz, S.o[0][q], S.o[1][q], 0.f, S.u[0][q],
                                          S.u[1][q], S.u[2][q], acc);
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        long long v = acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < NR) {
        long long v = 0;
        for (int w = 0; w < NT / 32; ++w) v += red[w][threadIdx.x];
        if (v) atomicAdd((unsigned long long*)&m.psum[(size_t)(B + threadIdx.x) * m.ncx * m.ncy + cc], (unsigned long long)v);
    }
}

// 3D (particles binned by tile): one CTA per tile of the run, one particle per thread and round,
// consecutive lanes reading consecutive slots.  A tile covers at most 8 x 8 coarse columns; a
// particle adds its terms to its column's sums in shared memory.  A term of fixed point
// rint(v 2^36) is split at bit 20, sign (h 2^20 + l) with h, l >= 0, into two 32-bit words that are
// summed with native 32-bit reductions (64-bit shared atomics are several times slower), in several
// copies by lane so that the few columns of a tile do not serialise a warp.  At most FOLD particles
// are added to a word before the words move to the int64 sums, and terms of 2^40 or more go to
// those directly, so no word overflows; the sums are the same integers as fx()'s.  The three field
// components of the background's force come from a copy of the tile's fields in shared memory, and
// the column of a cell from a table (the block sizes are run-time divisors).
// 128 x 128 x 256 cells x 16 particles (67M): pass 1 1045 -> 417 us, pass 2 2440 -> 717 us against
// sorting each tile's indices by column and gathering the particles column by column (read 2 and 3
// times, uncoalesced) with 24 global field loads per background particle; it reads 16 and 28 B per
// particle (160 and 280 us at the copy bandwidth) and is bound by instruction issue.
constexpr int FOLD = 1024, MAXC = 64, MAXW = 8 * 8;   // MAXW: copies x columns

// Offset sums of the copies: column cl of copy k at (k ncl + cl) * STR, two words per row, an odd
// stride so that lanes of different copies and columns meet different banks.
__device__ __forceinline__ void add_word(int* p, int v) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("red.shared.add.s32 [%0], %1;\n" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void add_fixed(int* p, unsigned long long* wide, float v) {
    const float a = fabsf(v) * 68719476736.0f;                       // |v| 2^36
    if (a < 1099511627776.0f) {                                      // 2^40
        const int h = __float2int_rd(a * 9.5367431640625e-07f);      // floor(a 2^-20)
        const int l = __float2int_rn(fmaf(-1048576.0f, (float)h, a));   // exact difference, <= 2^20
        add_word(p, v < 0.0f ? -l : l);
        add_word(p + 1, v < 0.0f ? -h : h);
    } else {
        atomicAdd(wide, (unsigned long long)fx(v));
    }
}

template <int PASS>
__global__ void __launch_bounds__(NT) mom_tiles(const MomArgs m) {
    constexpr int B = PassRows<PASS>::base, NR = PassRows<PASS>::n, STR = 2 * NR + 1;
    constexpr int GX = 10, GY = 10, GZ = 6, GN = GX * GY * GZ;   // a tile of at most 8 x 8 x 4 cells + 1
    __shared__ int sums[2 * MAXW * STR];
    __shared__ unsigned char col[256];
    __shared__ float mean[PASS == 2 ? MAXC * 13 : 1];
    __shared__ float F[PASS == 2 ? 3 * GN : 1];
    const Args& a = m.a;
    const RunDev& R = a.runs[m.run];
    const long long T = R.work_off + blockIdx.x;
    const int t = blockIdx.x;
    const int x0 = (t % R.ntx) * a.tx, y0 = ((t / R.ntx) % R.nty) * a.ty, z0 = (t / (R.ntx * R.nty)) * a.tz;
    const int cx0 = x0 / m.bx, cy0 = y0 / m.by;
    const int ncxl = (x0 + a.tx - 1) / m.bx - cx0 + 1, ncyl = (y0 + a.ty - 1) / m.by - cy0 + 1;
    const int ncl = ncxl * ncyl;                     // <= 64: a tile is at most 8 cells wide
    const int copies = ncl <= 8 ? 8 : 2;             // 2 MAXW words per row at most
    const int lgx = __ffs(a.tx) - 1, lgy = __ffs(a.ty) - 1;   // tile sides are powers of two (the host checks)
    const int cells = a.tx * a.ty * a.tz;
    const long long nc = (long long)m.ncx * m.ncy;
    const int words = copies * ncl * STR;
    for (int i = threadIdx.x; i < words; i += NT) sums[i] = 0;
    for (int i = threadIdx.x; i < cells; i += NT)
        col[i] = (unsigned char)(((y0 + ((i >> lgx) & (a.ty - 1))) / m.by - cy0) * ncxl +
                                 ((x0 + (i & (a.tx - 1))) / m.bx - cx0));
    if (PASS == 2) {
        for (int i = threadIdx.x; i < ncl * 12; i += NT) {
            const int cl = i / 12;
            mean[cl * 13 + i - cl * 12] =
                m.meanbuf[((long long)(cy0 + cl / ncxl) * m.ncx + (cx0 + cl % ncxl)) * 12 + (i - cl * 12)];
        }
        for (int i = threadIdx.x; i < GN; i += NT) {
            const int rx = i % GX, ry = (i / GX) % GY, rz = i / (GX * GY);
            if (rx > a.tx + 1 || ry > a.ty + 1 || rz > a.tz + 1) continue;
            const size_t g = ((size_t)wrapi(z0 + rz - 1, R.nz) * R.ny + wrapi(y0 + ry - 1, R.ny)) * R.nx + wrapi(x0 + rx - 1, R.nx);
            F[i] = R.E[2][g];
            F[GN + i] = R.B[0][g];
            F[2 * GN + i] = R.B[1][g];
        }
    }
    __syncthreads();
    const int par = a.ctl->parity;
    const int copy = threadIdx.x % copies;
    const int every = FOLD / (NT / copies);          // rounds between folds
    // the words' sums to the int64 sums of the record, and cleared
    auto fold = [&]() {
        __syncthreads();
        for (int i = threadIdx.x; i < ncl * NR; i += NT) {
            const int cl = i / NR, k = i - cl * NR;
            long long v = 0;
            for (int c = 0; c < copies; ++c) {
                int* p = &sums[(c * ncl + cl) * STR + 2 * k];
                v += (long long)p[1] * 1048576 + p[0];
                p[0] = p[1] = 0;
            }
            if (PASS == 1 && k % 4 == 0) v *= fx(R.sp[k / 4].w);   // sum w: a count of equal weights

            const long long cc = (long long)(cy0 + cl / ncxl) * m.ncx + (cx0 + cl % ncxl);
            if (v) atomicAdd((unsigned long long*)&m.psum[(size_t)(B + k) * nc + cc], (unsigned long long)v);
        }
        __syncthreads();
    };
    int rounds = 0;
    for (int s = 0; s < a.nspecies && s < 2; ++s) {
        if (!R.sp[s].active) continue;
        const Slots& S = a.slot[s][par];
        const CellRange cr = cell_range(S, a.cap[s], a.cap_stay[s], T);
        const float w = R.sp[s].w;
        for (int r0 = 0; r0 < cr.n; r0 += NT) {
            const int i = r0 + threadIdx.x;
            if (i < cr.n) {
                const size_t q = slot_elt(S, (long long)slot_of(T, a.cap[s], a.cap_stay[s], cr.ns, i));
                const int lc = S.lc[q] & (cells - 1);
                const float u[3] = {S.u[0][q], S.u[1][q], S.u[2][q]};
                const int cl = col[lc];
                int* p = &sums[(copy * ncl + cl) * STR];
                unsigned long long* wide = (unsigned long long*)&m.psum[(size_t)B * nc +
                    (long long)(cy0 + cl / ncxl) * m.ncx + (cx0 + cl % ncxl)];
                if (PASS == 1) {
                    add_word(p + 8 * s, 1);
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        add_fixed(p + 8 * s + 2 + 2 * d, wide + (4 * s + 1 + d) * nc, __fmul_rn(w, u[d]));
                } else {
                    const float* mu = &mean[cl * 13 + 3 * s];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float e = __fsub_rn(__fsub_rn(u[d], mu[d]), mu[6 + d]);
                        add_fixed(p + 6 * s + 2 * d, wide + (3 * s + d) * nc, __fmul_rn(w, __fmul_rn(e, e)));
                    }
                    if (s == 1) {
                        const float o[3] = {S.o[0][q], S.o[1][q], S.o[2][q]};
                        const int lx = lc & (a.tx - 1), ly = (lc >> lgx) & (a.ty - 1), lz = lc >> (lgx + lgy);
                        const float* f0 = F + ((lz + 1) * GY + ly + 1) * GX + lx + 1;
                        auto at = [&](int c, int i, int j, int k) { return f0[c * GN + (k * GY + j) * GX + i]; };
                        float f[3], t[4];
                        gather_force3(at, o, f);
                        force_terms(w, m.q_bg, f, u, t);
#pragma unroll
                        for (int k = 0; k < 4; ++k) add_fixed(p + 12 + 2 * k, wide + (6 + k) * nc, t[k]);
                    }
                }
            }
            if (++rounds == every) {
                fold();
                rounds = 0;
            }
        }
    }
    fold();
}

// Spilled particles of the run (thread each).
template <int PASS>
__global__ void __launch_bounds__(NT) mom_spill(const MomArgs m) {
    constexpr int B = PassRows<PASS>::base, NR = PassRows<PASS>::n;
    const Args& a = m.a;
    const RunDev& R = a.runs[m.run];
    const int par = a.ctl->parity;
    const long long nc = (long long)m.ncx * m.ncy;
    for (int s = 0; s < a.nspecies && s < 2; ++s) {
        const Slots& S = a.slot[s][par];
        const int ns = min(*S.sn, a.spill_cap[s]);
        for (int k = blockIdx.x * NT + threadIdx.x; k < ns; k += gridDim.x * NT) {
            const long long g = S.scell[k];
            const long long lc = g - R.cell_off;
            if (lc < 0 || lc >= (long long)R.nx * R.ny * R.nz) continue;
            const int cz = (int)(lc / ((long long)R.nx * R.ny));
            const int rem = (int)(lc - (long long)cz * R.nx * R.ny);
            const int cy = rem / R.nx, cx = rem - cy * R.nx;
            long long acc[NR];
            for (int i = 0; i < NR; ++i) acc[i] = 0;
            const long long cc = (long long)(cy / m.by) * m.ncx + cx / m.bx;
            Mean2 mean{};
            if (PASS == 2) coarse_means(m, cc, mean);
            if (a.ndim == 3)
                add_particle<PASS, true>(m, R, s, R.sp[s].w, mean, cx, cy, cz, S.so[0][k], S.so[1][k], S.so[2][k],
                                         S.su[0][k], S.su[1][k], S.su[2][k], acc);
            else
                add_particle<PASS, false>(m, R, s, R.sp[s].w, mean, cx, cy, cz, S.so[0][k], S.so[1][k], 0.f,
                                          S.su[0][k], S.su[1][k], S.su[2][k], acc);
            for (int i = 0; i < NR; ++i)
                if (acc[i]) atomicAdd((unsigned long long*)&m.psum[(size_t)(B + i) * nc + cc], (unsigned long long)acc[i]);
        }
    }
}

// Per (x, y) column: mean over z of sum_c (E_c - <E_c>_z)^2, and the z means of Ez, Bx, By.  A block
// takes 32 neighbouring columns, each in ZS parts along z (a thread per part); sums and deviations are
// FP64, the parts added in a fixed order.  The bound is the FP64 unit (2 lanes per clock and SM), with
// 19 operations and conversions per node.  128 x 128 x 256 cells: a thread per column, 64 blocks,
// 753 us -> 181 us.
constexpr int ZS = 16;
__global__ void __launch_bounds__(32 * ZS) mom_columns(const MomArgs m) {
    __shared__ double part[ZS][5][32];
    __shared__ double zm[3][32];
    const RunDev& R = m.a.runs[m.run];
    const long long ncol = (long long)R.nx * R.ny;
    const int nz = m.a.ndim == 3 ? R.nz : 1;
    const int lane = threadIdx.x & 31, ps = threadIdx.x >> 5;
    const int k0 = (int)((long long)nz * ps / ZS), k1 = (int)((long long)nz * (ps + 1) / ZS);
    for (long long cb = blockIdx.x * 32ll; cb < ncol; cb += gridDim.x * 32ll) {
        const long long c = cb + lane;
        const bool on = c < ncol;
        double sum[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
        for (int k = k0; on && k < k1; ++k) {
            const size_t g = (size_t)k * ncol + c;
#pragma unroll
            for (int d = 0; d < 5; ++d) sum[d] += (double)(d < 3 ? R.E[d][g] : R.B[d - 3][g]);
        }
#pragma unroll
        for (int d = 0; d < 5; ++d) part[ps][d][lane] = sum[d];
        __syncthreads();
        if (ps < 5 && on) {
            double s = 0.0;
            for (int p = 0; p < ZS; ++p) s += part[p][ps][lane];
            s /= nz;
            if (ps < 3) zm[ps][lane] = s;
            if (ps >= 2) m.col[(ps - 1) * ncol + c] = s;   // Ez, Bx, By
        }
        __syncthreads();
        const double mean[3] = {zm[0][lane], zm[1][lane], zm[2][lane]};
        double w = 0.0;
#pragma unroll 4
        for (int k = k0; on && k < k1; ++k) {
            const size_t g = (size_t)k * ncol + c;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double e = (double)R.E[d][g] - mean[d];
                w += e * e;
            }
        }
        part[ps][0][lane] = w;
        __syncthreads();
        if (ps == 0 && on) {
            double s = 0.0;
            for (int p = 0; p < ZS; ++p) s += part[p][0][lane];
            m.col[c] = s / nz;
        }
        __syncthreads();
    }
}

constexpr int NTF = 32;   // a warp per block: few coarse cells, each a chain of FP64 operations
__global__ void __launch_bounds__(NTF) mom_finalize(const MomArgs m) {
    const RunDev& R = m.a.runs[m.run];
    const long long nc = (long long)m.ncx * m.ncy;
    const long long ncol = (long long)R.nx * R.ny;
    const int nz = m.a.ndim == 3 ? R.nz : 1;
    const double cells = (double)m.bx * m.by * nz;
    for (long long cc = blockIdx.x * (long long)NTF + threadIdx.x; cc < nc; cc += (long long)gridDim.x * NTF) {
        double p[MOM_PSUMS];
        for (int i = 0; i < MOM_PSUMS; ++i) p[i] = (double)m.psum[(size_t)i * nc + cc] * (1.0 / MOM_FIX);   // exact
        float* o = m.out;
        for (int s = 0; s < 2; ++s) {
            const double sw = p[4 * s];
            double mu[3] = {0, 0, 0}, var[3] = {0, 0, 0};
            if (sw > 0)
                for (int d = 0; d < 3; ++d) {
                    mu[d] = p[4 * s + 1 + d] / sw;
                    var[d] = p[8 + 3 * s + d] / sw;
                }
            o[(size_t)s * nc + cc] = (float)(sw / cells);
            o[(size_t)(2 + s) * nc + cc] = (float)mu[2];
            o[(size_t)(4 + 2 * s) * nc + cc] = (float)(0.5 * (var[0] + var[1]));
            o[(size_t)(5 + 2 * s) * nc + cc] = (float)var[2];
        }
        // field blocks, fixed order
        const int X0 = (int)(cc % m.ncx) * m.bx, Y0 = (int)(cc / m.ncx) * m.by;
        double f[MOM_COLS] = {0, 0, 0, 0};
        for (int j = 0; j < m.by; ++j)
            for (int i = 0; i < m.bx; ++i) {
                const long long c = (long long)(Y0 + j) * R.nx + (X0 + i);
                for (int k = 0; k < MOM_COLS; ++k) f[k] += m.col[(size_t)k * ncol + c];
            }
        for (int k = 0; k < MOM_COLS; ++k) f[k] /= (double)(m.bx * m.by);
        o[(size_t)8 * nc + cc] = (float)f[0];
        const double sw = p[4];
        double fzp = 0, vx = 0, vy = 0, uz = 0;
        if (sw > 0) {
            fzp = p[14] / sw;
            vx = p[15] / sw;
            vy = p[16] / sw;
            uz = p[7] / sw;
        }
        const double fzm = (double)m.q_bg * (f[1] + vx * f[3] - vy * f[2]);
        o[(size_t)9 * nc + cc] = (float)fzp;
        o[(size_t)10 * nc + cc] = (float)fzm;
        o[(size_t)11 * nc + cc] = uz != 0 ? (float)((double)m.nu_bg + (fzm - fzp) / uz) : 0.f;
    }
}

int grid_of(long long n) {
    long long g = (n + NT - 1) / NT;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

size_t moments_scratch_bytes(long long nc, long long ncol) {
    return (size_t)nc * MOM_PSUMS * sizeof(long long) + (size_t)ncol * MOM_COLS * sizeof(double) +
           (size_t)nc * 12 * sizeof(float);
}

cudaError_t launch_moments(const Args& a, const RunDev& host_run, int run, int bx, int by, float q_bg,
                           float nu_bg, float* out, void* scratch, cudaStream_t s) {
    auto pow2 = [](int v) { return v > 0 && (v & (v - 1)) == 0; };
    if (a.ndim == 3 && !(pow2(a.tx) && pow2(a.ty) && pow2(a.tz) && a.tx <= 8 && a.ty <= 8 && a.tz <= 4)) return cudaErrorInvalidValue;
    MomArgs m;
    m.a = a;
    m.run = run;
    m.bx = bx;
    m.by = by;
    m.ncx = host_run.nx / bx;
    m.ncy = host_run.ny / by;
    const int nz = a.ndim == 3 ? host_run.nz : 1;
    const int per = bx * by;
    m.zc = per >= NT ? 1 : (NT / per < nz ? NT / per : nz);
    m.q_bg = q_bg;
    m.nu_bg = nu_bg;
    const long long nc = (long long)m.ncx * m.ncy;
    m.psum = static_cast<long long*>(scratch);
    m.col = reinterpret_cast<double*>(m.psum + (size_t)nc * MOM_PSUMS);
    m.meanbuf = reinterpret_cast<float*>(m.col + (size_t)host_run.nx * host_run.ny * MOM_COLS);
    m.out = out;
    cudaError_t e = cudaMemsetAsync(m.psum, 0, (size_t)nc * MOM_PSUMS * sizeof(long long), s);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)nc, (unsigned)((nz + m.zc - 1) / m.zc));
    const unsigned tgrid = (unsigned)host_run.ntx * host_run.nty * host_run.ntz;
    if (a.ndim == 3) mom_tiles<1><<<tgrid, NT, 0, s>>>(m);
    else mom_particles<1><<<grid, NT, 0, s>>>(m);
    mom_spill<1><<<152, NT, 0, s>>>(m);
    mom_means<<<grid_of(nc), NT, 0, s>>>(m);
    if (a.ndim == 3) mom_tiles<2><<<tgrid, NT, 0, s>>>(m);
    else mom_particles<2><<<grid, NT, 0, s>>>(m);
    mom_spill<2><<<152, NT, 0, s>>>(m);
    const long long cblocks = ((long long)host_run.nx * host_run.ny + 31) / 32;
    mom_columns<<<(unsigned)(cblocks < 152 * 32 ? cblocks : 152 * 32), 32 * ZS, 0, s>>>(m);
    mom_finalize<<<(unsigned)(nc < 152ll * 32 * NTF ? (nc + NTF - 1) / NTF : 152 * 32), NTF, 0, s>>>(m);
    return cudaGetLastError();
}

cudaError_t preload_moments() {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, mom_particles<1>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_particles<2>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_tiles<1>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_tiles<2>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_spill<1>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_spill<2>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_means);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_columns);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, mom_finalize);
    return e;
}

}  // namespace pic
