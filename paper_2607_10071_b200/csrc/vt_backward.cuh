// Texel-side backward Sampling-VT kernel (gradient with respect to the features) for B200 (sm_100a).  Included by flashbev.cu
// inside its anonymous namespace, after vt_tiled.cuh.
//
// A CTA owns one texel column of one camera's map: up to 64 rows of it and up to 8 warps' channels.  The column's gradient stays
// in registers (a warp: 16 rows by 8 NT channels, as the accumulators of m16n8 fragments) while the CTA goes through the BEV
// cells that reach the column, in rounds of 32 cells per warp:
//
//   survey    The cells in question.  Depth and the limits of the column and of its rows are linear functions of the position
//             that must be positive wherever the depth is.  A lane takes a grid row (one x) and solves for the interval of y in
//             which the largest value of each over the heights is not negative; the warp numbers the intervals' cells through
//             and appends them to the CTA's list, 32 at a time.
//   weights   A lane takes a cell: it projects the height bins that can reach the column in fp64 and adds their bilinear weights
//             to the cell's column of a dense (row, cell) table in shared memory.  The mean modes count the cameras that see a
//             bin by the signs of the validity conditions, and the factor is part of the weight.  For each tile of 16 rows a
//             list says which cells have weights in it.
//   products  gradient[row, channel] += weights[row, cell] x grad_out[cell, channel], 16 listed cells at a time on the tensor
//             cores.  Every fp32 number is the exact sum of three bf16 ones.  The product of the leading pieces (16 bits: exact
//             for one cell) and the sum of the five next ones are kept apart, and rounded to fp32 once, together; the three
//             smallest are left out.
//
// A single product of a weight and a grad_out is off by at most 1.2e-7 of it, 2.6e-8 root mean square (an fp32 product: 6.0e-8 and
// 2.5e-8).  Against fp64 the results are as near as the scatter's or nearer: relative 2-norm 5.8e-8 to 9.0e-8 over three problems,
// the scatter 6.4e-8 to 2.2e-7 (long sums of reductions in any order), and 5.4e-8 to 6.3e-8 against 5.4e-8 to 6.5e-8 where two cells
// in a hundred have a gradient.  Two tf32 pieces, a bit short of 24, and three products: 1.0e-7 to 1.4e-7 in all of them, single
// products off by 4.8e-7, 7.8e-8 root mean square; 31.5 us on 200 x 200 x 8, C = 80, this 35.0.  Eight products (all but lo x lo)
// 39.6 us.
//
// Why: the scatter hands two fp32 vector reductions per record to the crossbar -- 11.5 M sectors for a gradient of 0.17 M on
// 200 x 200 x 8, C = 80 -- and is bound by the rate at which an SM can do that.  Here a texel leaves the SM once: 92 -> 35 us a pass
// (in a graph, into one result buffer, 87 -> 34); 56 x 100 maps of tilted cameras, C = 128, Eq. 1: 141 -> 88 us (137 -> 88).
// What bounds it now: no unit (on these two, of the SMs' active cycles: issue 38 and 45 %, tensor pipe 19 %; L1 data pipe 25 and 35 %
// of the launch); 12 and 15 of at most 16 warps per SM that wait at the barriers of a round, for grad_out and for chains of fp64
// operations, in 0.9 and 2 waves of CTAs of unequal size: an SM is active for 72 and 77 % of the launch.
// Forms that lost (measured with the tf32 products): 80 registers (24 warps per SM), whose spills cost more than the warps bring
// (calibrated 87 -> 116 us), but for up to 32 channels per warp (94 x 58 x 5, C = 32: 16.5 -> 13.4 us); row tiles of 32 rows without
// lists 37 and 116 us; fp32 FMAs instead of fragments 48 and 88 us (row quads) or slower.

constexpr int kBwdRows = 16;       // texel rows of a warp's tile
constexpr int kBwdMaxTiles = 4;    // ... times this many per CTA
constexpr int kBwdMaxWarps = 8;    // of a CTA
constexpr int kBwdSmWarps = 16;    // that an SM holds (24 in the instances of 80 registers)
constexpr int kBwdList = 1024;     // cells that wait for their weights
constexpr int kBwdDeal = 8;        // cells along y that go to the same slice

struct BwdParams {
    KParams k;
    int row_tiles;                    // tiles of 16 rows per CTA
    int row_warps, ch_tiles, groups;  // warps of a CTA: groups of row_warps x ch_tiles; a warp has every row_warps-th row tile
    int slices;                       // CTAs that share a texel column, each with its share of the cells
    int exclusive;                    // one CTA per column: results are stored, not added
};

// A condition c . (x, y) + ... >= 0 in float, relaxed by far more than the rounding of its evaluation.
struct __align__(16) BwdCond {
    float cx, cy;
    float cell;   // constant, with the largest part of the height
    float bin0;   // constant at height bin 0
    float slope;  // per height bin
    float pad[3];
};

struct BwdSmem {
    float *weights;        // [16 row_tiles][32 warps + 4]: a texel's weights; at the end the sums of the other groups
    double *mats;
    double (*exact)[4];    // mean modes: the validity conditions of every camera, [N][5]{x, y, bin 0, per bin}
    BwdCond *tile, *sees;  // the five conditions of the column; of every camera (mean modes)
    uint32_t *list;        // waiting cells
    uint8_t *slots;        // [row_tiles][32 warps]: the round's cells that have weights in the row tile
};

__host__ __device__ inline size_t bwd_smem_layout(unsigned char *base, BwdSmem *t, int N, int row_tiles, int row_warps, int ch_tiles,
                                                  int groups, int NT, int RT, int reduce)
{
    size_t o = 0;
    auto take = [&](size_t bytes) {
        unsigned char *ptr = base ? base + o : nullptr;
        o += align16(bytes);
        return ptr;
    };
    const size_t warps = (size_t)row_warps * ch_tiles * groups, all = reduce == FLASHBEV_REDUCE_SUM ? 0 : (size_t)N;
    const size_t weights = (size_t)row_tiles * kBwdRows * (32 * warps + 4) * sizeof(float);
    const size_t sums = (size_t)(groups - 1) * row_warps * ch_tiles * RT * NT * 32 * sizeof(float4);
    unsigned char *p0 = take(weights > sums ? weights : sums);
    unsigned char *p1 = take((all ? all : 1) * 12 * sizeof(double));
    unsigned char *p2 = take(all * 5 * 4 * sizeof(double));
    unsigned char *p3 = take(5 * sizeof(BwdCond));
    unsigned char *p4 = take(all * 5 * sizeof(BwdCond));
    unsigned char *p5 = take(kBwdList * sizeof(uint32_t));
    unsigned char *p6 = take((size_t)row_tiles * 32 * warps);
    if (t) {
        t->weights = reinterpret_cast<float *>(p0), t->mats = reinterpret_cast<double *>(p1);
        t->exact = reinterpret_cast<double(*)[4]>(p2);
        t->tile = reinterpret_cast<BwdCond *>(p3), t->sees = reinterpret_cast<BwdCond *>(p4);
        t->list = reinterpret_cast<uint32_t *>(p5), t->slots = p6;
    }
    return o;
}

// Condition t of the samples that a camera (scaled matrix M) sees with their upper left tap in columns [x0, x1) and rows [y0, y1):
// depth, left, right, upper, lower limit, each relaxed by 1/64 texel or 0.05 m (samples are tested exactly later) and by a
// bound on the rounding of the coefficients and of the evaluation (a sum of four float products: below 1e-6 of their sizes).
__device__ __forceinline__ BwdCond bwd_condition(const KParams &p, const double *M, int t, float x0, float x1, float y0, float y1)
{
    const float eps = 1.f / 64.f;
    const float lim = t == 1 ? fmaxf(x0, -0.5f) + 0.5f - eps : t == 2 ? fminf(x1, (float)p.Wf - 0.5f) + 0.5f + eps
                    : t == 3 ? fmaxf(y0, -0.5f) + 0.5f - eps : fminf(y1, (float)p.Hf - 0.5f) + 0.5f + eps;
    const float zl = (float)(p.z_min + 0.5 * p.dz), zs = (float)p.dz * (float)(p.Z - 1);
    const float most[4] = {(float)fmax(fabs(p.x_min), fabs(p.x_min + p.dx * p.X)),
                           (float)fmax(fabs(p.y_min), fabs(p.y_min + p.dy * p.Y)), fmaxf(fabsf(zl), fabsf(zl + zs)), 1.f};
    float u[4], err = 0.f;  // the coefficients of (x, y, z, 1)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float d = (float)M[8 + e], v = (float)M[(t <= 2 ? 0 : 4) + e];
        u[e] = t == 0 ? d : ((t & 1) ? v - lim * d : lim * d - v);
        err += (t == 0 ? fabsf(d) : fabsf(v) + fabsf(lim * d)) * most[e];
    }
    if (t == 0) u[3] -= 0.05f;
    u[3] += 4e-6f * err;
    BwdCond c;
    c.cx = u[0], c.cy = u[1];
    c.bin0 = u[3] + u[2] * zl, c.slope = u[2] * (float)p.dz;
    c.cell = c.bin0 + fmaxf(0.f, u[2] * zs);
    return c;
}

// The whole numbers i in [0, n) with a[t] + i s[t] >= 0 for all five conditions (or a few more): [lo, hi].
__device__ __forceinline__ void bwd_interval(const float (&a)[5], const float (&s)[5], int n, int &lo, int &hi)
{
    float l = 0.f, h = (float)(n - 1);
    bool empty = false;
#pragma unroll
    for (int t = 0; t < 5; ++t) {
        float z;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(s[t]));
        z *= -a[t];
        l = s[t] > 0.f ? fmaxf(l, z) : l;
        h = s[t] < 0.f ? fminf(h, z) : h;
        empty |= (s[t] == 0.f) & (a[t] < 0.f);
    }
    const float guard = 0.05f + 2e-6f * (float)n;
    lo = max((int)ceilf(fminf(l, (float)n) - guard), 0);
    hi = empty ? -1 : min((int)floorf(fmaxf(h, -1.f) + guard), n - 1);
}

// a and b as sums of three bf16 numbers each, in pairs (a in the low half): 24 = 8 + 8 + 8 bits.  The differences are exact, and the
// last piece has at most 7 bits left: nothing is lost.  With |v| in [1, 2) the pieces after the first are at most 2^-8 and 2^-17.
// (Under 2^-109 the last bits fall below bf16's smallest number, 2^-133.  A number that rounds to infinity is one more
// grad_out that is not finite: see the end of the kernel.)
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t &hi, uint32_t &mid, uint32_t &lo)
{
    const auto minus = [](uint32_t v) {
        return make_float2(__uint_as_float((v << 16) ^ 0x80000000u), __uint_as_float((v & 0xffff0000u) ^ 0x80000000u));
    };
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
    float2 r = __fadd2_rn(make_float2(a, b), minus(hi));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(mid) : "f"(r.y), "f"(r.x));
    r = __fadd2_rn(r, minus(mid));
    lo = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632u);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// NT: channels per warp / 8.  RT: row tiles per warp.  SUM: the reduce mode without counts of other cameras.  WHOLE: the channels
// fill the warps' tiles (a quarter of the products' instructions would be checks).  (Every stage is in the kernel once and small: a
// CTA runs most of it once, through an instruction cache that it shares with others at other stages.)
template <int NT, int RT, bool SUM, bool WHOLE>
__global__ void __launch_bounds__(kBwdMaxWarps * 32, NT * RT <= 4 ? 3 : 2) vt_texel_backward_kernel(const BwdParams q)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int list_n, slots_n[kBwdMaxTiles];
    constexpr unsigned FULL = 0xffffffffu;
    const KParams &p = q.k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x, warps = threads >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool eq1 = !SUM && p.reduce == FLASHBEV_REDUCE_CAMERA_MEAN_Z_SUM;
    BwdSmem sm;
    bwd_smem_layout(smem_raw, &sm, p.N, q.row_tiles, q.row_warps, q.ch_tiles, q.groups, NT, RT, p.reduce);

    // (programmatic dependent launch: this grid's CTAs are placed while the one before drains, as in the forward)
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- which texel column (rows from blockIdx.z on, channels from blockIdx.y on)
    const unsigned column = blockIdx.x / (unsigned)q.slices, slice = blockIdx.x - column * (unsigned)q.slices;
    const unsigned map = column / (unsigned)p.Wf;  // b * N + n
    const int xt = (int)(column - map * (unsigned)p.Wf);
    const int rows = q.row_tiles * kBwdRows, ya = blockIdx.z * rows, rv = min(rows, p.Hf - ya), pitch = 32 * warps + 4;
    const int b = (int)(map / (unsigned)p.N), n = (int)(map - (unsigned)b * p.N);
    const size_t rowf = (size_t)p.Wf * p.C;
    float *const dst = p.gfeat + ((size_t)map * p.Hf + ya) * rowf + (size_t)xt * p.C;

    const double zl = p.z_min + 0.5 * p.dz;  // centre of bin 0
    const int cams = SUM ? 1 : p.N, cam0 = SUM ? n : 0;  // cameras in the tables
    const double *const M = sm.mats + (n - cam0) * 12;
    for (int i = tid; i < cams * 12; i += threads) {
        const int m = i / 12, e = i - m * 12;
        double v = (double)__ldg(p.l2i + ((size_t)b * p.N + cam0 + m) * 16 + e);
        if (e < 4) v *= p.sx;
        else if (e < 8) v *= p.sy;
        sm.mats[i] = v;
    }
    if (tid == 0) list_n = 0;
    if (tid < kBwdMaxTiles) slots_n[tid] = 0;
    __syncthreads();
    if (tid < 5) sm.tile[tid] = bwd_condition(p, M, tid, xt - 1, xt + 1, ya - 1, ya + rows);
    if (!SUM) {
        for (int i = tid; i < p.N * 10; i += threads) {
            const int mt = i < p.N * 5 ? i : i - p.N * 5, m = mt / 5, t = mt - m * 5;
            const double *A = sm.mats + m * 12;
            if (i < p.N * 5) {
                sm.sees[mt] = bwd_condition(p, A, t, -1, p.Wf, -1, p.Hf);
                continue;
            }
            // d > 0.1, fx > -1/2, fx < Wf - 1/2 (times the depth), likewise fy
            const double size = t == 2 ? (double)p.Wf : (double)p.Hf;
            const double *B = A + (t == 0 ? 8 : t <= 2 ? 0 : 4);
            double u[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] = t == 2 || t == 4 ? size * A[8 + e] - B[e] : B[e];
            double *x = sm.exact[mt];
            x[0] = u[0], x[1] = u[1], x[2] = u[3] + u[2] * zl - (t == 0 ? kDepthMin : 0.0), x[3] = u[2] * p.dz;
        }
    }
    __syncthreads();

    // ---- role of the warp in the products: row tiles row_warp, + row_warps, channels [ch0, ch0 + 8 NT)
    const int tiles = q.row_warps * q.ch_tiles, group = warp / tiles, row_warp = (warp - group * tiles) / q.ch_tiles;
    const int ch0 = (blockIdx.y * q.ch_tiles + warp % q.ch_tiles) * (NT * 8);
    float2 acc[RT][NT][2];  // fragment layout: rows lane / 4 and + 8, channels 2 (lane % 4) and + 1
    const float *const gout = p.gout + (size_t)b * p.X * p.Y * p.C;
    const float x_first = (float)(p.x_min + 0.5 * p.dx), y_first = (float)(p.y_min + 0.5 * p.dy);
    const float dxf = (float)p.dx, dyf = (float)p.dy;
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[i][j][0] = acc[i][j][1] = make_float2(0.f, 0.f);
    // (a second pass, if a grad_out that is not finite was met: see the end)
    for (bool again = false;; again = true) {
        int row0 = 32 * (warp - warps);    // a chunk is 32 grid rows, a row per lane
        int y_lo = 0, y_n = 0, y_sum = 0;  // the lane's row: first cell, cells, cells up to the end of it
        unsigned chunk_n = 0, next = 0;    // cells of the chunk; this slice's next one
        unsigned sl = (slice + (unsigned)warp) % (unsigned)q.slices;

        for (bool done = false;;) {
            // ---- survey: cells that can reach the column, until the list is full
            for (;;) {
                // this slice's cells of the chunk, numbered from 0: every slices-th group of kBwdDeal
                const unsigned j = ((next + lane) / kBwdDeal * q.slices + sl) * kBwdDeal + (next + lane) % kBwdDeal;
                if (__shfl_sync(FULL, j, 0) >= chunk_n) {
                    if (row0 + 32 * warps >= p.X) {
                        done = true;
                        break;
                    }
                    row0 += 32 * warps;
                    const float x = fmaf((float)(row0 + lane), dxf, x_first);
                    float a[5], s[5];
#pragma unroll
                    for (int t = 0; t < 5; ++t) {
                        a[t] = fmaf(sm.tile[t].cx, x, fmaf(sm.tile[t].cy, y_first, sm.tile[t].cell));
                        s[t] = sm.tile[t].cy * dyf;
                    }
                    int y_hi;
                    bwd_interval(a, s, p.Y, y_lo, y_hi);
                    y_n = row0 + lane < p.X ? max(0, y_hi - y_lo + 1) : 0;
                    y_sum = y_n;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int v = __shfl_up_sync(FULL, y_sum, off);
                        if (lane >= off) y_sum += v;
                    }
                    chunk_n = (unsigned)__shfl_sync(FULL, y_sum, 31), next = 0;
                    sl = sl + 1u >= (unsigned)q.slices ? 0u : sl + 1u;
                    continue;
                }
                // (every warp may add 32 cells before it sees another's)
                if (*(volatile int *)&list_n > kBwdList - 32 * warps) break;
                const bool keep = j < chunk_n;
                int r = 0;  // the first row whose cells end behind j
#pragma unroll
                for (int step = 16; step; step >>= 1) {
                    const int v = __shfl_sync(FULL, y_sum, r + step - 1);
                    if ((unsigned)v <= j) r += step;
                }
                const int iy = __shfl_sync(FULL, y_lo - (y_sum - y_n), r) + (int)j;
                const unsigned bal = __ballot_sync(FULL, keep);
                int at = 0;
                if (lane == 0) at = atomicAdd(&list_n, __popc(bal));
                at = __shfl_sync(FULL, at, 0);
                at += __popc(bal & lt_mask);
                if (keep) sm.list[FB_IDX(at, kBwdList, p.err)] = FB_IDX((row0 + r) * p.Y + iy, p.X * p.Y, p.err);
                next += 32;
            }
            const bool all_done = __syncthreads_and(done);
            const int waiting = list_n;

            for (int first = 0; first < waiting; first += 32 * warps) {
                if (first + 32 * warp < waiting) {
                    // ---- weights of 32 cells, a cell per lane
                    float *const own = sm.weights + 32 * warp + lane;
                    for (int i = lane; i < rows * 8; i += 32) {
                        float *const at = sm.weights + 32 * warp + (i >> 3) * pitch + (i & 7) * 4;
                        *reinterpret_cast<float4 *>(at) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    __syncwarp();
                    unsigned touched = 0u;  // bit t: the cell has weights in row tile t
                    if (first + 32 * warp + lane < waiting) {
                        const uint32_t cell = sm.list[first + 32 * warp + lane];
                        const int ix = (int)(cell / (unsigned)p.Y), iy = (int)(cell - (unsigned)ix * (unsigned)p.Y);
                        const float xf = fmaf((float)ix, dxf, x_first), yf = fmaf((float)iy, dyf, y_first);
                        const double2 xy = make_double2(p.x_min + ((double)ix + 0.5) * p.dx, p.y_min + ((double)iy + 0.5) * p.dy);
                        int klo, khi;  // height bins that can reach the column
                        {
                            float a[5], s[5];
#pragma unroll
                            for (int t = 0; t < 5; ++t) {
                                a[t] = fmaf(sm.tile[t].cx, xf, fmaf(sm.tile[t].cy, yf, sm.tile[t].bin0));
                                s[t] = sm.tile[t].slope;
                            }
                            bwd_interval(a, s, p.Z, klo, khi);
                        }
                        float scale = 1.f;
                        unsigned long long seen = 0ull;  // cameras that may see the cell (Eq. 1: the other ones)
                        // how many of the bins [k, k + n) camera m sees, bit by bit
                        const auto bins = [&](int m, int k, int n) {
                            unsigned in = (1u << n) - 1u;
#pragma unroll
                            for (int t = 0; t < 5; ++t) {
                                const double *c = sm.exact[m * 5 + t];
                                const double v = fma(c[0], xy.x, fma(c[1], xy.y, c[2]));
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (!(fma((double)(k + j), c[3], v) > 0.0)) in &= ~(1u << j);
                            }
                            return in;
                        };
                        if (!SUM && klo <= khi) {
                            for (int m = 0; m < p.N; ++m) {
                                bool sees = !(eq1 && m == n);
#pragma unroll
                                for (int t = 0; t < 3; ++t) {  // (depth, left, right)
                                    const BwdCond &c = sm.sees[m * 5 + t];
                                    sees &= !(fmaf(c.cx, xf, fmaf(c.cy, yf, c.cell)) < 0.f);
                                }
                                if (sees) seen |= 1ull << m;
                            }
                            if (!eq1) {
                                int count = 0;
                                for (unsigned long long s = seen; s; s &= s - 1ull) {
                                    const int m = __ffsll((long long)s) - 1;
                                    for (int k = 0; k < p.Z; k += 4) count += __popc(bins(m, k, min(4, p.Z - k)));
                                }
                                scale = 1.f / (float)max(count, 1);
                            }
                        }
                        const double a0 = fma(M[1], xy.y, fma(M[0], xy.x, M[3]));
                        const double a1 = fma(M[5], xy.y, fma(M[4], xy.x, M[7]));
                        const double a2 = fma(M[9], xy.y, fma(M[8], xy.x, M[11]));
                        const double wlim = (double)p.Wf - 0.5, hlim = (double)p.Hf - 0.5;
                        // bins projected together: a projection is a chain of a dozen fp64 operations
                        constexpr int K = NT * RT <= 4 ? 2 : 4;
                        for (int k0 = klo; k0 <= khi; k0 += K) {
                            int rr[K];
                            float wx[K], ty[K];
#pragma unroll
                            for (int j = 0; j < K; ++j) {
                                const double zw = fma((double)(k0 + j), p.dz, zl);
                                const double d = fma(M[10], zw, a2), r = fast_rcp(d);  // (d <= 0 and NaN fail below)
                                const double fx = fma(fma(M[2], zw, a0), r, -0.5), fy = fma(fma(M[6], zw, a1), r, -0.5);
                                bool ok = (k0 + j <= khi) & (d > kDepthMin);
                                ok &= (fx > -0.5) & (fx < wlim) & (fy > -0.5) & (fy < hlim);
                                double flx, fly;
                                const int c = floor_int(fx, flx) - xt, row = floor_int(fy, fly) - ya;
                                const float tx = (float)(fx - flx);
                                ok &= (c == 0) | (c == -1);
                                wx[j] = c == 0 ? 1.f - tx : tx;
                                rr[j] = ok && row >= -1 && row < rv ? row : -2;
                                ty[j] = (float)(fy - fly);
                            }
                            unsigned den = 0u;  // Eq. 1: other cameras that see the bins, a byte each
                            if (eq1)
                                for (unsigned long long s = seen; s; s &= s - 1ull) {
                                    const unsigned in = bins(__ffsll((long long)s) - 1, k0, K);
                                    den += (in & 1u) | (in & 2u) << 7 | (in & 4u) << 14 | (in & 8u) << 21;
                                }
#pragma unroll
                            for (int j = 0; j < K; ++j) {
                                const int r = rr[j];
                                if (r < -1) continue;
                                const float sc = eq1 ? 1.f / (float)(1u + ((den >> (8 * j)) & 0xffu)) : scale;
                                const float w = wx[j] * sc;
                                if (r >= 0) {
                                    own[FB_IDX(r, rows, p.err) * pitch] += w * (1.f - ty[j]);
                                    touched |= 1u << (r / kBwdRows);
                                }
                                if (r + 1 < rv) {
                                    own[FB_IDX(r + 1, rows, p.err) * pitch] += w * ty[j];
                                    touched |= 1u << ((r + 1) / kBwdRows);
                                }
                            }
                        }
                    }
                    for (int t = 0; t < q.row_tiles; ++t) {
                        const unsigned bal = __ballot_sync(FULL, (touched >> t) & 1u);
                        int at = 0;
                        if (lane == 0) at = atomicAdd(&slots_n[t], __popc(bal));
                        at = __shfl_sync(FULL, at, 0) + __popc(bal & lt_mask);
                        if ((bal >> lane) & 1u) {
                            at = FB_IDX(t * 32 * warps + at, q.row_tiles * 32 * warps, p.err);
                            sm.slots[at] = (uint8_t)(32 * warp + lane);
                        }
                    }
                }
                __syncthreads();

                // ---- products: 16 cells at a time
                if (!again) {
#pragma unroll
                    for (int i = 0; i < RT; ++i) {
                        const int row_tile = row_warp + i * q.row_warps;
                        if (RT > 1 && row_tile >= q.row_tiles) break;
                        const float *const wt = sm.weights + (row_tile * kBwdRows + (lane >> 2)) * pitch;
                        const uint8_t *const slots = sm.slots + row_tile * 32 * warps;
                        const int n_slots = slots_n[row_tile];
#pragma unroll 1
                        for (int k = 16 * group; k < n_slots; k += 16 * q.groups) {
                            // (fragments: rows lane / 4 and + 8, cells 2 (lane % 4) and + 1, + 8, + 9.  Cells past the last
                            // one: the last one, with weight 0)
                            float g[4][NT], w[4][2];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int at = k + 2 * (lane & 3) + (c & 1) + (c >> 1) * 8, slot = slots[min(at, n_slots - 1)];
                                const size_t cell = FB_IDX(sm.list[first + slot], p.X * p.Y, p.err);
                                const float *const src = gout + cell * (unsigned)p.C + ch0 + (lane >> 2);
#pragma unroll
                                for (int j = 0; j < NT; ++j)
                                    g[c][j] = WHOLE || ch0 + 8 * j + (lane >> 2) < p.C ? __ldg(src + 8 * j) : 0.f;
                                w[c][0] = at < n_slots ? wt[slot] : 0.f, w[c][1] = at < n_slots ? wt[8 * pitch + slot] : 0.f;
                            }
                            uint32_t ah[4], am[4], al[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) split_bf16(w[h & 2][h & 1], w[(h & 2) + 1][h & 1], ah[h], am[h], al[h]);
#pragma unroll
                            for (int j = 0; j < NT; ++j) {
                                uint32_t bh[2], bm[2], bl[2];
                                split_bf16(g[0][j], g[1][j], bh[0], bm[0], bl[0]);
                                split_bf16(g[2][j], g[3][j], bh[1], bm[1], bl[1]);
                                float t[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f};
                                // (mid x lo, lo x mid and lo x lo are left out: at most 2^-24 of a product, 2^-27 root mean
                                // square)
                                mma_bf16(t, ah, bh[0], bh[1]);
                                mma_bf16(u, ah, bl[0], bl[1]);
                                mma_bf16(u, al, bh[0], bh[1]);
                                mma_bf16(u, am, bm[0], bm[1]);
                                mma_bf16(u, ah, bm[0], bm[1]);
                                mma_bf16(u, am, bh[0], bh[1]);
                                const float2 s0 = __fadd2_rn(make_float2(t[0], t[1]), make_float2(u[0], u[1]));
                                const float2 s1 = __fadd2_rn(make_float2(t[2], t[3]), make_float2(u[2], u[3]));
                                acc[i][j][0] = __fadd2_rn(acc[i][j][0], s0);
                                acc[i][j][1] = __fadd2_rn(acc[i][j][1], s1);
                            }
                        }
                    }
                } else if (group == 0) {
                    for (int c = 0; c < min(32 * warps, waiting - first); ++c) {
                        const float *src = gout + (size_t)FB_IDX(sm.list[first + c], p.X * p.Y, p.err) * (unsigned)p.C;
                        for (int r = row_warp * kBwdRows; r < rv; ++r) {
                            if (r / kBwdRows % q.row_warps != row_warp) continue;
                            const float w = sm.weights[r * pitch + c];
                            if (w == 0.f) continue;
                            for (int ch = ch0 + lane; ch < min(ch0 + 8 * NT, p.C); ch += 32)
                                atomicAdd(dst + (size_t)r * rowf + ch, w * __ldg(src + ch));
                        }
                    }
                }
                __syncthreads();  // the weights have been taken
                if (tid < kBwdMaxTiles) slots_n[tid] = 0;
                if (first + 32 * warps < waiting) __syncthreads();
            }
            if (all_done) break;
            if (tid == 0) list_n = 0;
            __syncthreads();
        }
        if (again) return;

        // An infinite or NaN grad_out leaves no finite number in its channel's products, whatever the weights.  Then the column
        // stays zero for now and is made once more, record by record.
        float big = 0.f;
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) big = fmaf(acc[i][j][h].x, 0.f, big), big = fmaf(acc[i][j][h].y, 0.f, big);
        const bool odd = __syncthreads_or(big != 0.f);

        // ---- the groups' sums, then the column's gradient leaves the SM
        if (q.groups > 1) {
            float4 *const sums = reinterpret_cast<float4 *>(sm.weights) + lane;
            if (group > 0) {
#pragma unroll
                for (int i = 0; i < RT; ++i)
#pragma unroll
                    for (int j = 0; j < NT; ++j)
                        sums[(((warp - tiles) * RT + i) * NT + j) * 32] =
                            make_float4(acc[i][j][0].x, acc[i][j][0].y, acc[i][j][1].x, acc[i][j][1].y);
            }
            __syncthreads();
            if (group == 0)
#pragma unroll 1
                for (int g = 1; g < q.groups; ++g)
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int j = 0; j < NT; ++j) {
                            const float4 v = sums[(((warp + (g - 1) * tiles) * RT + i) * NT + j) * 32];
                            acc[i][j][0] = __fadd2_rn(acc[i][j][0], make_float2(v.x, v.y));
                            acc[i][j][1] = __fadd2_rn(acc[i][j][1], make_float2(v.z, v.w));
                        }
        }
        if (group == 0) {
#pragma unroll
            for (int ih = 0; ih < 2 * RT; ++ih) {
                const int i = ih >> 1, h = ih & 1, r = (row_warp + i * q.row_warps) * kBwdRows + 8 * h + (lane >> 2);
                if (r >= rv) continue;
                float *row = dst + (size_t)r * rowf + ch0 + 2 * (lane & 3);
#ifdef FLASHBEV_DEBUG_BOUNDS
                row = p.gfeat + FB_IDX64((size_t)(row - p.gfeat), (size_t)p.B * p.N * p.Hf * rowf + 8, p.err);
#endif
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    if (ch0 + 8 * j + 2 * (lane & 3) >= p.C) continue;  // (C is a multiple of 4)
                    const float2 v = odd ? make_float2(0.f, 0.f) : acc[i][j][h];
                    if (q.exclusive) *reinterpret_cast<float2 *>(row + 8 * j) = v;
                    else if (v.x != 0.f || v.y != 0.f) atomicAdd(reinterpret_cast<float2 *>(row + 8 * j), v);
                }
            }
        }
        if (!odd) return;
        if (tid == 0) list_n = 0;
        __syncthreads();
    }
}
