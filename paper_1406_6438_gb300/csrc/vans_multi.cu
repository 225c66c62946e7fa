// vans_multi.cu -- two to four time steps per launch with the steps in between
// held on chip (launch kind 9, D2Q9).
//
// One step of the other kinds reads and writes every population: 76 bytes per
// cell update, which is what bounds them (4096^2: 197 us per step, 0.95 of the copy
// bandwidth).  Here a warp walks down a strip of rows of one 64-column block, two
// adjacent cells per lane, and carries T steps along as a wave: when it has loaded
// row r it computes step 1 of row r, step 2 of row r-1, ..., step T of row r-T+1,
// and stores only the last.  What step l+1 of a row still needs of step l's rows
// stays with the lane (the +-1 column shift of the pull is a shuffle), so a launch
// moves 76 bytes per cell for T steps.  No barrier, no shared state between warps:
// the outer ghost_cols columns of a block are computed redundantly (8 of 64 for
// T = 3, 4), as are the T-1 rows before and after a strip.
//
// What bounds it is the FP32 pipe and its latency: an update of a pair of cells is
// 91 packed instructions (fma.rn.f32x2 takes the pipe for two cycles, three with
// three register operands, but one issue slot), 220 cycles per warp at four warps
// per scheduler, 350 for a lone one.  Hence what does not change from step to step
// (the porosity terms, 13 pairs per cell) is formed once per row and kept in
// shared memory, the e_y > 0 values that wait two turns are kept there too (in
// registers they cost 12 per step and as many moves), and the next row's loads go
// out before the last step: 160-168 registers, 12 warps per SM, none spilled.
// Measured at 4096^2 (us per step; ncu: DRAM 0.3 of its peak): T = 2 135.6, 3 106.7,
// 4 100.7, between walls 135.8, 108.0, 101.2; with the autotuner's shape 2048^2 27.0,
// between walls 27.4, 1024^2 8.4 and 9.2 (kind 7: 12.1), 512^2
// 3.8 and 4.4 (kind 0: 4.8).  With 128 registers (16 warps) T = 2 gains 3 %, 3 and 4
// spill and lose.
//
// The result does not depend on T, on the strips or on the column blocks
// (vans_pair.cuh).
#include <atomic>

#include "vans_pair.cuh"

namespace vans {

namespace {

constexpr int kPorBytes = 13 * 8 * 32;   // Por of one warp and row

// columns on each side of a block that are computed but not stored: one per
// step, even so that the pairs stay aligned
__host__ __device__ constexpr int ghost_cols(int T) { return (T + 1) & ~1; }
__host__ __device__ constexpr int out_cols(int T) { return 64 - 2 * ghost_cols(T); }

__device__ __forceinline__ void por_put(float4 *slot, int lane, const Por &P) {
    slot[0 * 32] = make_float4(P.e0.x, P.e0.y, P.hx.x, P.hx.y);
    slot[1 * 32] = make_float4(P.hy.x, P.hy.y, P.al.x, P.al.y);
    slot[2 * 32] = make_float4(P.be.x, P.be.y, P.wd[1].x, P.wd[1].y);
    slot[3 * 32] = make_float4(P.wd[2].x, P.wd[2].y, P.wd[3].x, P.wd[3].y);
    slot[4 * 32] = make_float4(P.wd[4].x, P.wd[4].y, P.wd[5].x, P.wd[5].y);
    slot[5 * 32] = make_float4(P.wd[6].x, P.wd[6].y, P.wd[7].x, P.wd[7].y);
    reinterpret_cast<f2 *>(slot - lane + 6 * 32)[lane] = P.wd[8];
}

__device__ __forceinline__ void por_get(const float4 *slot, int lane, Por &P) {
    float4 t = slot[0 * 32];
    P.e0 = make_float2(t.x, t.y); P.hx = make_float2(t.z, t.w);
    t = slot[1 * 32];
    P.hy = make_float2(t.x, t.y); P.al = make_float2(t.z, t.w);
    t = slot[2 * 32];
    P.be = make_float2(t.x, t.y); P.wd[1] = make_float2(t.z, t.w);
    t = slot[3 * 32];
    P.wd[2] = make_float2(t.x, t.y); P.wd[3] = make_float2(t.z, t.w);
    t = slot[4 * 32];
    P.wd[4] = make_float2(t.x, t.y); P.wd[5] = make_float2(t.z, t.w);
    t = slot[5 * 32];
    P.wd[6] = make_float2(t.x, t.y); P.wd[7] = make_float2(t.z, t.w);
    P.wd[8] = reinterpret_cast<const f2 *>(slot - lane + 6 * 32)[lane];
}

__device__ __forceinline__ int wrap(int c, int n) {
    while (c < 0) c += n;
    while (c >= n) c -= n;
    return c;
}

// One warp's strip of rows [y0, y1) of a 64-column block.  WALLS: bounce-back
// walls on the y faces.  The wave runs through the rows past a wall as well (they
// wrap around like a periodic axis's and nothing of them is kept); what a row
// next to a wall pulls from there is put in its place first: the entry that
// bounced off, at the column from which the shift brings it home.
template <int T, bool WALLS, int GL = ghost_cols(T)>
struct Strip {
    const VDom &d;
    const float *__restrict__ fin;
    float *__restrict__ fout;
    unsigned char *ring;           // this warp's T rows of Por words
    f2 *up;                        // this lane's part of the kept e_y > 0 values
    int x, ia, y0, y1, lane, r, slot, odd;
    int yp;                        // the row at op
    uint32_t second;               // bytes from the lane's first column to its second
    uint32_t om, oz, op, out;      // byte offsets of the rows below, at and above the
                                   // next row to load, and of the next row to store
    bool inside, xedge;
    Row em, ez;                    // porosity rows r-1, r
    f2 raw[9], enext;              // row r of step 1 and porosity row r+1, loaded a turn ahead
    // per step l = 1 .. T-1: what step l+1 still needs of earlier rows, shifted:
    // the e_y = 0 values of one row back in registers, the e_y > 0 values of two
    // rows back in shared memory, [l][turn parity][direction]
    f2 mid[T - 1][3];

    // pair of plane p at byte offset `off` of this lane's first column
    __device__ __forceinline__ f2 load(const float *p, uint32_t off) const {
        const char *q = reinterpret_cast<const char *>(p);
        return inside ? __ldg(reinterpret_cast<const f2 *>(q + off))
                      : make_float2(__ldg(reinterpret_cast<const float *>(q + off)),
                                    __ldg(reinterpret_cast<const float *>(q + (uint32_t)(off + second))));
    }
    // the pair s columns to the right (s = -1, 1) in row y
    __device__ __forceinline__ f2 load_beside(const float *p, int y, int s) const {
        const float *row = p + (long long)y * d.pitch + d.off;
        return make_float2(__ldg(row + wrap(x + s, d.nx)), __ldg(row + wrap(x + 1 + s, d.nx)));
    }
    __device__ __forceinline__ float4 *por_row(int k) const {
        return reinterpret_cast<float4 *>(ring + k * kPorBytes) + lane;
    }
    __device__ __forceinline__ f2 *up_row(int l, int par) const {
        return up + ((l - 1) * 2 + par) * (3 * 32);
    }
    __device__ __forceinline__ uint32_t row_off(int y) const {       // 0 <= y < ny
        return ((uint32_t)y * (uint32_t)d.pitch + (uint32_t)(d.off + ia)) * 4u;
    }
    // the populations that step 1 of row y (at offset oz; rows om, op below and
    // above it) pulls, not yet shifted in x, and the porosity row above
    template <bool W>
    __device__ __forceinline__ void load_row(int y) {
        const long long plane = d.plane;
        enext = load(d.eps, op);
        raw[0] = load(fin, oz);
        raw[1] = load(fin + 1 * plane, oz);
        raw[3] = load(fin + 3 * plane, oz);
        raw[2] = load(fin + 2 * plane, om);
        raw[5] = load(fin + 5 * plane, om);
        raw[6] = load(fin + 6 * plane, om);
        raw[4] = load(fin + 4 * plane, op);
        raw[7] = load(fin + 7 * plane, op);
        raw[8] = load(fin + 8 * plane, op);
        if (W && d.wall_y && y == 0) {
            raw[2] = load(fin + 4 * plane, oz);
            raw[5] = load_beside(fin + 7 * plane, y, 1);
            raw[6] = load_beside(fin + 8 * plane, y, -1);
        }
        if (W && d.wall_y && y == d.ny - 1) {
            raw[4] = load(fin + 2 * plane, oz);
            raw[7] = load_beside(fin + 5 * plane, y, -1);
            raw[8] = load_beside(fin + 6 * plane, y, 1);
        }
    }
    template <bool W>
    __device__ __forceinline__ void prefetch() {                     // row r + 1
        om = oz;
        oz = op;
        if (++yp == d.ny) yp = 0;
        op = row_off(yp);
        load_row<W>(r + 1);
    }
    __device__ __forceinline__ void moving_wall(const Por &P, f2 h[9]) const {
        h[4] = fma2(P.e0, bc(wall_gain<9>(d, 4, 1.f)), h[4]);
        h[7] = fma2(P.e0, bc(wall_gain<9>(d, 7, 1.f)), h[7]);
        h[8] = fma2(P.e0, bc(wall_gain<9>(d, 8, 1.f)), h[8]);
    }
    // step 1 of row r
    template <bool W>
    __device__ __forceinline__ void first(f2 o[9]) {
        const Row ep = with_neighbours(enext);
        f2 h[9];
        h[0] = raw[0];
        h[1] = from_left(raw[1]);
        h[3] = from_right(raw[3]);
        h[2] = raw[2];
        h[5] = from_left(raw[5]);
        h[6] = from_right(raw[6]);
        h[4] = raw[4];
        h[7] = from_right(raw[7]);
        h[8] = from_left(raw[8]);
        Por P;
        const bool above = W && d.wall_y && r == d.ny - 1;
        porosity_terms(d, em, ez, ep, W && d.wall_y && r == 0, above, P);
        por_put(por_row(slot), lane, P);
        em = ez;
        ez = ep;
        if (above && d.moving) moving_wall(P, h);
        collide_pair(d, h, P, o);
    }
    // step l+1 of the row before the one whose step-l values are o
    template <bool W>
    __device__ __forceinline__ void next(int l, const f2 o[9], f2 on[9]) {
        Por P;
        const int back = slot - l < 0 ? slot - l + T : slot - l;
        por_get(por_row(back), lane, P);
        f2 h[9];
        h[0] = mid[l - 1][0];
        h[1] = mid[l - 1][1];
        h[3] = mid[l - 1][2];
        const f2 *u = up_row(l, odd);                  // written two turns ago
        h[2] = u[0 * 32];
        h[5] = u[1 * 32];
        h[6] = u[2 * 32];
        h[4] = o[4];
        h[7] = from_right(o[7]);
        h[8] = from_left(o[8]);
        if (W && d.moving && r - l == d.ny - 1) moving_wall(P, h);
        collide_pair(d, h, P, on);
    }
    // what step l+1 needs later of step l's row o (shifted only now: shifted before
    // next() ran, the new values would need registers beside the old ones)
    __device__ __forceinline__ void keep(int l, const f2 o[9]) {
        f2 *u = up_row(l, odd);
        u[0 * 32] = o[2];
        u[1 * 32] = from_left(o[5]);
        u[2 * 32] = from_right(o[6]);
        mid[l - 1][0] = o[0];
        mid[l - 1][1] = from_left(o[1]);
        mid[l - 1][2] = from_right(o[3]);
    }
    // step T's row y
    __device__ __forceinline__ void store(const f2 o[9]) {
        const long long plane = d.plane;
        char *q = reinterpret_cast<char *>(fout) + out;
        out += (uint32_t)d.pitch * 4u;
        if (!xedge) {
            if (lane >= GL / 2 && lane < 32 - GL / 2) {
#pragma unroll
                for (int i = 0; i < 9; ++i) *reinterpret_cast<f2 *>(q + i * plane * 4) = o[i];
            }
            return;
        }
        if (lane < GL / 2 || lane >= 32 - GL / 2 || x >= d.nx) return;
        float *row = reinterpret_cast<float *>(q);
        const bool both = x + 1 < d.nx;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            row[i * plane] = o[i].x;
            if (both) row[i * plane + 1] = o[i].y;
        }
        if (x == 0) {                                  // column nx mirrors column 0 (e_x < 0)
            row[3 * plane + d.nx] = o[3].x;
            row[6 * plane + d.nx] = o[6].x;
            row[7 * plane + d.nx] = o[7].x;
        }
        if (x + 2 >= d.nx) {                           // column -1 mirrors column nx-1 (e_x > 0)
            float *left = row - x - 1;
            left[1 * plane] = both ? o[1].y : o[1].x;
            left[5 * plane] = both ? o[5].y : o[5].x;
            left[8 * plane] = both ? o[8].y : o[8].x;
        }
    }
    // one turn with steps 1 .. N running (N < T while the wave starts up).  W: a
    // step's row of this turn, or the row loaded for the next, may lie next to a
    // wall or just past one
    template <int N, bool W>
    __device__ __forceinline__ void turn(bool more) {
        f2 o[9];
        first<W>(o);
#pragma unroll
        for (int l = 1; l < T; ++l) {
            if (l > N) break;
            // the next turn's row, before the last step: earlier, the twenty
            // registers it lands in would be live through every step
            if (l == T - 1 && more) prefetch<W>();
            if (W && d.wall_y && r - l + 1 == d.ny) {  // past the upper wall: row ny-1 bounced
                const f2 *u = up_row(l, odd ^ 1);
                o[4] = u[0 * 32];
                o[7] = u[1 * 32];
                o[8] = u[2 * 32];
            }
            f2 on[9];
            if (l < N) next<W>(l, o, on);
            keep(l, o);
            if (W && d.wall_y && r - l + 1 == 0) {     // below the lower wall: row 0 bounced
                f2 *u = up_row(l, odd ^ 1);
                u[0 * 32] = o[4];
                u[1 * 32] = o[7];
                u[2 * 32] = o[8];
            }
            if (l < N) {
#pragma unroll
                for (int i = 0; i < 9; ++i) o[i] = on[i];
            }
        }
        if (N < T - 1 && more) prefetch<W>();
        if (N == T) store(o);
        ++r;
        odd ^= 1;
        if (++slot == T) slot = 0;
    }
    // step l+1 starts two turns after step l: its first row is one further on, and
    // the row before it takes one more
    template <int N>
    __device__ __forceinline__ void start() {
        if constexpr (N < T) {
#pragma unroll 1
            for (int k = 0; k < 2; ++k) turn<N, WALLS>(true);
            start<N + 1>();
        }
    }
    __device__ __forceinline__ void run(int xs) {
        x = xs - GL + 2 * lane;                        // the lane's first column
        inside = xs - GL >= 0 && xs - GL + 64 <= d.nx;
        xedge = xs == 0 || xs + 64 - 2 * GL >= d.nx;
        ia = inside ? x : wrap(x, d.nx);
        second = inside ? 4u : (uint32_t)(wrap(x + 1, d.nx) - ia) * 4u;
        slot = 0;
        odd = 0;
        r = y0 - (T - 1);
        out = ((uint32_t)y0 * (uint32_t)d.pitch + (uint32_t)(d.off + x)) * 4u;
        om = row_off(wrap(r - 1, d.ny));
        oz = row_off(wrap(r, d.ny));
        yp = wrap(r + 1, d.ny);
        op = row_off(yp);
        em = with_neighbours(load(d.eps, om));
        ez = with_neighbours(load(d.eps, oz));
        load_row<WALLS>(r);
#pragma unroll
        for (int l = 1; l < T; ++l)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                mid[l - 1][k] = bc(0.f);
                up_row(l, 0)[k * 32] = up_row(l, 1)[k * 32] = bc(0.f);
            }
        const int last = y1 - 1 + (T - 1);             // row of step 1 in the last turn
        start<1>();
        if constexpr (!WALLS) {
#pragma unroll 1
            while (r <= last) turn<T, false>(r < last);
        } else {
            // near the lower wall, away from walls, near the upper one (a turn also
            // loads row r + 1): one copy of the wall's turn, so that the registers
            // of the plain one are left alone
            int until = min(last, T - 1);
#pragma unroll 1
            for (;;) {
#pragma unroll 1
                while (r <= until) turn<T, true>(r < last);
                if (r > last) break;
#pragma unroll 1
                while (r <= min(last, d.ny - 3)) turn<T, false>(r < last);
                until = last;
            }
        }
    }
};

// shared memory of one warp: T rows of Por, two turns of three pairs for each
// step but the last
template <int T>
__host__ __device__ constexpr int warp_smem() {
    return T * kPorBytes + (T - 1) * 2 * 3 * 8 * 32;
}

// The strip and column block of unit `unit` of a domain cut into ncol x nstrip.
template <int T, bool WALLS, int GL>
__device__ __forceinline__ void run_unit(const VDom &d, const float *fin, float *fout, int unit,
                                         int ncol, int nstrip, unsigned char *smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int strip = unit / ncol, col = unit - strip * ncol;
    unsigned char *ring = smem + warp * warp_smem<T>();
    f2 *up = reinterpret_cast<f2 *>(ring + T * kPorBytes) + lane;
    Strip<T, WALLS, GL> s{d, fin, fout, ring, up};
    s.y0 = (int)((long long)strip * d.ny / nstrip);
    s.y1 = (int)((long long)(strip + 1) * d.ny / nstrip);
    s.lane = lane;
    s.run(col * (64 - 2 * GL));
}

template <int T, bool WALLS>
__global__ void __launch_bounds__(32 * kMultiWarps, 3)
    k_multi(const VDom d, const float *__restrict__ fin, float *__restrict__ fout, int ncol,
            int nstrip) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int unit = blockIdx.x * kMultiWarps + (threadIdx.x >> 5);
    if (unit >= ncol * nstrip) return;
    run_unit<T, WALLS, ghost_cols(T)>(d, fin, fout, unit, ncol, nstrip, smem);
}

// Batched: block b takes four consecutive units of one domain, table entry {dom,
// first unit, column blocks, strips}.  GL: ghost columns that the table was built
// for (a remainder of fewer steps runs on the table of the full launches).
template <int T, int GL>
__global__ void __launch_bounds__(32 * kMultiWarps, 3)
    k_multi_batched(const VDom *__restrict__ doms, const Tile *__restrict__ tiles, int parity) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ VDom d;
    const Tile t = tiles[blockIdx.x];
    for (int k = threadIdx.x; k < (int)(sizeof(VDom) / 4); k += blockDim.x)
        reinterpret_cast<int *>(&d)[k] = reinterpret_cast<const int *>(doms + t.dom)[k];
    __syncthreads();
    const int unit = t.row + (threadIdx.x >> 5);
    if (unit >= t.x0 * t.pad) return;
    run_unit<T, true, GL>(d, parity ? d.f[1] : d.f[0], parity ? d.f[0] : d.f[1], unit, t.x0, t.pad,
                          smem);
}

// SMs and blocks per SM of a kernel, its shared memory allowed for: asked for once
// per device, not at every launch (a run's first pass captures up to 126 launches;
// the four queries cost several us each).
struct Prepared {
    static constexpr int kDevices = 64;
    std::atomic<int> sms_[kDevices] = {}, occ_[kDevices] = {};      // 0: not asked yet
    cudaError_t get(const void *kern, size_t smem, int &sms, int &occ) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kDevices) return cudaErrorInvalidDevice;
        occ = occ_[dev].load(std::memory_order_acquire);
        if (occ > 0) {
            sms = sms_[dev].load(std::memory_order_relaxed);
            return cudaSuccess;
        }
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 32 * kMultiWarps, smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        sms_[dev].store(sms, std::memory_order_relaxed);
        occ_[dev].store(occ, std::memory_order_release);
        return cudaSuccess;
    }
    template <class K> cudaError_t get(K *kern, size_t smem, int &sms, int &occ) {
        return get((const void *)kern, smem, sms, occ);
    }
};

template <int T, bool WALLS>
Prepared &prepared() {
    static Prepared ready;
    return ready;
}

// Strips per column block: the count with the smallest waves x turns (a strip
// of n rows takes n + 2 (T-1) turns, and its start is worth one more), a wave
// being as many warps as the chip holds, or ctas blocks per SM in one wave:
// fewer and longer strips repeat fewer rows, which is the better choice where
// short strips would be half repetition (512^2, T = 2: 4.09 us per step with
// 3 blocks per SM, 3.85 with 2).  The search takes up to ny turns of the host (three launches
// of 96 x 20000: 95 us of it, now 6.5), so a handle makes it when its shape is set.
template <int T, bool WALLS>
cudaError_t strips_t(const VDom &d, int ctas, int *strips) {
    int sms = 0, occ = 0;
    const cudaError_t e =
        prepared<T, WALLS>().get(k_multi<T, WALLS>, (size_t)kMultiWarps * warp_smem<T>(), sms, occ);
    if (e != cudaSuccess) return e;
    const int ncol = (d.nx + out_cols(T) - 1) / out_cols(T);
    const long long resident = (long long)sms * (ctas > 0 && ctas < occ ? ctas : occ) * kMultiWarps;
    *strips = 1;
    double best = 1e300;
    for (int s = 1; s <= d.ny; ++s) {
        const long long units = (long long)ncol * s;
        const long long waves = (units + resident - 1) / resident;
        const double cost = (double)waves * ((d.ny + s - 1) / s + 2 * (T - 1) + 1);
        if (cost < best) {
            best = cost;
            *strips = s;
        }
        if (units > (ctas > 0 ? 1 : 8) * resident) break;
    }
    return cudaSuccess;
}

template <int T, bool WALLS>
cudaError_t launch_multi_t(const VDom &d, const float *fin, float *fout, int strips,
                           cudaStream_t stream) {
    int sms = 0, occ = 0;
    const size_t smem = (size_t)kMultiWarps * warp_smem<T>();
    const cudaError_t e = prepared<T, WALLS>().get(k_multi<T, WALLS>, smem, sms, occ);
    if (e != cudaSuccess) return e;
    const int ncol = (d.nx + out_cols(T) - 1) / out_cols(T);
    const long long grid = ((long long)ncol * strips + kMultiWarps - 1) / kMultiWarps;
    if (strips < 1 || strips > d.ny || grid > 0x7fffffffLL / kMultiWarps) return cudaErrorInvalidConfiguration;
    k_multi<T, WALLS><<<(unsigned)grid, 32 * kMultiWarps, smem, stream>>>(d, fin, fout, ncol, strips);
    return cudaGetLastError();
}

}  // namespace

template <int T, int GL>
static cudaError_t launch_batched_t(const VDom *doms, const Tile *tiles, int ntiles, int parity,
                                    cudaStream_t stream) {
    auto kern = k_multi_batched<T, GL>;
    static Prepared ready;
    int sms = 0, occ = 0;
    const size_t smem = (size_t)kMultiWarps * warp_smem<T>();
    const cudaError_t e = ready.get(kern, smem, sms, occ);
    if (e != cudaSuccess) return e;
    kern<<<ntiles, 32 * kMultiWarps, smem, stream>>>(doms, tiles, parity);
    return cudaGetLastError();
}

int multi_out_cols(int steps) { return out_cols(steps); }

cudaError_t launch_multi_batched(const VDom *doms, const Tile *tiles, int ntiles, int parity,
                                 int table_steps, int steps, cudaStream_t stream) {
    if (ntiles < 1) return cudaErrorInvalidValue;
    if (table_steps == 2 && steps == 2) return launch_batched_t<2, 2>(doms, tiles, ntiles, parity, stream);
    if (table_steps < 3) return cudaErrorInvalidValue;
    switch (steps) {
        case 2: return launch_batched_t<2, 4>(doms, tiles, ntiles, parity, stream);
        case 3: return launch_batched_t<3, 4>(doms, tiles, ntiles, parity, stream);
        case 4: return launch_batched_t<4, 4>(doms, tiles, ntiles, parity, stream);
    }
    return cudaErrorInvalidValue;
}

bool multi_fits(int q, const VDom &d) {
    // byte offsets within a plane are 32-bit
    return q == 9 && !d.nee && d.xwrap && d.plane < (1LL << 30);
}

cudaError_t multi_strips(const VDom &d, int steps, int ctas, int *strips) {
    switch (steps) {
        case 2: return d.wall_y ? strips_t<2, true>(d, ctas, strips) : strips_t<2, false>(d, ctas, strips);
        case 3: return d.wall_y ? strips_t<3, true>(d, ctas, strips) : strips_t<3, false>(d, ctas, strips);
        case 4: return d.wall_y ? strips_t<4, true>(d, ctas, strips) : strips_t<4, false>(d, ctas, strips);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_multi(const VDom &d, const float *fin, float *fout, int steps, int strips,
                         cudaStream_t stream) {
    if (!multi_fits(9, d)) return cudaErrorInvalidValue;
    switch (steps) {
        case 2: return d.wall_y ? launch_multi_t<2, true>(d, fin, fout, strips, stream)
                                : launch_multi_t<2, false>(d, fin, fout, strips, stream);
        case 3: return d.wall_y ? launch_multi_t<3, true>(d, fin, fout, strips, stream)
                                : launch_multi_t<3, false>(d, fin, fout, strips, stream);
        case 4: return d.wall_y ? launch_multi_t<4, true>(d, fin, fout, strips, stream)
                                : launch_multi_t<4, false>(d, fin, fout, strips, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace vans
