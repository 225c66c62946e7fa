// vans_cluster.cu -- many steps in one launch for domains that fit in the
// shared memory of one thread-block cluster (launch kind 8).
//
// A small domain (the 128x64 channel, the 80x80 Couette case) is a few
// hundred KB of populations: one step is a few microseconds of launch
// overhead around less than a microsecond of work.  Here one cluster of up to
// 16 CTAs holds the whole state in its distributed shared memory for the
// whole run: CTA k owns a band of consecutive rows (row = z * ny + y) and keeps
// two copies of its band, the populations the step reads and the ones it
// writes, each row with its halo columns -1 and nx.  A step is the same pull,
// collision and store as every other kernel here (the functions of
// vans_device.cuh, so the same arithmetic); a pull that crosses into another
// band reads the owning CTA's shared memory through the cluster's
// distributed shared memory window.  One cluster barrier per step separates
// the writes of step t from the reads of step t + 1; because the two copies
// alternate, the writes of step t + 1 (into the copy read at step t) also
// come after every read of step t.  The band is loaded from the state buffer
// `fin` at the start and written back to `fout` at the end (columns -1 .. nx
// of every row and direction, the library's padded layout).
//
// D2Q9 domains that fit take a second form, k_step_cluster_pair: two adjacent cells
// per thread in packed arithmetic, the edge rows pushed to the neighbour instead of
// pulled, no cluster barrier (0.547 us per step instead of 1.01 on the 128x64 channel).
// The form above stays for D3Q19, for shapes that do not fit, and for the forward
// steps of a reverse pass, which round as the single-step kernels do.
#include <cooperative_groups.h>

#include <type_traits>

#include "vans_pair.cuh"
#include "vans_tma.cuh"

namespace cg = cooperative_groups;

namespace vans {

namespace {

constexpr int kClusterMax = 16;
constexpr int kClusterSmemMax = 227 * 1024;

// floats per row copy in shared memory: columns -1 .. nx, rounded up to 4
__host__ __device__ inline int cluster_row_floats(int nx) { return (nx + 2 + 3) & ~3; }

// cells per thread at most: D2Q9 2, D3Q19 1 (its 19 addresses and porosities
// per cell stay in registers for the whole launch)
template <int Q> struct CellsMax { static constexpr int N = (Q == 9) ? 2 : 1; };

// Address, in the cluster's shared-memory window, of `local` (a shared-memory
// address of this CTA) in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const float *local, int rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ float ld_cluster(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" :: "r"(addr), "f"(v) : "memory");
}

}  // namespace

// Every thread keeps at most CellsMax<Q>::N cells of its CTA's band for the
// whole launch.  What a cell's update needs besides the populations does not
// change from step to step, so it is formed once, before the first step: the
// address (in the cluster's shared-memory window, so in the shared memory of
// the CTA that owns the row) of each of the Q entries its pull reads, and its
// own and its neighbours' porosities.  A step is then Q loads, the collision
// and Q stores per cell.
// PL (plates on nodes, wall_kind 1): rows 0 and ny-1 are plate nodes and are
// not stepped; the fluid row next to a plate writes the plate node's inward
// populations (f^eq of the plate plus this cell's non-equilibrium part,
// relaxed), as the other step kernels do, into the plate row's entries, which
// may lie in the neighbouring CTA's band (a store through the cluster window).
template <int Q, int NT, bool PL>
__global__ void __launch_bounds__(NT) k_step_cluster(const VDom d, const float *fin, float *fout,
                                                     int nsteps, int band) {
    using L = Lat<Q>;
    constexpr int kCellsMax = CellsMax<Q>::N;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int sp = cluster_row_floats(d.nx);
    const long long copy = (long long)Q * band * sp;     // floats of one copy of a band
    extern __shared__ __align__(16) float sm[];
    const int r0 = rank * band;
    const int nr = max(0, min(band, d.rows - r0));
    const int nx = d.nx;

    // the band's rows of the state buffer, columns -1 .. nx
    for (long long t = threadIdx.x; t < (long long)Q * nr * (nx + 2); t += NT) {
        const int c = (int)(t % (nx + 2));
        const long long pr = t / (nx + 2);
        const int rl = (int)(pr % nr), i = (int)(pr / nr);
        sm[((long long)i * band + rl) * sp + c] =
            fin[i * d.plane + (long long)(r0 + rl) * d.pitch + d.off - 1 + c];
    }

    // per cell, fixed for the launch: pull addresses (copy 0), porosities,
    // the row offset of its stores, and whether it sits under a moving wall
    uint32_t src[kCellsMax][Q];
    float e0[kCellsMax], et[kCellsMax][Q];
    int dst[kCellsMax], xs[kCellsMax];
    bool top[kCellsMax], live[kCellsMax];
    Nb3 Zs[kCellsMax];
    // plates on nodes: sides (bit 0 the plate below, bit 1 the plate above:
    // both for the one fluid row between plates 2 rows apart), and each plate
    // row's entry of this column (copy 0, plane 0, cluster window)
    int pside[kCellsMax];
    uint32_t pdst[kCellsMax][2];
#pragma unroll
    for (int k = 0; k < kCellsMax; ++k) {
        const int t = threadIdx.x + k * NT;
        live[k] = t < nr * nx;
        const int tt = live[k] ? t : 0;
        const int rl = tt / nx, x = tt - rl * nx;
        const int r = r0 + rl, y = r % d.ny, z = r / d.ny;
        pside[k] = 0;
        pdst[k][0] = pdst[k][1] = 0;
        if (PL) {
            if (y == 0 || y == d.ny - 1) live[k] = false;          // plate node: not stepped
            if (live[k]) {
                pside[k] = (y == 1 ? 1 : 0) | (y == d.ny - 2 ? 2 : 0);
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (!(pside[k] & (1 << side))) continue;
                    const int rp = side == 0 ? r - 1 : r + 1, owner = rp / band;
                    pdst[k][side] =
                        cluster_addr(sm + (long long)(rp - owner * band) * sp + 1 + x, owner);
                }
            }
        }
        const Nb3 Y = nb3<true>(y, d.ny, d.wall_y);
        Nb3 Z;
        if (Q == 19) {
            Z = nb3<true>(z, d.nz, d.wall_z);
        } else {
            Z.r[0] = Z.r[1] = Z.r[2] = 0;
            Z.wall[0] = Z.wall[1] = Z.wall[2] = false;
        }
        Zs[k] = Z;
        top[k] = Y.wall[2];
        xs[k] = x;
        dst[k] = rl * sp + 1 + x;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            // the entry at x - e_i of row (y - e_y, z - e_z), or the opposite
            // direction of this cell past a wall; that row lives in the band
            // of CTA row / band
            const int ey = L::ey(i), ez = L::ez(i);
            const bool bb = Y.wall[1 - ey] || Z.wall[1 - ez];
            const int sr = bb ? r : Z.r[1 - ez] * d.ny + Y.r[1 - ey];
            const int owner = sr / band;
            const int plane = bb ? L::opp(i) : i;
            const int col = bb ? x : x - L::ex(i);
            src[k][i] = cluster_addr(sm + ((long long)plane * band + (sr - owner * band)) * sp +
                                         col + 1, owner);
        }
        e0[k] = live[k] ? __ldg(d.eps + row_offset(d, y, z) + x) : 1.f;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const bool wall = Y.wall[1 + L::ey(i)] || Z.wall[1 + L::ez(i)];
            et[k][i] = (i == 0 || wall || !live[k])
                           ? e0[k]
                           : __ldg(d.eps + row_offset(d, Y.r[1 + L::ey(i)], Z.r[1 + L::ez(i)]) + x +
                                   L::ex(i));
        }
    }
    cl.sync();

    int b = 0;
    for (int s = 0; s < nsteps; ++s) {
        const uint32_t cur = (uint32_t)(b * copy * sizeof(float));   // the copy read this step
        float *nxt = sm + (b ^ 1) * copy;
#pragma unroll
        for (int k = 0; k < kCellsMax; ++k) {
            if (!live[k]) continue;
            float h[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) h[i] = ld_cluster(src[k][i] + cur);
            apply_moving_wall<Q>(d, top[k], Zs[k], e0[k], h);
            float o[Q];
            Macro<Q> M;
            collide<Q>(d, h, e0[k], et[k], o, (PL && pside[k]) ? &M : nullptr);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                float *row = nxt + (long long)i * band * sp + dst[k];   // this cell's column
                row[0] = o[i];
                if (xs[k] == 0 && L::ex(i) < 0) row[nx] = o[i];         // halo copies of the wrap
                if (xs[k] == nx - 1 && L::ex(i) > 0) row[-nx] = o[i];
            }
            if (PL && pside[k]) {
                // the plate node's populations toward this row: e_y > 0 from
                // the plate below, e_y < 0 from the plate above, each stored
                // against the porosity of the row cell it streams to
                constexpr int jym = dir_index<Q>(0, -1, 0), jyp = dir_index<Q>(0, 1, 0);
                constexpr int jxp = dir_index<Q>(1, 0, 0), jxm = dir_index<Q>(-1, 0, 0);
                constexpr int jzp = dir_index<Q>(0, 0, 1), jzm = dir_index<Q>(0, 0, -1);
                const float om1 = 1.f - d.omega, zero[3] = {0.f, 0.f, 0.f};
                const uint32_t next = (uint32_t)((b ^ 1) * copy * sizeof(float));
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const int ey = L::ey(i);
                    if (ey == 0 || !(pside[k] & (ey > 0 ? 1 : 2))) continue;
                    const bool lo = ey > 0;
                    const int ex = L::ex(i), ez = L::ez(i);
                    const float enb = ex > 0 ? et[k][jxp] : ex < 0 ? et[k][jxm]
                                    : ez > 0 ? et[k][jzp] : ez < 0 ? et[k][jzm] : e0[k];
                    const float v = plate_value<Q>(d, i, h[i], M, lo ? et[k][jym] : et[k][jyp], enb,
                                                   lo ? zero : d.uw, om1);
                    const uint32_t a = pdst[k][lo ? 0 : 1] + next +
                                       (uint32_t)((long long)i * band * sp * sizeof(float));
                    st_cluster(a, v);
                    if (xs[k] == 0 && ex < 0) st_cluster(a + (uint32_t)(nx * sizeof(float)), v);
                    if (xs[k] == nx - 1 && ex > 0) st_cluster(a - (uint32_t)(nx * sizeof(float)), v);
                }
            }
        }
        cl.sync();
        b ^= 1;
    }

    const float *res = sm + b * copy;
    for (long long t = threadIdx.x; t < (long long)Q * nr * (nx + 2); t += NT) {
        const int c = (int)(t % (nx + 2));
        const long long pr = t / (nx + 2);
        const int rl = (int)(pr % nr), i = (int)(pr / nr);
        fout[i * d.plane + (long long)(r0 + rl) * d.pitch + d.off - 1 + c] =
            res[((long long)i * band + rl) * sp + c];
    }
}

// ------------------------------------------------ D2Q9, a pair per thread ----
// The D2Q9 form.  A thread owns two adjacent cells of its CTA's band for the whole
// launch (packed arithmetic, vans_pair.cuh), with its porosity terms and the
// shared-memory address of each of the 18 entries its pulls read in registers.  A
// band keeps one row of its neighbours' above and below its own, so that every
// pull is a local load: the CTA that steps an edge row sends the three populations
// per cell that cross it into the neighbour's row with st.async, which also counts
// the bytes on the neighbour's mbarrier, and only the warps of the neighbour's edge
// row wait for them.  Within the CTA one __syncthreads separates the steps; there
// is no cluster-wide barrier in the loop.
//
// A step is a chain of latencies: the neighbours' rows on their way (about 700
// cycles per step with the arithmetic taken out), the update of a pair (350 cycles
// alone on a scheduler, vans_multi.cu), the loads, stores and the barrier (0.39 us
// per step without any exchange).  128x64 on 16 CTAs of 8 warps 0.547 us per step,
// the 80x81 Couette case between plates on nodes 0.632 (the form above, one cell
// per thread, pulls through the cluster window and a cluster barrier per step: 1.006
// and 1.07).  It takes D2Q9 domains whose pairs find a thread each and whose copies
// fit; the form above takes the rest and D3Q19.
//
// The entries sent in step s go to copy s+1 mod 2 and are counted on the barrier of
// that copy; those of step s+2 are only sent after the neighbour has received all
// that this CTA's edge row sent in step s+1, and that row has read the entries of
// step s by then, so two copies and two barriers per side suffice.

constexpr int kPairCopy = 113 * 1024;           // bytes from one copy of the band to the other
constexpr int kPairBars = 64;                   // the barriers, in front of the copies

// A row, columns -1 .. nx, is kept as its even columns followed by its odd ones,
// pair_half floats each: the lanes of a warp, one per pair, read and write
// consecutive words whichever way a population moves (interleaved, every 4-byte
// access of a pair's half was a two-way bank conflict, 36 instead of 18 shared-memory
// cycles per warp and step for the pulls).
__host__ __device__ inline int pair_half(int nx) { return nx / 2 + 2; }
__host__ __device__ inline int pair_row_floats(int nx) { return 2 * pair_half(nx); }

// bytes of one copy: 9 planes of the band's rows and one beyond it on either side
inline long long pair_copy_bytes(const VDom &d, int band) {
    return 9LL * (band + 2) * pair_row_floats(d.nx) * (long long)sizeof(float);
}

__device__ __forceinline__ float lds(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
// store into another CTA's shared memory that counts 4 bytes on that CTA's barrier
__device__ __forceinline__ void st_async(uint32_t a, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a),
                 "f"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t a, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// What a plate node (wall_kind 1) sends into its fluid neighbour's row: plate_value
// of vans_device.cuh for the three inward directions of a pair of columns.
// ebi = eps_b / eps, eb the plate's porosity, df[k] = eps_b - eps of the cell the
// k-th direction streams to; ub the plate's velocity; dirs the inward directions.
__device__ __forceinline__ f2 plate_pair(int i, f2 h, const PairMoments &m, f2 ebi, f2 df,
                                         const float ub[3], float om1) {
    using L = Lat<9>;
    const f2 eu = fma2(bc((float)L::ex(i)), m.ux, mul2(bc((float)L::ey(i)), m.uy));
    const f2 uu = fma2(m.ux, m.ux, mul2(m.uy, m.uy));
    const f2 A = fma2(bc(3.f), eu, fma2(bc(4.5f), mul2(eu, eu), mul2(bc(-1.5f), uu)));
    const float B = eq_bracket<9>(i, ub);
    const f2 neq = fma2(bc(-L::w(i)), fma2(m.R, A, m.dl), h);
    const f2 eq = add2(df, mul2(ebi, fma2(m.R, bc(B), m.dl)));
    return fma2(bc(om1), neq, mul2(bc(L::w(i)), eq));
}

template <int NT, bool PL>
__global__ void __launch_bounds__(NT) k_step_cluster_pair(const VDom d, const float *fin, float *fout,
                                                          int nsteps, int band) {
    using L = Lat<9>;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
    const int nx = d.nx, ny = d.ny, half = pair_half(nx), sp = 2 * half;
    const int r0 = rank * band, nr = max(0, min(band, ny - r0));
    extern __shared__ __align__(16) unsigned char smem[];
    // barriers [side][copy]: side 0 the row below the band, 1 the row above it
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    const uint32_t base = smem_addr(smem) + kPairBars;
    // address (copy 0) of column c of local row rl (-1 .. band) of plane i
    auto at = [&](int i, int rl, int c) {
        return base + (uint32_t)(((i * (band + 2) + rl + 1) * sp + ((c + 2) >> 1) + (c & 1 ? half : 0)) * 4);
    };
    const bool periodic = !d.wall_y;
    const int below = r0 > 0 ? r0 - 1 : ny - 1;                 // row under the band
    const int above = r0 + nr < ny ? r0 + nr : 0;               // row over it
    const bool has_below = nr > 0 && (r0 > 0 || periodic), has_above = nr > 0 && (r0 + nr < ny || periodic);
    auto dead = [&](int y) { return PL && (y == 0 || y == ny - 1); };   // plate nodes

    const int npx = (nx + 1) / 2;
    const uint32_t row_bytes = (uint32_t)(3 * 2 * npx) * 4u;    // what a neighbour sends per step
    const bool recv_lo = has_below && !dead(below) && !dead(r0);
    const bool recv_hi = has_above && !dead(above) && !dead(r0 + nr - 1);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 4; ++k) mbar_init(&bars[k], 1);
        mbar_init_fence();
        for (int k = 0; k < 2; ++k) {
            if (recv_lo) mbar_arrive_expect_tx(&bars[k], row_bytes);
            if (recv_hi) mbar_arrive_expect_tx(&bars[2 + k], row_bytes);
        }
    }

    // the band and the rows beside it, columns -1 .. nx, into copy 0
    const int w = nx + 2;
    for (int t = threadIdx.x; t < 9 * (nr + 2) * w; t += NT) {
        const int c = t % w, pr = t / w, rl = pr % (nr + 2) - 1, i = pr / (nr + 2);
        if ((rl < 0 && !has_below) || (rl == nr && !has_above)) continue;
        const int y = rl < 0 ? below : rl == nr ? above : r0 + rl;
        sts(at(i, rl, c - 1), fin[i * d.plane + (long long)y * d.pitch + d.off - 1 + c]);
    }

    const int rl = threadIdx.x / npx, x = 2 * (threadIdx.x - rl * npx), y = r0 + rl;
    const bool live = rl < nr && !dead(y);
    // an odd row's last pair is one cell and a copy of it, which goes to the unused
    // column nx
    const int x1 = x + 1 < nx ? x + 1 : x;
    uint32_t a0[9], a1[9];
    Por P = {};
    const bool top = d.wall_y && !d.nee && y == ny - 1, bottom = d.wall_y && !d.nee && y == 0;
    const bool plate_lo = PL && live && y == 1, plate_hi = PL && live && y == ny - 2;
    f2 ebi[2], df[2][3];                                        // plates below, above
    f2 gain[3];                                                 // of the moving wall: 4, 7, 8
    if (live) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const bool bb = (bottom && L::ey(i) > 0) || (top && L::ey(i) < 0);
            const int plane = bb ? L::opp(i) : i, row = bb ? rl : rl - L::ey(i), dx = bb ? 0 : L::ex(i);
            // periodic x: from the row's other end; a slab (one step per call): the
            // halo columns
            auto column = [&](int c) { return !d.xwrap ? c : c < 0 ? nx - 1 : c >= nx ? 0 : c; };
            a0[i] = at(plane, row, column(x - dx));
            a1[i] = at(plane, row, column(x1 - dx));
        }
        const int ym = y > 0 ? y - 1 : ny - 1, yp = y < ny - 1 ? y + 1 : 0;
        auto eps_row = [&](int yy) {
            const float *e = d.eps + row_offset(d, yy, 0);
            return Row{e[x - 1], make_float2(e[x], e[x + 1]), e[x1 + 1]};
        };
        const Row m = eps_row(ym), z = eps_row(y), p = eps_row(yp);
        porosity_terms(d, m, z, p, bottom, top, P);
        gain[0] = mul2(P.e0, bc(wall_gain<9>(d, 4, 1.f)));
        gain[1] = mul2(P.e0, bc(wall_gain<9>(d, 7, 1.f)));
        gain[2] = mul2(P.e0, bc(wall_gain<9>(d, 8, 1.f)));
        if (PL) {
            const f2 inv = rcp2(P.e0);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const f2 eb = s ? p.c : m.c;
                ebi[s] = mul2(eb, inv);
                df[s][0] = sub2(eb, z.c);
                df[s][1] = sub2(eb, z.right());
                df[s][2] = sub2(eb, z.left());
            }
        }
    }
    // the neighbours' rows that this thread's edge rows are sent to: e_y < 0 of the
    // band's first row go into the row above the band below, e_y > 0 of the last
    // row into the row below the band above
    const int lower = rank > 0 ? rank - 1 : ctas - 1, upper = rank < ctas - 1 ? rank + 1 : 0;
    const int lower_rows = min(band, ny - lower * band);
    const bool send_lo = live && rl == 0 && has_below && !dead(below);
    const bool send_hi = live && rl == nr - 1 && has_above && !dead(above);
    const bool wait_lo = rl == 0 && recv_lo, wait_hi = rl == nr - 1 && recv_hi;
    const uint32_t to_lo = map_rank(at(0, lower_rows, x), lower), to_hi = map_rank(at(0, -1, x), upper);
    const uint32_t bar_lo = map_rank(smem_addr(&bars[2]), lower), bar_hi = map_rank(smem_addr(&bars[0]), upper);
    const uint32_t plane_bytes = (uint32_t)((band + 2) * sp * 4);
    const uint32_t own = at(0, min(rl, nr), x);
    const uint32_t dnext = (uint32_t)half * 4;                  // from column x to column x + 1
    cl.sync();

    bool late = false;
    // one step from copy FROM (0 or 1) to the other; phase: of the copy's barriers
    auto step = [&](auto from, uint32_t phase, bool wait, bool send) {
        constexpr int kF = decltype(from)::value, kT = 1 - kF;
        constexpr uint32_t FROM = kF * kPairCopy, TO = kT * kPairCopy;
        if (wait) {
            // a thread that gave up once waits no more: the run ends with garbage
            // and the status word set
            if (wait_lo) {
                late = late || !mbar_wait_bounded<true>(&bars[kF], phase);
                if (x == 0) mbar_arrive_expect_tx(&bars[kF], row_bytes);       // for two steps on
            }
            if (wait_hi) {
                late = late || !mbar_wait_bounded<true>(&bars[2 + kF], phase);
                if (x == 0) mbar_arrive_expect_tx(&bars[2 + kF], row_bytes);
            }
        }
        if (live) {
            f2 h[9], o[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = make_float2(lds(a0[i] + FROM), lds(a1[i] + FROM));
            if (top && d.moving) {
                h[4] = add2(h[4], gain[0]);
                h[7] = add2(h[7], gain[1]);
                h[8] = add2(h[8], gain[2]);
            }
            PairMoments mom;
            collide_pair(d, h, P, o, PL && (plate_lo || plate_hi) ? &mom : nullptr);
            auto put = [&](uint32_t row, f2 v) {
                sts(row, v.x);
                sts(row + dnext, v.y);
            };
            auto push = [&](uint32_t row, f2 v, uint32_t bar) {
                st_async(row, v.x, bar);
                st_async(row + dnext, v.y, bar);
            };
            if (send && send_lo) {
#pragma unroll
                for (int i : {4, 7, 8}) push(to_lo + i * plane_bytes + TO, o[i], bar_lo + 8 * kT);
            }
            if (send && send_hi) {
#pragma unroll
                for (int i : {2, 5, 6}) push(to_hi + i * plane_bytes + TO, o[i], bar_hi + 8 * kT);
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) put(own + i * plane_bytes + TO, o[i]);
            if (PL && (plate_lo || plate_hi)) {
                // the plate node's inward populations, kept in this band's own
                // copy of the plate's row
                const float om1 = 1.f - d.omega, zero[3] = {0.f, 0.f, 0.f};
                const uint32_t dn = own - sp * 4 + TO, over = own + sp * 4 + TO;
                if (plate_lo) {
                    put(dn + 2 * plane_bytes, plate_pair(2, h[2], mom, ebi[0], df[0][0], zero, om1));
                    put(dn + 5 * plane_bytes, plate_pair(5, h[5], mom, ebi[0], df[0][1], zero, om1));
                    put(dn + 6 * plane_bytes, plate_pair(6, h[6], mom, ebi[0], df[0][2], zero, om1));
                }
                if (plate_hi) {
                    put(over + 4 * plane_bytes, plate_pair(4, h[4], mom, ebi[1], df[1][0], d.uw, om1));
                    put(over + 8 * plane_bytes, plate_pair(8, h[8], mom, ebi[1], df[1][1], d.uw, om1));
                    put(over + 7 * plane_bytes, plate_pair(7, h[7], mom, ebi[1], df[1][2], d.uw, om1));
                }
            }
        }
        __syncthreads();
    };
    // copy 0 is read by steps 0, 2, ..: step 0 reads what was loaded, step s the
    // entries of step s-1; a copy's barriers complete once per use
    uint32_t ph0 = 0, ph1 = 0;
    for (int s = 0; s < nsteps; ++s) {
        if ((s & 1) == 0) {
            step(std::integral_constant<int, 0>{}, ph0, s > 0, s + 1 < nsteps);
            if (s > 0) ph0 ^= 1u;
        } else {
            step(std::integral_constant<int, 1>{}, ph1, true, s + 1 < nsteps);
            ph1 ^= 1u;
        }
    }
    if (late && d.status) atomicOr(d.status, 2);

    const uint32_t res = (nsteps & 1) ? kPairCopy : 0;
    for (int t = threadIdx.x; t < 9 * nr * w; t += NT) {
        const int c = t % w, pr = t / w, rr = pr % nr, i = pr / nr, yy = r0 + rr;
        if ((c == 0 && L::ex(i) <= 0) || (c == nx + 1 && L::ex(i) >= 0)) continue;   // no halo copy
        // a plate node's inward entries are those of the band that steps its neighbour
        if (PL && ((yy == 0 && L::ey(i) > 0) || (yy == ny - 1 && L::ey(i) < 0))) continue;
        const bool keep = PL && dead(yy);       // never written: as loaded
        // (column nx mirrors column 0 and column -1 column nx-1)
        const int cc = c == 0 ? nx - 1 : c == nx + 1 ? 0 : c - 1;
        fout[i * d.plane + (long long)yy * d.pitch + d.off - 1 + c] =
            lds(at(i, rr, cc) + (keep ? 0 : res));
    }
    if (PL)
        for (int t = threadIdx.x; t < 6 * w; t += NT) {
            const int c = t % w, k = t / w, hi = k >= 3;
            const int i = hi ? (k == 3 ? 4 : k + 3) : (k == 0 ? 2 : k + 4);    // 2 5 6, 4 7 8
            const int yf = hi ? ny - 2 : 1, rr = yf - r0;
            if (rr < 0 || rr >= nr) continue;
            if ((c == 0 && L::ex(i) <= 0) || (c == nx + 1 && L::ex(i) >= 0)) continue;
            const int cc = c == 0 ? nx - 1 : c == nx + 1 ? 0 : c - 1;
            fout[i * d.plane + (long long)(hi ? ny - 1 : 0) * d.pitch + d.off - 1 + c] =
                lds(at(i, hi ? rr + 1 : rr - 1, cc) + res);
        }
    cl.sync();          // no CTA leaves while another may still send to it
}

// Rows per CTA and CTAs of the cluster for a cluster of at most cmax CTAs.
static void cluster_shape(const VDom &d, int cmax, int &band, int &ctas) {
    band = (d.rows + cmax - 1) / cmax;
    ctas = (d.rows + band - 1) / band;
}

// whether the pair form takes the domain (not rows of one cell, whose pairs are half
// empty: 200 of them 0.78 us per step, 0.75 by the other form)
static bool pair_fits(int q, const VDom &d, int cmax, int warps) {
    if (q != 9 || d.nx < 2) return false;
    int band = 0, ctas = 0;
    cluster_shape(d, cmax, band, ctas);
    return (long long)band * ((d.nx + 1) / 2) <= 32 * warps && pair_copy_bytes(d, band) <= kPairCopy;
}

size_t cluster_smem_bytes(int q, const VDom &d, int cmax) {
    int band = 0, ctas = 0;
    cluster_shape(d, cmax, band, ctas);
    return 2 * (size_t)q * band * cluster_row_floats(d.nx) * sizeof(float);
}

bool cluster_fits(int q, const VDom &d, int cmax, int warps) {
    if (cmax < 1 || cmax > kClusterMax) return false;
    int band = 0, ctas = 0;
    cluster_shape(d, cmax, band, ctas);
    const int cells_max = (q == 9) ? CellsMax<9>::N : CellsMax<19>::N;
    if ((long long)band * d.nx > (long long)cells_max * 32 * warps) return false;
    return cluster_smem_bytes(q, d, cmax) <= (size_t)kClusterSmemMax;
}

template <int Q, int NT>
static cudaError_t launch_cluster_t(const VDom &d, const float *fin, float *fout, int nsteps,
                                    int cmax, bool pairs, cudaStream_t stream) {
    int band = 0, ctas = 0;
    cluster_shape(d, cmax, band, ctas);
    const bool pair = pairs && pair_fits(Q, d, cmax, NT / 32);
    const size_t smem = pair ? kPairBars + kPairCopy + (size_t)pair_copy_bytes(d, band)
                             : cluster_smem_bytes(Q, d, cmax);
    const void *kern = pair ? (d.nee ? (const void *)k_step_cluster_pair<NT, true>
                                     : (const void *)k_step_cluster_pair<NT, false>)
                            : (d.nee ? (const void *)k_step_cluster<Q, NT, true>
                                     : (const void *)k_step_cluster<Q, NT, false>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (ctas > 8) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    e = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg);
    if (e != cudaSuccess) return e;
    if (nclusters < 1) return cudaErrorInvalidConfiguration;
    void *args[] = {(void *)&d, &fin, &fout, &nsteps, &band};
    e = cudaLaunchKernelExC(&cfg, kern, args);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// kind 8: `warps` warps per CTA (8 or 16), `rows` = the largest cluster (2..16)
cudaError_t launch_step_cluster(int q, const VDom &d, const float *fin, float *fout, int nsteps,
                                Launch L, bool pairs, cudaStream_t stream) {
    if (nsteps < 1) return cudaErrorInvalidValue;
    if (!cluster_fits(q, d, L.rows, L.warps)) return cudaErrorInvalidValue;
    if (q == 9) {
        if (L.warps == 8) return launch_cluster_t<9, 256>(d, fin, fout, nsteps, L.rows, pairs, stream);
        if (L.warps == 16) return launch_cluster_t<9, 512>(d, fin, fout, nsteps, L.rows, pairs, stream);
    } else if (q == 19) {
        if (L.warps == 8) return launch_cluster_t<19, 256>(d, fin, fout, nsteps, L.rows, pairs, stream);
        if (L.warps == 16) return launch_cluster_t<19, 512>(d, fin, fout, nsteps, L.rows, pairs, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace vans
