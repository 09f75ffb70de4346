// sw_potts.cu -- the q-state Potts model on 2D and 3D lattices
// (sw_create_potts, pcc_create_potts in include/swgpu.h): the cluster update
// of Sec. I with "equal spins" read as "equal states", on the d-dimensional
// lattice the paper states its method for (Sec. II), split as the 2D Ising
// sweep of sw_device.cuh is (Sec. II.A's slaves and master inside one GPU):
//
//   k_ptile   one CTA per tile (128 x 64 sites in 2D, 32 x 16 x 16 in 3D).
//             It finishes sweep k-1 (each site's 2-byte tile-local cluster
//             code, the border clusters' new states from the merged node
//             table, the halo from the neighbours' tables, the observables)
//             and starts sweep k on those states, which stay in shared
//             memory: Philox bonds between equal states, a shared-memory
//             union-find over the bonds inside the tile, the new state of
//             every cluster that ends inside the tile, one node per site of
//             each tile face, and the site codes.
//   k_pmerge_union / k_pmerge_resolve
//             the master's step 2: a union-find over the face nodes joined by
//             the bonds that leave a tile (the wrapping links included),
//             smaller key (cluster minimum) wins; then every representative
//             node gets its cluster's root and new state.
//   k_ppcc_cover
//             PCC (Sec. III): the extension rule per axis on the merged
//             clusters, and the feedback on the threshold.
//
// Conventions (both sides implement them; the CPU oracle is the reference):
//   - N = L^d sites, i = x + L*y (+ L*L*z); site i owns link dir = 0 (+x),
//     1 (+y), 2 (+z) with index l = d*i + dir; bond byte bit dir.  Under open
//     boundaries the + link of the last coordinate along an axis does not
//     exist.
//   - A link between equal states bonds iff word (l mod 4) of Philox(l/4, k,
//     BOND) < t, t = floor((1 - exp(-J/T)) 2^32).
//   - A cluster with root r (its minimum site) takes state floor(w q / 2^32),
//     w = word (r mod 4) of Philox(r/4, k, QSPIN); the hot start is the same
//     function of word (i mod 4) of Philox(i/4, 0, INIT).
//   - bond_sum = sum over links of (2 delta - 1), mag = sum over sites of
//     (q [s_i = 0] - 1).
#include "swgpu.h"
#include "sw_device.cuh"
#include "sw_internal.h"
#include "sw_launch.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <mutex>

using namespace swg;

namespace {

constexpr uint32_t STREAM_QSPIN = 3;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int PT = 256;   // threads of the per-site helper kernels

__device__ __forceinline__ uint8_t potts_state(uint32_t w, int q)
{
    return (uint8_t)(((uint64_t)w * (uint32_t)q) >> 32);
}

// New state of the cluster whose root is global site r in sweep k.
__device__ __forceinline__ uint8_t cluster_state(uint32_t r, uint32_t klo, uint32_t khi, uint32_t k0, uint32_t k1,
                                                 int q)
{
    const U4 u = philox4x32_10(r >> 2, klo, khi, STREAM_QSPIN, k0, k1);
    return potts_state(u4_word(u, (int)(r & 3u)), q);
}

// ------------------------------------------------------------ tile geometry
// A tile is TX x TY (x TZ) sites; its rows (y, z) are row index r = y + TY z,
// each of TWW 32-site words.  One thread per word: WT = 256 threads.  Where the grid
// leaves an SM with few warps a CTA has M = 2 or 4 times as many (launch_tile).
// Face nodes: for each axis a, a "-" face (local coordinate a = 0) and a "+"
// face (the tile's last valid coordinate along a), each of Fa slots indexed
// by the site's other coordinates (axis 0: y + TY z; axis 1: x + TX z; axis
// 2: x + TX y).  Slot layout: [x-, x+, y-, y+, z-, z+].
template <int DIM>
struct PG {
    static constexpr int TX = DIM == 2 ? 128 : 32;
    static constexpr int TY = DIM == 2 ? 64 : 16;
    static constexpr int TZ = DIM == 2 ? 1 : 16;
    static constexpr int TWW = TX / 32;
    static constexpr int NR = TY * TZ;          // rows
    static constexpr int WT = NR * TWW;         // threads that own a word (and threads of a tile CTA, M = 1)
    static constexpr int NS = TX * TY * TZ;     // sites
    static constexpr int PW = TX + 1;           // forest row pitch (rows on distinct banks)
    static constexpr int RS = TX + 4;           // state row pitch in bytes (the halo column, padded)
    static constexpr int HY = TY + 1, HZ = DIM == 2 ? 1 : TZ + 1;
    static constexpr int F0 = TY * TZ, F1 = TX * TZ, F2 = DIM == 3 ? TX * TY : 0;
    static constexpr int FT = F0 + F1 + F2;     // + face sites: crossing links, and halo sites
    static constexpr int S = 2 * FT;            // node slots
    static constexpr int CW = FT / 32;          // crossing-bit words
    static constexpr int PMW = DIM == 2 ? 6 : 2;   // PCC coverage words of a piece
    static_assert(WT == 256 && NS == 8 * 4 * WT, "tile launch shape");
    static_assert(F0 % 32 == 0 && F1 % 32 == 0 && F2 % 32 == 0, "faces of whole words");
    static_assert(S <= 0x7FFF, "slots fit the code");
};

template <int DIM>
__device__ __forceinline__ int face_off(int a, int side)
{
    using G = PG<DIM>;
    return (a == 0 ? 0 : a == 1 ? 2 * G::F0 : 2 * G::F0 + 2 * G::F1) +
           side * (a == 0 ? G::F0 : a == 1 ? G::F1 : G::F2);
}

// The local site of slot s (false past the tile's valid sites).
template <int DIM>
__device__ __forceinline__ bool slot_xyz(int s, const int (&e)[3], int &x, int &y, int &z)
{
    using G = PG<DIM>;
    if (s < 2 * G::F0) {
        const int side = s >= G::F0, f = s - side * G::F0;
        x = side ? e[0] - 1 : 0;
        y = f % G::TY;
        z = f / G::TY;
    } else if (s < 2 * G::F0 + 2 * G::F1) {
        const int s2 = s - 2 * G::F0, side = s2 >= G::F1, f = s2 - side * G::F1;
        y = side ? e[1] - 1 : 0;
        x = f % G::TX;
        z = f / G::TX;
    } else {
        const int s2 = s - 2 * G::F0 - 2 * G::F1, side = s2 >= G::F2, f = s2 - side * G::F2;
        z = side ? e[2] - 1 : 0;
        x = f % G::TX;
        y = f / G::TX;
    }
    return x < e[0] && y < e[1] && z < e[2];
}

// The same for slot tid + 256 M q, the q-th of a tile kernel's thread (q is known
// when the code is compiled, and with it the face but for M = 4).
template <int DIM, int M>
__device__ __forceinline__ bool slot_of(int q, int tid, const int (&e)[3], int &x, int &y, int &z)
{
    using G = PG<DIM>;
    if constexpr (M == 4) {
        return slot_xyz<DIM>(tid + 1024 * q, e, x, y, z);
    } else if constexpr (DIM == 2) {
        static_assert(DIM != 2 || (G::F0 == 64 && G::F1 == 128), "slots of a thread");
        const bool side = tid < 128;   // M = 1, q = 0: x-, x+, y-; q = 1: y+.  M = 2: all
        z = 0;
        x = q == 0 ? (side ? (tid < 64 ? 0 : e[0] - 1) : (tid - 128) & 127) : tid;
        y = q == 0 ? (side ? tid & 63 : tid < 256 ? 0 : e[1] - 1) : e[1] - 1;
    } else {
        static_assert(DIM != 3 || (G::F0 == 256 && G::F1 == 512 && G::F2 == 512), "slots of a thread");
        const int f0 = M == 1 ? q : tid >> 8;   // q < 2 / M: x-, x+
        if (q < 2 / M) {
            x = f0 ? e[0] - 1 : 0;
            y = tid & 15;
            z = (tid >> 4) & 15;
        } else {
            const int f = M == 1 ? tid + 256 * (q & 1) : tid, face = M == 1 ? q >> 1 : q;   // 1, 2: y-, y+; 3, 4: z-, z+
            x = f & 31;
            y = face == 1 ? 0 : face == 2 ? e[1] - 1 : f >> 5;
            z = face < 3 ? f >> 5 : face == 3 ? 0 : e[2] - 1;
        }
    }
    return x < e[0] && y < e[1] && z < e[2];
}

struct PTile {
    int c[3];      // tile coordinates
    int o[3];      // origin (sites)
    int e[3];      // extent (valid sites; 1 along z in 2D)
    int nb[3];     // tile index of the + neighbour along each axis (periodic)
    uint32_t gbase;   // global index of local site (0, 0, 0)
};

template <int DIM>
__device__ __forceinline__ PTile ptile_of(const PottsDev &p, int lt)
{
    using G = PG<DIM>;
    PTile t;
    const int n[3] = {p.ntx, p.nty, p.ntz};
    const int T[3] = {G::TX, G::TY, G::TZ};
    const int step[3] = {1, p.ntx, p.ntx * p.nty};
    const int r = (int)((uint32_t)lt / (uint32_t)p.ntx);
    t.c[2] = DIM == 3 ? (int)((uint32_t)r / (uint32_t)p.nty) : 0;
    t.c[1] = r - t.c[2] * p.nty;
    t.c[0] = lt - r * p.ntx;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t.o[a] = t.c[a] * T[a];
        t.e[a] = a < DIM ? min(T[a], p.L - t.o[a]) : 1;
        t.nb[a] = lt + (t.c[a] + 1 < n[a] ? step[a] : step[a] * (1 - n[a]));
    }
    const uint32_t uL = (uint32_t)p.L;
    t.gbase = (uint32_t)t.o[0] + uL * ((uint32_t)t.o[1] + uL * (uint32_t)t.o[2]);
    return t;
}

// A node's link under the topological rule (below): its parent and its
// displacement from it.
struct alignas(16) WLink {
    int32_t parent, dx, dy, dz;
};

// ------------------------------------------------- 3D tile union-find
// Connected components of the bonds inside a 32 x 16 x 16 tile, B[r] = {run heads
// by the +x bonds, +y, +z bonds} of row r = y + 16 z, all without the links that leave
// the tile.  Warp w holds the rows y = 4 (w mod 4) .. + 3, z = ZW (w / 4) .. + ZW - 1,
// ZW = 8 / M,
// lane = column, and goes through them with y innermost, the labels of the
// row before along y and of the four rows before along z in registers:
//   1. a run (maximal chain of x bonds in a row) takes the label of its last
//      contact along y, else along z, by shuffle, or starts a new label, its own
//      head; contacts with another label are kept as masks per column and united
//      afterwards (sw_device.cuh's tile_label_rows with a second direction: at
//      the 3D critical point 85% of the contacts inside a warp's rows need
//      no union);
//   2. the y and z bonds between the warps' row blocks, eight sites a thread.
// With the thread-per-word comparisons and the table codes below this took the
// tile kernel (bound by instruction issue) from 2.07 to 1.32 ms at L=512, q=2,
// T_c, and the 2D one from 0.62 to 0.38 ms at L=8192, q=3; run heads kept by the thread
// of the word, births by label and the tile's rows tested after the loop made a 3D
// sweep 3% faster (1715 -> 1660 us).
// Links hang the larger root under the smaller, so roots are piece minima in
// local row-major order, which is global order.  Returns, to lane x, the rows
// (bit 4 zz + yy) of the warp whose site x started a label.
template <int M>
__device__ __forceinline__ uint32_t tile_label3(volatile int *par, const uint32_t (*B)[3], int tw, int th, int td)
{
    using G = PG<3>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int ZW = 8 / M;
    const int yb = 4 * (warp & 3), zb = ZW * (warp >> 2);
    const uint32_t le = 0xFFFFFFFFu >> (31 - lane), gt = ~le;
    uint32_t born = 0u, cy = 0u, cz = 0u;
    {
        int labz[4] = {0, 0, 0, 0};
        uint32_t zw[4] = {0u, 0u, 0u, 0u};
        for (int zz = 0; zz < ZW && zb + zz < td; ++zz) {
            // first everything of the four rows that does not need the labels
            // (rows past the tile's have no bonds)
            int hd[4], py[4], pz[4];
            uint32_t yw[4], zo[4];
#pragma unroll
            for (int yy = 0; yy < 4; ++yy) {
                const int r = yb + yy + G::TY * (zb + zz);
                const uint32_t heads = B[r][0];
                const uint32_t n = heads & gt, m = (n - 1u) & ~n;   // m: up to the run's end
                hd[yy] = top_bit(heads & le);
                yw[yy] = yy > 0 ? B[r - 1][1] : 0u;
                zo[yy] = zw[yy];
                py[yy] = top_bit(yw[yy] & m);
                pz[yy] = top_bit(zo[yy] & m);
                zw[yy] = B[r][2];
            }
            int laby = 0;
#pragma unroll
            for (int yy = 0; yy < 4; ++yy) {
                const int row = (yb + yy + G::TY * (zb + zz)) * G::PW;
                const int ly = __shfl_sync(FULL, laby, py[yy]), lz = __shfl_sync(FULL, labz[yy], pz[yy]);
                const bool hy = py[yy] >= hd[yy], hz = pz[yy] >= hd[yy];
                const int lab = hy ? ly : hz ? lz : row + hd[yy];
                const uint32_t bit = 1u << (4 * zz + yy);
                if (((yw[yy] >> lane) & 1u) && laby != lab) cy |= bit;
                if (((zo[yy] >> lane) & 1u) && labz[yy] != lab) cz |= bit;
                if (lab == row + lane) born |= bit;   // (a label is its first site's node)
                par[row + lane] = lab;
                laby = labz[yy] = lab;
            }
        }
    }
    __syncwarp();
    const int col = (yb + G::TY * zb) * G::PW + lane;
    auto node = [&](int i) { return col + ((i & 3) + G::TY * (i >> 2)) * G::PW; };
    for (; cy; cy &= cy - 1) {
        const int i = node(__ffs(cy) - 1);
        shook<4>(par, par[i - G::PW], par[i]);
    }
    for (; cz; cz &= cz - 1) {
        const int i = node(__ffs(cz) - 1);
        shook<4>(par, par[i - G::TY * G::PW], par[i]);
    }
    __syncthreads();
    // y bonds from rows y = 3, 7, 11 (every z), z bonds from the last layer of every
    // warp but the top ones (every y): 64, 96 or 160 rows, a quarter of a row's word a
    // thread
    {
        const int w = threadIdx.x >> 2, x0 = 8 * (threadIdx.x & 3);
        const bool yd = w < 48;
        const int y = yd ? 4 * (w % 3) + 3 : w & 15, z = yd ? w / 3 : ZW * ((w >> 4) - 2) - 1;
        const int A = y + G::TY * z, step = (yd ? 1 : G::TY) * G::PW;
        uint32_t bits = w < 48 + 16 * (16 / ZW - 1) && y < th && z < td ? (B[A][yd ? 1 : 2] >> x0) & 0xFFu : 0u;
        int pa = -1, pb = -1;
        for (; bits; bits &= bits - 1) {
            const int i = A * G::PW + x0 + __ffs(bits) - 1;
            const int a = par[i], b = par[i + step];
            if (a != pa || b != pb) shook<2>(par, a, b);
            pa = a;
            pb = b;
        }
    }
    __syncthreads();
    if (yb + 4 > th) born &= 0x11111111u * ((1u << max(th - yb, 0)) - 1u);   // rows of the tile
    return tw > lane ? born : 0u;
}

// ------------------------------------------------------------ shared layout
// The states are dead once the bonds are drawn and the forest is not written
// before the labelling, so the two share memory: five CTAs fit an SM (48
// registers a thread), which runs the kernel 5% faster than four.
template <int DIM>
struct PSmem {
    using G = PG<DIM>;
    static constexpr int BW = DIM == 2 ? 2 * G::TWW : 3;   // bond words of a row
    union {
        int par[G::NR * G::PW];             // from the labelling on: union-find forest over the sites
        struct {
            alignas(16) uint16_t code[G::NS];  // finish half: the tile's site codes
            alignas(16) uint32_t raw[G::NR][DIM == 2 ? 2 * G::TWW : 4];   // a row's random bond bits
            // finish half: the table the codes index, the new states of the
            // tile's pieces by slot, then every state itself
            uint8_t fst[G::S + 256];
            uint8_t st[G::HZ][G::HY][G::RS];   // states; row TY, layer TZ and column tw: + halo
        } s;
    } f;
    uint8_t qs[G::NR][G::TX];               // each site's state drawn from the QSPIN stream
    // a row's bonds inside the tile: in 2D [2c] the +x (heads_word) and [2c + 1] the
    // +y bonds of word c, in 3D the run heads by the +x bonds, the +y and the +z bonds
    alignas(16) uint32_t b[G::NR][BW];
    int acc[4];                             // sums of the tile: bond_sum, mag (sweep j-1), nbonds, nclusters (sweep j)
    unsigned long long acc_c2[2];           // RF_CSIZE: sum |C|^2 of sweep j-1 and of sweep j
    uint32_t pm[G::S][G::PMW];              // PCC: coordinates each border piece occupies
};

static_assert(sizeof(PSmem<2>::f) == sizeof(int) * PG<2>::NR * PG<2>::PW, "the finish half fits the forest's space");
static_assert(sizeof(PSmem<3>::f) == sizeof(int) * PG<3>::NR * PG<3>::PW, "the finish half fits the forest's space");

template <int DIM>
constexpr size_t ptile_smem(bool pcc)
{
    return pcc ? sizeof(PSmem<DIM>) : offsetof(PSmem<DIM>, pm);
}

// Top bit of every byte of t that is zero (t = a ^ b: the bytes where a and b agree).
__device__ __forceinline__ uint32_t zero_bytes(uint32_t t)
{
    return ~(((t & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | t) & 0x80808080u;
}

// The four flags of zero_bytes in bits 28-31.
__device__ __forceinline__ uint32_t byte_flags(uint32_t z)
{
    return z * 0x00204081u;
}

// Bit m of byte q of v (q < 4, m < 8) to bit 4 m + q.
__device__ __forceinline__ uint32_t interleave4x8(uint32_t v)
{
    auto spread = [](uint32_t x) {   // bit m to bit 4 m
        x = (x | (x << 12)) & 0x000F000Fu;
        x = (x | (x << 6)) & 0x03030303u;
        return (x | (x << 3)) & 0x11111111u;
    };
    return spread(v & 0xFFu) | (spread((v >> 8) & 0xFFu) << 1) | (spread((v >> 16) & 0xFFu) << 2) |
           (spread(v >> 24) << 3);
}

// ----------------------------------------------------------------- k_ptile
// Launch j finishes sweep j-1 (j >= 1) and starts sweep j (j < nsweeps).
// F: FEAT_* bits compiled in (0: periodic plain lattices only).
template <int DIM, int F, int M>
__global__ void __launch_bounds__(M * PG<DIM>::WT, M == 1 ? 5 : M == 2 ? 2 : 1)
    k_ptile(const PottsDev p, int j, int nsweeps, uint64_t sweep0, DevObs *obs)
{
    using G = PG<DIM>;
    constexpr int WT = G::WT, NT = M * WT, NW = NT / 32, S = G::S, TWW = G::TWW;
    constexpr int NQ = G::NS / 8 / NT;          // 8-site groups per thread
    constexpr int SPT = (S + NT - 1) / NT;      // node slots per thread
    constexpr int LR = 32 / M;                  // rows of a warp in the labelling
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PSmem<DIM> &sm = *reinterpret_cast<PSmem<DIM> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool wind = (F & FEAT_WIND) && (p.flags & RF_WIND);
    if (!wind) chain_next();   // (topological rule: below)
    const int lt = blockIdx.x;   // the grid is the lattice's tiles
    const bool fin = j >= 1, start = j < nsweeps;
    const PTile t = ptile_of<DIM>(p, lt);
    const int tw = t.e[0], th = t.e[1], td = t.e[2];
    const uint32_t uL = (uint32_t)p.L;
    const int q = p.q;
    const bool open = (F & FEAT_OPEN) && (p.flags & RF_OPEN);
    const bool open_x = open && t.c[0] == p.ntx - 1;
    const bool open_y = open && t.c[1] == p.nty - 1;
    const bool open_z = DIM == 3 && open && t.c[2] == p.ntz - 1;
    const bool csz = (F & FEAT_CSIZE) && (p.flags & RF_CSIZE);
    const bool ext = (F & FEAT_PCC) && (p.flags & RF_PCC) && !(p.flags & RF_WIND);   // PCC by the extension rule
    uint16_t *code = p.code + (size_t)lt * G::NS;
    const size_t nbase = (size_t)lt * S;
    const uint32_t k0 = (uint32_t)p.seed, k1 = (uint32_t)(p.seed >> 32);
    // global index of a local site, and of a forest index
    auto gidx = [&](int x, int y, int z) { return t.gbase + (uint32_t)x + uL * ((uint32_t)y + uL * (uint32_t)z); };
    auto gfor = [&](int fi) {
        const int r = fi / G::PW;
        return gidx(fi - r * G::PW, r % G::TY, r / G::TY);
    };
    // local site of 8-site group idx (row-major order), false past the valid rows
    auto group = [&](int idx, int &x, int &y, int &z) {
        const int li = 8 * idx, r = li / G::TX;
        x = li - r * G::TX;
        y = r % G::TY;
        z = r / G::TY;
        return y < th && z < td;
    };
    // the word of a thread of the first WT: row wr = (wy, wz), sites 32 wc .. 32 wc
    // + 31; of their warps, w holds rows WROWS w .. WROWS (w + 1) - 1.  In 3D all warps
    // draw, DROWS rows each
    constexpr int WROWS = G::NR / (WT / 32), DROWS = DIM == 2 ? WROWS : G::NR / NW;
    const int wr = tid / TWW, wc = tid % TWW, wy = wr % G::TY, wz = wr / G::TY;
    const bool row_ok = wy < th && wz < td;

    // ---- loads of the finish half, in flight during the draws
    auto finish_loads = [&]() {
        chain_wait();
        if (!fin) return;
        // the tile's codes, 8 sites per 16-byte asynchronous copy straight
        // into shared memory (the forest's space, free until the labelling),
        // and the states of its own pieces
        const uint4 *code4 = reinterpret_cast<const uint4 *>(code);
        uint4 *scode4 = reinterpret_cast<uint4 *>(sm.f.s.code);
#pragma unroll
        for (int qq = 0; qq < NQ; ++qq) {
            int x, y, z;
            const int idx = tid + qq * NT;
            if (group(idx, x, y, z)) cp_async16(scode4 + idx, code4 + idx);
        }
        for (int w = tid; w < S / 16; w += NT) cp_async16(sm.f.s.fst + 16 * w, p.nstate + nbase + 16 * w);
        if (M == 1 || tid < 256) sm.f.s.fst[S + tid] = (uint8_t)tid;
    };
    // a block of the first wave draws first (sw_device.cuh's k_tile)
    const bool early = lt < FIRST_WAVE_SMS * 5 && !p.thr_dev;
    if (!early) finish_loads();
    if (tid < 4) sm.acc[tid] = 0;
    if ((F & FEAT_CSIZE) && tid < 2) sm.acc_c2[tid] = 0ull;

    // ---- Step 1 (Sec. I) of sweep j, its random part: which links' Philox
    // words are below the threshold, and every site's QSPIN state (the draws
    // need no state, so they run while the loads above are in flight).  Each
    // warp draws its own rows; ballots leave them in shared memory for the
    // thread that owns the word.
    const uint64_t k = sweep0 + (uint64_t)j;
    const uint64_t thr = p.thr_dev ? *p.thr_dev : p.thr;
    const uint32_t klo = (uint32_t)k, khi = (uint32_t)(k >> 32);
    const bool any_bond = start && thr != 0;
    const uint32_t tm1 = (uint32_t)(thr - 1);
    // every row starts a QSPIN block (4 divides L): the bond draws also fill qs.
    // Otherwise qs is drawn apart, or every interior root and representative
    // draws its own: in 3D, where they are many (L=255, q=3, T_c: 279 us a sweep
    // against 298; q=2, T=2.0 the same), and in 2D grids of one wave, where the
    // roots' draws are a chain (L=1001: 35.5 us against 38.2; L=8190: 492 against 485)
    const bool aligned = (uL & 3u) == 0;
    const bool qsm = any_bond && (aligned || DIM == 3 || p.ntiles <= FIRST_WAVE_SMS * 5);
    auto ballots = [&](const U4 &u, bool act) {
        return make_uint4(__ballot_sync(FULL, act && below(u.x, tm1)), __ballot_sync(FULL, act && below(u.y, tm1)),
                          __ballot_sync(FULL, act && below(u.z, tm1)), __ballot_sync(FULL, act && below(u.w, tm1)));
    };
    auto states4 = [&](const U4 &u) {
        return (uint32_t)potts_state(u.x, q) | ((uint32_t)potts_state(u.y, q) << 8) |
               ((uint32_t)potts_state(u.z, q) << 16) | ((uint32_t)potts_state(u.w, q) << 24);
    };
    uint32_t extra = 0u;   // 2D, rows from an odd site: lane r's first two words of its row's 65th block
    if (any_bond) {
        if constexpr (DIM == 2) {
            // link l = 2i + d: sites 2m and 2m + 1 share Philox block m (the
            // Ising path's draws, sw_device.cuh)
            const bool wide = tw > 64;
            for (int i = 0; i < WROWS; i += 2) {
                const int y = WROWS * warp + i;
                if (y >= th) break;
                const uint32_t g0 = t.gbase + (uint32_t)y * uL, g2 = g0 + uL;
                const uint32_t b0 = (g0 >> 1) + lane, b2 = (g2 >> 1) + lane;
                const U4 r0 = philox4x32_10(b0, klo, khi, STREAM_BOND, k0, k1);
                const U4 r2 = philox4x32_10(b2, klo, khi, STREAM_BOND, k0, k1);
                U4 r1{}, r3{};
                if (wide) {
                    r1 = philox4x32_10(b0 + 32, klo, khi, STREAM_BOND, k0, k1);
                    r3 = philox4x32_10(b2 + 32, klo, khi, STREAM_BOND, k0, k1);
                }
                const uint4 q0 = ballots(r0, true), q1 = ballots(r1, true), q2 = ballots(r2, true), q3 = ballots(r3, true);
                if (lane == 0) {
                    uint4 *raw = reinterpret_cast<uint4 *>(&sm.f.s.raw[y][0]);
                    raw[0] = q0;
                    raw[1] = q1;
                    raw[2] = q2;
                    raw[3] = q3;
                }
                if (aligned) {
                    // lane l: the QSPIN block of sites 4l .. 4l + 3 of each row
                    const U4 s0 = philox4x32_10((g0 >> 2) + lane, klo, khi, STREAM_QSPIN, k0, k1);
                    const U4 s2 = philox4x32_10((g2 >> 2) + lane, klo, khi, STREAM_QSPIN, k0, k1);
                    *reinterpret_cast<uint32_t *>(&sm.qs[y][4 * lane]) = states4(s0);
                    *reinterpret_cast<uint32_t *>(&sm.qs[y + 1][4 * lane]) = states4(s2);
                }
            }
            if ((uL | t.gbase) & 1u) {
                const uint32_t g0 = t.gbase + (uint32_t)(WROWS * warp + (lane & (WROWS - 1))) * uL;
                const U4 r = philox4x32_10((g0 >> 1) + 64u, klo, khi, STREAM_BOND, k0, k1);
                extra = (below(r.x, tm1) ? 1u : 0u) | (below(r.y, tm1) ? 2u : 0u);
            }
        } else if (aligned) {
            // link l = 3i + d.  Every row starts on a multiple of 4, so its 96
            // links are exactly the 24 Philox blocks from 3 i0 / 4: three blocks
            // for four sites.  Lane 8 c + m draws block 3 m + c (c < 3), so that
            // byte c of the ballot of word w holds link 4 c + w of the m-th four
            // sites at bit m; lanes 24-31 draw the row's eight QSPIN blocks.
            const bool bl = lane < 24;
            const uint32_t st_ = bl ? STREAM_BOND : STREAM_QSPIN;
            const uint32_t off = bl ? 3u * (lane & 7) + (lane >> 3) : (uint32_t)(lane - 24);
            for (int i = 0; i < DROWS; i += 2) {
                // two rows y, y + 1 of a layer (DROWS and TY are even)
                const int r = DROWS * warp + i, y = r % G::TY, z = r / G::TY;
                if (y >= th || z >= td) continue;
                const uint32_t i0 = gidx(0, y, z) >> 2, i2 = i0 + (uL >> 2);
                const U4 u0 = philox4x32_10((bl ? 3u * i0 : i0) + off, klo, khi, st_, k0, k1);
                const U4 u2 = philox4x32_10((bl ? 3u * i2 : i2) + off, klo, khi, st_, k0, k1);
                const uint4 q0 = ballots(u0, true), q2 = ballots(u2, true);
                if (lane == 0) {
                    *reinterpret_cast<uint4 *>(&sm.f.s.raw[r][0]) = q0;
                    *reinterpret_cast<uint4 *>(&sm.f.s.raw[r + 1][0]) = q2;
                }
                if (!bl) {
                    *reinterpret_cast<uint32_t *>(&sm.qs[r][4 * (lane - 24)]) = states4(u0);
                    *reinterpret_cast<uint32_t *>(&sm.qs[r + 1][4 * (lane - 24)]) = states4(u2);
                }
            }
        } else {
            // a row starts anywhere in a block: its 96 links lie in the 25 blocks
            // from the one that holds its first; lane x takes its three bits
            // from the ballots
            for (int i = 0; i < DROWS; ++i) {
                const int r = DROWS * warp + i, y = r % G::TY, z = r / G::TY;
                if (y >= th || z >= td) continue;
                const uint32_t l0 = 3u * gidx(0, y, z);
                const U4 u = philox4x32_10((l0 >> 2) + lane, klo, khi, STREAM_BOND, k0, k1);
                const uint4 B = ballots(u, true);
                const int l = (int)(l0 & 3u) + 3 * lane;
                auto bit_of = [&](int e) {
                    const uint32_t w = e & 2 ? (e & 1 ? B.w : B.z) : (e & 1 ? B.y : B.x);
                    return (w >> (e >> 2)) & 1u;
                };
                const uint32_t rx = __ballot_sync(FULL, bit_of(l)), ry = __ballot_sync(FULL, bit_of(l + 1)),
                               rz = __ballot_sync(FULL, bit_of(l + 2));
                if (lane == 0) *reinterpret_cast<uint4 *>(&sm.f.s.raw[r][0]) = make_uint4(rx, ry, rz, 0u);
            }
        }
        if (qsm && !aligned) {
            // rows that start inside a QSPIN block: the blocks of all the warp's rows
            // dealt to its lanes
            const int nb = (tw + 3) / 4 + 1;   // blocks of a row
            constexpr int QROWS = G::NR / NW;
            for (int i = lane; i < QROWS * nb; i += 32) {
                const int r = QROWS * warp + i / nb, b = i % nb, y = r % G::TY, z = r / G::TY;
                if (y >= th || z >= td) continue;
                const uint32_t i0 = gidx(0, y, z);
                const uint32_t v = states4(philox4x32_10((i0 >> 2) + (uint32_t)b, klo, khi, STREAM_QSPIN, k0, k1));
                const int x = 4 * b - (int)(i0 & 3u);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((uint32_t)(x + e) < (uint32_t)G::TX) sm.qs[r][x + e] = (uint8_t)(v >> (8 * e));
            }
        }
    }

    uint8_t *st = &sm.f.s.st[0][0][0];
    if (early) finish_loads();
    if (fin) {
        // ---- finish sweep j-1: every site's new state
        const bool last = j == nsweeps;
        // the + halo: new states of the neighbours' "-" face sites (the merge
        // gives every "-" face slot its cluster's state)
        constexpr int HPT = (G::FT + NT - 1) / NT;
#pragma unroll
        for (int qq = 0; qq < HPT; ++qq) {
            const int h = tid + qq * NT;
            int hnode = -1, hpos = 0;
            if (h < G::F0) {
                const int y = h % G::TY, z = h / G::TY;
                if (y < th && z < td) {
                    hnode = t.nb[0] * S + face_off<DIM>(0, 0) + h;
                    hpos = (z * G::HY + y) * G::RS + tw;
                }
            } else if (h < G::F0 + G::F1) {
                const int f = h - G::F0, x = f % G::TX, z = f / G::TX;
                if (x < tw && z < td) {
                    hnode = t.nb[1] * S + face_off<DIM>(1, 0) + f;
                    hpos = (z * G::HY + th) * G::RS + x;
                }
            } else if (h < G::FT) {
                const int f = h - G::F0 - G::F1, x = f % G::TX, y = f / G::TX;
                if (x < tw && y < th) {
                    hnode = t.nb[2] * S + face_off<DIM>(2, 0) + f;
                    hpos = (td * G::HY + y) * G::RS + x;
                }
            }
            if (hnode >= 0) st[hpos] = p.nstate[hnode];
        }
        cp_async_wait_all();
        __syncthreads();
        const uint4 *scode4 = reinterpret_cast<const uint4 *>(sm.f.s.code);
#pragma unroll
        for (int qq = 0; qq < NQ; ++qq) {
            int x, y, z;
            const int idx = tid + qq * NT;
            if (!group(idx, x, y, z)) continue;
            const uint4 cq = scode4[idx];
            const uint32_t wv[4] = {cq.x, cq.y, cq.z, cq.w};
            uint32_t lo = 0u, hi = 0u;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t s = sm.f.s.fst[e & 1 ? wv[e >> 1] >> 16 : wv[e >> 1] & 0xFFFFu];
                if (e < 4) lo |= s << (8 * e);
                else hi |= s << (8 * (e - 4));
            }
            const int nval = min(8, tw - x);
            uint8_t *row = st + (z * G::HY + y) * G::RS + x;
            if (nval == 8) {
                reinterpret_cast<uint32_t *>(row)[0] = lo;
                reinterpret_cast<uint32_t *>(row)[1] = hi;
            } else {
                for (int e = 0; e < nval; ++e) row[e] = (uint8_t)((e < 4 ? lo >> (8 * e) : hi >> (8 * (e - 4))) & 0xFFu);
            }
            if (last) {
                const uint32_t gi0 = gidx(x, y, z);
                if (nval == 8 && (gi0 & 7u) == 0) {
                    *reinterpret_cast<uint2 *>(p.spin + gi0) = make_uint2(lo, hi);
                } else {
                    for (int e = 0; e < nval; ++e)
                        p.spin[gi0 + e] = (uint8_t)((e < 4 ? lo >> (8 * e) : hi >> (8 * (e - 4))) & 0xFFu);
                }
                // border sites' labels: their cluster's root (the interior
                // clusters' were written when the sweep started)
                for (int e = 0; e < nval; ++e) {
                    const uint32_t u = (wv[e >> 1] >> (16 * (e & 1))) & 0xFFFFu;
                    if (u < (uint32_t)S) p.label[gi0 + e] = (int32_t)(p.nfinal[nbase + u] & ROOT_MASK);
                }
            }
        }
    } else {
        // first sweep of the call: states and + halos from global memory
        const int hrows = (th + 1) * (DIM == 3 ? td + 1 : 1);
        for (int rw = warp; rw < hrows; rw += NW) {
            const int hy = rw % (th + 1), hz = rw / (th + 1);
            const uint32_t gy = (uint32_t)((t.o[1] + hy) % p.L), gz = DIM == 3 ? (uint32_t)((t.o[2] + hz) % p.L) : 0u;
            const uint8_t *grow = p.spin + (size_t)uL * (gy + (size_t)uL * gz);
            for (int x = lane; x <= tw; x += 32) {
                int gx = t.o[0] + x;
                if (gx >= p.L) gx -= p.L;
                sm.f.s.st[hz][hy][x] = grow[gx];
            }
        }
    }
    __syncthreads();

    // ---- the thread's word: state agreement along its links (four sites a
    //      comparison), the sums of sweep j-1 and the bonds of sweep j
    const bool last_start = j == nsweeps - 1;
    if (M == 1 || tid < WT) {
        const uint32_t vm = row_ok ? valid_mask(wc, tw) : 0u;
        const uint32_t vx = open_x && row_ok ? valid_mask(wc, tw - 1) : vm;
        const uint32_t vy = open_y && wy == th - 1 ? 0u : vm;
        const uint32_t vz = DIM == 2 || (open_z && wz == td - 1) ? 0u : vm;
        uint32_t ex = 0u, ey = 0u, ez = 0u, zero = 0u;
        if (row_ok) {
            const uint32_t *row = reinterpret_cast<const uint32_t *>(st + (wz * G::HY + wy) * G::RS + 32 * wc);
            const uint32_t *rowy = row + G::RS / 4;
            const uint32_t *rowz = row + G::HY * (G::RS / 4);
            uint32_t nxt = row[8];
#pragma unroll
            for (int m = 7; m >= 0; --m) {
                const uint32_t cur = row[m];
                ex = __funnelshift_l(byte_flags(zero_bytes(cur ^ __funnelshift_r(cur, nxt, 8))), ex, 4);
                ey = __funnelshift_l(byte_flags(zero_bytes(cur ^ rowy[m])), ey, 4);
                if (DIM == 3) ez = __funnelshift_l(byte_flags(zero_bytes(cur ^ rowz[m])), ez, 4);
                if (fin) zero = __funnelshift_l(byte_flags(zero_bytes(cur)), zero, 4);
                nxt = cur;
            }
            ex &= vx;
            ey &= vy;
            ez &= vz;
        }
        if (fin) {
            // bond_sum: +1 a link between equal states, -1 otherwise
            const int bs = 2 * (__popc(ex) + __popc(ey) + __popc(ez)) - __popc(vx) - __popc(vy) - __popc(vz);
            const int mag = q * __popc(zero & vm) - __popc(vm);
            const int ws = __reduce_add_sync(FULL, bs), wm = __reduce_add_sync(FULL, mag);
            if (lane == 0) {
                atomicAdd(&sm.acc[0], ws);
                atomicAdd(&sm.acc[1], wm);
            }
        }
        if (start) {
            uint32_t rx = 0u, ry = 0u, rz = 0u;
            if (any_bond) {
                const uint4 raw = *reinterpret_cast<const uint4 *>(&sm.f.s.raw[wr][DIM == 2 ? 4 * (wc >> 1) : 0]);
                if (DIM == 2) {
                    rx = interleave16(raw.x, raw.z, wc & 1);
                    ry = interleave16(raw.y, raw.w, wc & 1);
                    if ((uL | t.gbase) & 1u) {
                        // rows that start on an odd site are one site ahead of their blocks
                        const uint32_t e = __shfl_sync(FULL, extra, lane / TWW);
                        uint32_t nx = __shfl_down_sync(FULL, rx, 1), ny = __shfl_down_sync(FULL, ry, 1);
                        if (wc == TWW - 1) {
                            nx = e;
                            ny = e >> 1;
                        }
                        if ((t.gbase + (uint32_t)wy * uL) & 1u) {
                            rx = __funnelshift_r(rx, nx, 1);
                            ry = __funnelshift_r(ry, ny, 1);
                        }
                    }
                } else if (aligned) {
                    // byte c of word w: link 4 c + w of the twelve links of four
                    // sites; direction d of site i is link 3 i + d
                    rx = interleave4x8(__byte_perm(__byte_perm(raw.x, raw.w, 0x0040), __byte_perm(raw.z, raw.y, 0x0061), 0x5410));
                    ry = interleave4x8(__byte_perm(__byte_perm(raw.y, raw.x, 0x0050), __byte_perm(raw.w, raw.z, 0x0061), 0x5410));
                    rz = interleave4x8(__byte_perm(__byte_perm(raw.z, raw.y, 0x0050), __byte_perm(raw.x, raw.w, 0x0062), 0x5410));
                } else {
                    rx = raw.x;
                    ry = raw.y;
                    rz = raw.z;
                }
            }
            const uint32_t bx = rx & ex, by = ry & ey, bz = rz & ez;
            const int nb = __reduce_add_sync(FULL, __popc(bx) + __popc(by) + __popc(bz));
            if (lane == 0) atomicAdd(&sm.acc[2], nb);
            // crossing bonds, bit f of face a at word (f / 32) of that face's block:
            // x face f = r (the row), y face f = x + TX z, z face f = x + TX y
            {
                uint32_t *cross = p.cross + (size_t)lt * G::CW;
                const int last_c = (tw - 1) >> 5, last_b = (tw - 1) & 31;
                const uint32_t e = __ballot_sync(FULL, wc == last_c && ((bx >> last_b) & 1u)) >> last_c;
                if (DIM == 2) {
                    // a warp's eight rows a byte: bit 4 r of e is row r
                    uint32_t v = e & 0x11111111u;
                    v = (v | (v >> 3)) & 0x03030303u;
                    v = (v | (v >> 6)) & 0x000F000Fu;
                    v = (v | (v >> 12)) & 0xFFu;
                    if (lane == 0) reinterpret_cast<uint8_t *>(cross)[warp] = (uint8_t)v;
                } else if (lane == 0) {
                    cross[warp] = e;
                }
                // (layers past the tile: no bonds, by = bz = 0)
                if (wy == th - 1) cross[G::F0 / 32 + wc + TWW * wz] = by;
                if (DIM == 3 && wz == td - 1) cross[(G::F0 + G::F1) / 32 + wy] = bz;
            }
            auto put = [&](uint32_t x, uint32_t y, uint32_t z) {
                if constexpr (DIM == 2) {
                    *reinterpret_cast<uint2 *>(&sm.b[wr][2 * wc]) = make_uint2(x, y);
                } else {
                    sm.b[wr][0] = x;
                    sm.b[wr][1] = y;
                    sm.b[wr][2] = z;
                }
            };
            if (last_start) {
                // the last sweep of the call keeps its bond bytes (the warp's own rows)
                put(bx, by, bz);
                __syncwarp();
                for (int i = 0; i < WROWS; ++i) {
                    const int r = WROWS * warp + i, y = r % G::TY, z = r / G::TY;
                    if (y >= th || z >= td) continue;
                    const uint32_t g0 = gidx(0, y, z);
#pragma unroll
                    for (int c = 0; c < TWW; ++c) {
                        const int x = 32 * c + lane;
                        if (x >= tw) break;
                        uint32_t b = ((sm.b[r][DIM == 2 ? 2 * c : 0] >> lane) & 1u) |
                                     (((sm.b[r][DIM == 2 ? 2 * c + 1 : 1] >> lane) & 1u) << 1);
                        if (DIM == 3) b |= ((sm.b[r][2] >> lane) & 1u) << 2;
                        p.bond[g0 + (uint32_t)x] = (uint8_t)b;
                    }
                }
                __syncwarp();
            }
            const uint32_t in_x = bx & valid_mask(wc, tw - 1);
            put(DIM == 2 ? heads_word(in_x) : run_heads(in_x), wy < th - 1 ? by : 0u, wz < td - 1 ? bz : 0u);
        }
    }
    // clusters that touch a tile face: their sizes were summed at their root nodes
    // by the merge; each root node is in exactly one tile
    if (csz && fin) {
        unsigned long long c2 = 0ull;
#pragma unroll
        for (int qq = 0; qq < SPT; ++qq) {
            const long long c = tid + qq * NT < S ? p.csize[nbase + tid + qq * NT] : 0;
            c2 += (unsigned long long)(c * c);
        }
        warp_add64(&sm.acc_c2[0], c2);
    }
    if (start && ext) {
        for (int w = tid; w < S * G::PMW; w += NT) (&sm.pm[0][0])[w] = 0u;
        // the tiles together clear what the last sweep's candidates left (the union
        // kernel then resets their counts)
        const int64_t W = (p.L + 31) / 32, FS = DIM == 2 ? (int64_t)p.L : (int64_t)p.L * p.L;
        const int64_t i0 = (int64_t)lt * NT + tid, di = (int64_t)p.ntiles * NT;
        for (int a = 0; a < DIM; ++a) {
            const int64_t nc = p.ncand[a];
            for (int64_t i = i0; i < nc * W; i += di) p.cov[a * FS * W + i] = 0u;
            for (int64_t i = i0; i < nc; i += di) p.ccount[a * FS + i] = 0;
        }
    }
    if (start && lt == 0 && tid == 0) {
        obs[j].threshold = thr;
        obs[j].spans_x = 0;
        obs[j].spans_y = 0;
    }
    __syncthreads();

    if (start) {
        // Step 2 inside the tile
        uint32_t born;
        if constexpr (DIM == 2)
            born = tile_label_rows<64, LR>(sm.f.par, sm.b, th, tw);
        else
            born = tile_label3<M>(sm.f.par, sm.b, tw, th, td);
        // the warp's rows of the labelling: bit i of its masks is row lrow(i) and
        // its lanes are the sites lx
        const int lx = DIM == 2 ? 32 * (warp % TWW) + lane : lane;
        auto lrow = [&](int i) {
            return DIM == 2 ? LR * (warp / TWW) + i : 4 * (warp & 3) + (i & 3) + G::TY * (LR / 4 * (warp >> 2) + (i >> 2));
        };

        // The labels' nodes that are no roots point at theirs, so that a site's
        // root is two loads away below (a walk a slot took a quarter of the 3D
        // kernel: 10 slots a thread).
        uint32_t linked = 0u;
        for (uint32_t bits = born; bits; bits &= bits - 1) {
            const int x = lrow(__ffs(bits) - 1) * G::PW + lx;
            int v = sm.f.par[x];
            if (v == x) continue;
            linked |= bits & -bits;
            int w = sm.f.par[v];
            if (w == v) continue;
            while (w != v) {
                v = w;
                w = sm.f.par[v];
            }
            sm.f.par[x] = v;
        }
        const uint32_t roots = born & ~linked;
        __syncthreads();

        // One node per face site: key = global index of the piece's local root,
        // parent = the piece's first face slot (the representative).
        // (A slot whose left neighbour has the same root leaves the mark to it: at
        // T_c a few big pieces hold most slots, and 32 lanes at one address wait
        // for each other.)
        int rs[SPT];
#pragma unroll
        for (int qq = 0; qq < SPT; ++qq) {
            const int s = tid + qq * NT;
            int x, y, z;
            rs[qq] = -1;
            if (s < S && slot_of<DIM, M>(qq, tid, t.e, x, y, z))
                rs[qq] = sroot_marked(sm.f.par, (y + G::TY * z) * G::PW + x);
            const int left = __shfl_up_sync(FULL, rs[qq], 1);
            if (rs[qq] >= 0 && (lane == 0 || left != rs[qq])) {
                const int mark = (int)(INFO_BORDER | (uint32_t)s);
                if (*(volatile int *)&sm.f.par[rs[qq]] > mark) atomicMin(&sm.f.par[rs[qq]], mark);
            }
        }
        __syncthreads();
        // Every interior root gets its record, its cluster's new state (Sec. I
        // step 3), and is counted; the other labels' nodes take a copy of their
        // root's record where it is there already (cluster sizes are added at
        // the roots and labels are root indices: they keep the root's index).
        {
            int ncl = 0;
            for (uint32_t bits = roots; bits; bits &= bits - 1) {
                const int r = lrow(__ffs(bits) - 1), x = r * G::PW + lx;
                const int v = sm.f.par[x];
                if (v == x) {
                    const uint32_t s = qsm ? sm.qs[r][lx] : cluster_state(gidx(lx, r % G::TY, r / G::TY), klo, khi, k0, k1, q);
                    sm.f.par[x] = (int)(INFO_INTERIOR | (S + s));
                    ++ncl;
                }
            }
            ncl = __reduce_add_sync(FULL, ncl);
            if (lane == 0 && ncl) atomicAdd(&sm.acc[3], ncl);
            if (!csz && !last_start)
                for (; linked; linked &= linked - 1) {
                    const int x = lrow(__ffs(linked) - 1) * G::PW + lx;
                    sm.f.par[x] = sm.f.par[sm.f.par[x]];   // (a root that has no record yet is its own entry)
                }
        }
#pragma unroll
        for (int qq = 0; qq < SPT; ++qq) {
            const int s = tid + qq * NT;
            if (s >= S) break;
            const size_t node = nbase + s;
            if (rs[qq] >= 0) {
                const int rep = sm.f.par[rs[qq]] & 0xFFFF;
                const uint32_t key = gfor(rs[qq]);
                p.node[node] = make_int2((int)(nbase + rep), (int)(key | (rep == s ? KEY_REP : 0u)));
                // a representative's new state if its piece's minimum is its
                // cluster's
                if (rep == s) {
                    const int r = rs[qq] / G::PW;
                    p.kstate[node] = qsm ? sm.qs[r][rs[qq] - r * G::PW] : cluster_state(key, klo, khi, k0, k1, q);
                }
            } else {
                p.node[node] = make_int2(NODE_NONE, 0);
            }
            if (csz) p.csize[node] = 0;   // the merge adds piece sizes at root nodes
            if (ext)
                for (int a = 0; a < DIM; ++a) p.cid[node * DIM + a] = 0;
            if (wind) {
                // topological rule: the node's link before the unions -- its
                // representative and its displacement from it, both in this tile
                WLink w{(int)node, 0, 0, 0};
                int x, y, z, xr, yr, zr;
                if (rs[qq] >= 0) {
                    const int rep = sm.f.par[rs[qq]] & 0xFFFF;
                    if (slot_xyz<DIM>(s, t.e, x, y, z) && slot_xyz<DIM>(rep, t.e, xr, yr, zr))
                        w = WLink{(int)(nbase + rep), x - xr, y - yr, z - zr};
                }
                reinterpret_cast<WLink *>(p.wlink)[node] = w;
            }
        }
        __syncthreads();
        if (wind) chain_next();
        // Every site's 2-byte code (the low half of its root's record): border
        // pieces by representative slot, interior clusters S + their new state.
        // Lane = column: a site's entry, its label's node, seldom a third one.
        const bool gather = (F & (FEAT_CSIZE | FEAT_PCC)) && (csz || ext);
        if (!gather && !last_start && tw == G::TX && th == G::TY && td == G::TZ) {
#pragma unroll 2
            for (int i = 0; i < LR; i += 4) {
                int v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = sm.f.par[lrow(i + e) * G::PW + lx];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((uint32_t)v[e] < INFO_INTERIOR) v[e] = sm.f.par[v[e]];   // records: negative or >= INFO_INTERIOR
                while (min(min((uint32_t)v[0], (uint32_t)v[1]), min((uint32_t)v[2], (uint32_t)v[3])) < INFO_INTERIOR) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((uint32_t)v[e] < INFO_INTERIOR) v[e] = sm.f.par[v[e]];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) code[lrow(i + e) * G::TX + lx] = (uint16_t)v[e];
            }
        } else {
            // Cluster sizes and piece masks, gathered down the lane's rows and added
            // when its cluster changes: a size goes to bits 16-30 of the root's
            // record (a piece or cluster holds at most 8192 sites; the codes read
            // bits 0-15 only), the coordinates of a border piece to its masks.
            int cur = -1, cur_v = 0;
            uint32_t cur_rows = 0u;
            auto flush = [&]() {
                if (!cur_rows) return;
                if (csz) atomicAdd(&sm.f.par[cur], __popc(cur_rows) << 16);
                if (ext && cur_v < 0) {
                    uint32_t *pm = sm.pm[cur_v & 0xFFFF];
                    if (DIM == 2) {
                        atomicOr(pm + (warp % TWW), 1u << lane);
                        const int y0 = LR * (warp / TWW);
                        atomicOr(pm + 4 + (y0 >> 5), cur_rows << (y0 & 31));
                    } else {
                        // bits y and 16 + z of the rows (bit 4 zz + yy of the mask)
                        uint32_t ys = cur_rows | (cur_rows >> 16);
                        ys |= ys >> 8;
                        ys |= ys >> 4;
                        uint32_t zs = cur_rows | (cur_rows >> 1);
                        zs = (zs | (zs >> 2)) & 0x11111111u;   // bit 4 zz
                        zs = (zs | (zs >> 3)) & 0x03030303u;
                        zs = (zs | (zs >> 6)) & 0x000F000Fu;
                        zs = (zs | (zs >> 12)) & 0xFFu;
                        atomicOr(pm, 1u << lane);
                        atomicOr(pm + 1, ((ys & 0xFu) << (4 * (warp & 3))) | (zs << (16 + LR / 4 * (warp >> 2))));
                    }
                }
            };
            for (int i = 0; i < LR; i += 4) {   // four rows' look-ups in flight
                int v[4], root[4];
                bool row[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = lrow(i + e);
                    row[e] = r % G::TY < th && r / G::TY < td;
                    root[e] = r * G::PW + lx;
                    v[e] = row[e] && lx < tw ? sm.f.par[root[e]] : (int)(INFO_INTERIOR | (uint32_t)S);
                }
                while (min(min((uint32_t)v[0], (uint32_t)v[1]), min((uint32_t)v[2], (uint32_t)v[3])) < INFO_INTERIOR) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((uint32_t)v[e] < INFO_INTERIOR) {
                            root[e] = v[e];
                            v[e] = sm.f.par[v[e]];
                        }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (!row[e]) continue;
                    const int r = lrow(i + e);
                    code[r * G::TX + lx] = (uint16_t)v[e];
                    if (lx >= tw) continue;
                    if (last_start && v[e] >= 0) p.label[gidx(lx, r % G::TY, r / G::TY)] = (int32_t)gfor(root[e]);
                    if (gather) {
                        const int key = csz ? root[e] : v[e];
                        if (key != cur) {
                            flush();
                            cur = key;
                            cur_v = v[e];
                            cur_rows = 0u;
                        }
                        cur_rows |= 1u << (i + e);
                    }
                }
            }
            if (gather) flush();
        }
        if (gather) {
            __syncthreads();
            if (ext)
                for (int w = tid; w < S * G::PMW; w += NT) p.pmask[nbase * G::PMW + w] = (&sm.pm[0][0])[w];
            if (csz) {
                // every root: an interior cluster adds its |C|^2; a border piece hands
                // its size to its representative node for the merge
                unsigned long long c2 = 0ull;
                for (uint32_t bits = roots; bits; bits &= bits - 1) {
                    const int v = sm.f.par[lrow(__ffs(bits) - 1) * G::PW + lx];
                    if (v < 0) {   // piece size: bits 16-30 (bit 31 is the border flag)
                        p.psize[nbase + (v & 0xFFFF)] = (int32_t)(((uint32_t)v >> 16) & 0x7FFFu);
                    } else if ((uint32_t)v >= INFO_INTERIOR) {   // bits 16-29 (bit 30 is the flag)
                        const unsigned long long size = ((uint32_t)v >> 16) & 0x3FFFu;
                        c2 += size * size;
                    }
                }
                warp_add64(&sm.acc_c2[1], c2);
                __syncthreads();
            }
        }
    }
    // the tile's sums (every contribution but a sweep's own csize2 was added
    // before a barrier above)
    if (tid < 4) {
        const int half = tid >> 1;            // 0: sweep j-1, 1: sweep j
        if (half == 0 ? fin : start) {
            DevObs *o = obs + (j - 1 + half);
            const long long v = sm.acc[tid];
            unsigned long long *dst = tid == 0 ? &o->bond_sum : tid == 1 ? &o->mag : tid == 2 ? &o->nbonds : &o->nclusters;
            if (v) atomicAdd(dst, (unsigned long long)v);
        }
    } else if ((F & FEAT_CSIZE) && tid < 6) {
        const int half = tid - 4;
        if (csz && (half == 0 ? fin : start) && sm.acc_c2[half])
            atomicAdd(&obs[j - 1 + half].csize2, sm.acc_c2[half]);
    }
}

// ------------------------------------------------ topological rule (RF_WIND)
// A cluster percolates when it winds around the box (Sec. III): some closed
// path of its bonds has a non-zero net displacement.  Every node carries its
// parent and its unwrapped displacement from that parent, one 16-byte word
// changed by 16-byte compare-and-swap so that the four move together; a root
// links to itself with displacement 0.  The displacements are exact: a set's
// nodes lift to a connected set of at most N sites, so they stay below 2^30.
__device__ __forceinline__ WLink wl_read(const WLink *w)
{
    // one 16-byte load, single-copy atomic as the swaps are (a swap by equal
    // words as the read serialised the walks of a big cluster at its root: 3D
    // L=256, T=2.0: 1956 us a sweep against 338)
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(w)
                 : "memory");
    return WLink{(int32_t)(uint32_t)lo, (int32_t)(uint32_t)(lo >> 32), (int32_t)(uint32_t)hi,
                 (int32_t)(uint32_t)(hi >> 32)};
}

// Root of x with pos(x) - pos(root); the walk halves the path (x's link is
// moved to its grandparent with the summed displacement: a failed swap means
// another walk moved it first).
__device__ __forceinline__ int wfind3(WLink *wl, int x, int &ox, int &oy, int &oz)
{
    ox = oy = oz = 0;
    WLink w = wl_read(wl + x);
    while (w.parent != x) {
        const WLink g = wl_read(wl + w.parent);
        if (g.parent != w.parent) {
            const WLink nw{g.parent, w.dx + g.dx, w.dy + g.dy, w.dz + g.dz};
            atomicCAS(wl + x, w, nw);
            ox += nw.dx;
            oy += nw.dy;
            oz += nw.dz;
            x = g.parent;
            w = wl_read(wl + x);
        } else {
            ox += w.dx;
            oy += w.dy;
            oz += w.dz;
            x = w.parent;
            w = g;
        }
    }
    return x;
}

// The link from node a to node b steps +1 along axis ax.  Roots of the same
// set: the cycle it closes has net displacement pos(a) + e_ax - pos(b) through
// the tree, non-zero exactly when it winds (recorded per axis).  Else the root
// of larger key hangs under the other with its displacement from it.
__device__ __forceinline__ void wunite3(WLink *wl, const int2 *node, int a, int b, int ax, DevObs *o)
{
    for (;;) {
        int oax, oay, oaz, obx, oby, obz;
        const int ra = wfind3(wl, a, oax, oay, oaz);
        const int rb = wfind3(wl, b, obx, oby, obz);
        // pos(rb) - pos(ra) = (pos(a) - off_a ... ) through the link: off_a + e_ax - off_b
        const int cx = oax + (ax == 0) - obx, cy = oay + (ax == 1) - oby, cz = oaz + (ax == 2) - obz;
        if (ra == rb) {
            if (cx) atomicOr(&o->spans_x, 1);
            if (cy || cz) atomicOr(&o->spans_y, 1);   // y, or in 3D y or z
            return;
        }
        const bool a_lo = (uint32_t)node[ra].y < (uint32_t)node[rb].y;
        const int lo = a_lo ? ra : rb, hi = a_lo ? rb : ra;
        const WLink root{hi, 0, 0, 0};
        const WLink nl = a_lo ? WLink{lo, cx, cy, cz} : WLink{lo, -cx, -cy, -cz};
        const WLink old = atomicCAS(wl + hi, root, nl);
        if (old.parent == hi && old.dx == 0 && old.dy == 0 && old.dz == 0) return;
    }
}

// ------------------------------------------------------------------ merge
template <int DIM>
struct PMC {
    // threads of the union kernel (two links each a pass) and of the others;
    // measured over 2D 64-128 and 96-192, 3D 128-512 and 160-640: 3D L=512,
    // q=2 within 1% from 320 / 256 to 384 / 320, which is the best of the small
    // lattices (L=50 PCC with the topological rule 97 us a sweep against 102)
    static constexpr int UT = DIM == 2 ? 96 : 384;
    static constexpr int UB = DIM == 2 ? 21 : 5;          // its blocks per SM (WB: with the topological rule)
    static constexpr int WB = DIM == 2 ? 12 : 3;
    static constexpr int MT = DIM == 2 ? 64 : 320;
    static constexpr int NPT = PG<DIM>::S / MT;           // slots per thread
    static constexpr int CT = DIM == 2 ? 384 : 512;       // threads of the cover kernel
    static_assert(PG<DIM>::S % MT == 0 && PG<DIM>::S % 16 == 0, "merge launch shape");
};

// Master step 2 of Sec. II.A on the face nodes: link e of a tile joins slot
// f of its + face along axis a to slot f of the - face of the next tile
// along a (e = f, F0 + f, F0 + F1 + f for a = 0, 1, 2); union by key, the
// finds of a thread's two links advancing in lock step.  (A per-block
// shared-memory forest that filters links joining pieces already joined, as
// the Ising merge has, made the 3D merge slower: its pieces are small and
// seldom meet twice.)
template <int DIM, bool W>
__global__ void __launch_bounds__(PMC<DIM>::UT, W ? PMC<DIM>::WB : PMC<DIM>::UB) k_pmerge_union(const PottsDev p, int j, DevObs *obs)
{
    const bool late = W || (p.flags & RF_PCC) || chain_crowds(p.ntiles);   // (sw_device.cuh)
    if (!late) chain_next();
    chain_wait();
    if (late) chain_next();
    using G = PG<DIM>;
    using MC = PMC<DIM>;
    constexpr int S = G::S, EPT = 2;
    __shared__ uint16_t links[G::FT];   // the bonded crossing links
    const int lt = blockIdx.x;
    if ((p.flags & RF_PCC) && lt == 0 && threadIdx.x < DIM) p.ncand[threadIdx.x] = 0;
    const PTile t = ptile_of<DIM>(p, lt);
    const uint32_t *cross = p.cross + (size_t)lt * G::CW;
    const int total = list_bits<G::CW, MC::UT>([&](int w) { return cross[w]; }, links);
    __syncthreads();
    for (int i0 = threadIdx.x; i0 < total; i0 += EPT * MC::UT) {
        int na[EPT], nb[EPT], ax[EPT];
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq) {
            const int i = i0 + qq * MC::UT;
            na[qq] = -1;
            ax[qq] = 0;
            if (i < total) {
                const int e = links[i];
                const int a = e < G::F0 ? 0 : e < G::F0 + G::F1 ? 1 : 2;
                const int f = e - (a == 0 ? 0 : a == 1 ? G::F0 : G::F0 + G::F1);
                na[qq] = lt * S + face_off<DIM>(a, 1) + f;
                nb[qq] = (a == 0 ? t.nb[0] : a == 1 ? t.nb[1] : t.nb[2]) * S + face_off<DIM>(a, 0) + f;
                ax[qq] = a;
            }
        }
        if (W && (p.flags & RF_WIND)) {
            WLink *wl = reinterpret_cast<WLink *>(p.wlink);
#pragma unroll
            for (int qq = 0; qq < EPT; ++qq)
                if (na[qq] >= 0) wunite3(wl, p.node, na[qq], nb[qq], ax[qq], obs + j);
            continue;
        }
        int pa[EPT], pb[EPT], ka[EPT], kb[EPT];
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq) {
            if (na[qq] < 0) continue;
            const int2 va = nload(p.node + na[qq]), vb = nload(p.node + nb[qq]);
            pa[qq] = va.x;
            ka[qq] = va.y;
            pb[qq] = vb.x;
            kb[qq] = vb.y;
        }
        bool live[EPT];
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq) live[qq] = na[qq] >= 0;
        // First try, one compare-and-swap: hang the larger-key one of the two
        // pieces' representatives under the other.  Every parent carries a smaller
        // key than its children, so a root of key k holds no node of smaller key:
        // if that representative is still a root, the two sets differ and the
        // link joins them (its new parent need not be a root).
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq) {
            if (!live[qq]) continue;
            const bool ra = ((uint32_t)ka[qq] & KEY_REP) != 0u, rb = ((uint32_t)kb[qq] & KEY_REP) != 0u;
            const int u = ra ? na[qq] : pa[qq], v = rb ? nb[qq] : pb[qq];
            if (u == v) {
                live[qq] = false;
                continue;
            }
            const bool u_hi = ((uint32_t)ka[qq] & KEY_MASK) > ((uint32_t)kb[qq] & KEY_MASK);
            const int hi = u_hi ? u : v, lo = u_hi ? v : u;
            // a representative whose parent was read as another node is no root
            const bool inner = u_hi ? (ra && pa[qq] != na[qq]) : (rb && pb[qq] != nb[qq]);
            if (!inner && atomicCAS(&p.node[hi].x, hi, lo) == hi) live[qq] = false;
        }
        // the remaining unions in lock step (path splitting on the way up; the
        // larger key's root is hung under the smaller by compare-and-swap)
        int xa[EPT], xb[EPT], sa[EPT], sb[EPT];
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq) {
            xa[qq] = na[qq];
            xb[qq] = nb[qq];
            sa[qq] = sb[qq] = -1;
        }
        for (;;) {
            bool more = false;
#pragma unroll
            for (int qq = 0; qq < EPT; ++qq) {
                if (!live[qq]) continue;
                const bool ra = pa[qq] == xa[qq], rb = pb[qq] == xb[qq];
                if (!ra || !rb) {
                    // path splitting rewrites representatives only: a slot that
                    // is not one keeps its own representative as its parent
                    if (!ra) {
                        if (sa[qq] >= 0) pstore(p.node + sa[qq], pa[qq]);
                        sa[qq] = ((uint32_t)ka[qq] & KEY_REP) ? xa[qq] : -1;
                        xa[qq] = pa[qq];
                    }
                    if (!rb) {
                        if (sb[qq] >= 0) pstore(p.node + sb[qq], pb[qq]);
                        sb[qq] = ((uint32_t)kb[qq] & KEY_REP) ? xb[qq] : -1;
                        xb[qq] = pb[qq];
                    }
                    more = true;
                } else if (xa[qq] == xb[qq]) {
                    live[qq] = false;
                } else {
                    const bool a_lo = ka[qq] < kb[qq];
                    const int lo = a_lo ? xa[qq] : xb[qq], hi = a_lo ? xb[qq] : xa[qq];
                    if (atomicCAS(&p.node[hi].x, hi, lo) == hi) live[qq] = false;
                    else more = true;
                }
            }
            if (!more) break;
#pragma unroll
            for (int qq = 0; qq < EPT; ++qq) {
                if (!live[qq]) continue;
                const int2 va = nload(p.node + xa[qq]), vb = nload(p.node + xb[qq]);
                pa[qq] = va.x;
                ka[qq] = va.y;
                pb[qq] = vb.x;
                kb[qq] = vb.y;
            }
        }
    }
}

// Every representative that is not its cluster's root walks to the root r and
// takes r's state, which the tile kernel left in kstate (Sec. I step 3; nstate
// itself the tile kernel must not write: its neighbours read it for their
// halos meanwhile).  On the last sweep of a call every representative also stores
// its root's key (the label); under PCC it points every node of its walk at r.
// A slot that is not a representative then takes its representative's state
// (its parent, in the same tile: the unions rewrite representatives only) for
// the neighbour's halo.  Counts the clusters that
// touch a tile face (one root node each).
template <int DIM, bool W>
__global__ void __launch_bounds__(PMC<DIM>::MT) k_pmerge_resolve(const PottsDev p, int j, bool last, uint64_t sweep0, DevObs *obs)
{
    const bool late = W || (p.flags & RF_PCC) || chain_crowds(p.ntiles);   // (sw_device.cuh)
    if (!late) chain_next();
    chain_wait();
    if (late) chain_next();
    using MC = PMC<DIM>;
    const int base = blockIdx.x * PG<DIM>::S;
    // under the topological rule the forest lives in the node links (their
    // first word is the parent); node.x keeps each node's representative
    const bool wind = W && (p.flags & RF_WIND);
    const int32_t *wpar = reinterpret_cast<const int32_t *>(p.wlink);
    auto parent = [&](int x) { return wind ? gload(wpar + 4 * (size_t)x) : pload(p.node + x); };
    __shared__ alignas(16) uint8_t rst[PG<DIM>::S];   // the new state of every slot
    __shared__ int2 walks[PG<DIM>::S];   // representatives that are no roots: slot, parent
    __shared__ int nwalks;
    // under the topological rule the unions have recorded the flags: feed back
    if (wind && (p.flags & RF_PCC) && base == 0 && threadIdx.x == 0)
        pcc_feedback(p.thr_dev, obs[j].spans_x | obs[j].spans_y, sweep0 + (uint64_t)j);
    if (threadIdx.x == 0) nwalks = 0;
    // (every slot's state, kept for the representatives below)
    for (int i = threadIdx.x; i < PG<DIM>::S / 16; i += MC::MT)
        reinterpret_cast<uint4 *>(rst)[i] = reinterpret_cast<const uint4 *>(p.kstate + base)[i];
    bool is_rep[MC::NPT];
    int rep[MC::NPT];
#pragma unroll
    for (int qq = 0; qq < MC::NPT; ++qq) {
        const int2 v = nload(p.node + base + threadIdx.x + qq * MC::MT);
        is_rep[qq] = ((uint32_t)v.y & KEY_REP) != 0u;
        rep[qq] = v.x;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    int nroots = 0;
#pragma unroll
    for (int qq = 0; qq < MC::NPT; ++qq) {
        const int s = threadIdx.x + qq * MC::MT, n = base + s;
        const int up = wind && is_rep[qq] ? parent(n) : rep[qq];
        const bool walk = is_rep[qq] && up != n;
        if (is_rep[qq] && !walk) {   // a cluster's root: its own state
            ++nroots;
            if (p.flags & RF_CSIZE) atomicAdd(p.csize + n, p.psize[n]);
            if (last) p.nfinal[n] = (uint32_t)p.node[n].y & KEY_MASK;
        }
        const unsigned m = __ballot_sync(FULL, walk);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&nwalks, __popc(m));
        at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (walk) walks[at] = make_int2(s, up);
    }
    __syncthreads();
    const bool ext = (p.flags & RF_PCC) != 0 && !wind;   // PCC by the extension rule
    for (int i = threadIdx.x; i < nwalks; i += MC::MT) {
        const int2 w = walks[i];
        const int n = base + w.x;
        int r = w.y;
        for (int up = parent(r); up != r; up = parent(r)) r = up;
        if (ext) {
            // the cover kernel reads a representative's root from its parent
            for (int x = n; x != r;) {
                const int nx = pload(p.node + x);
                pstore(p.node + x, r);
                x = nx;
            }
        }
        if (p.flags & RF_CSIZE) atomicAdd(p.csize + r, p.psize[n]);
        if (last) p.nfinal[n] = (uint32_t)p.node[r].y & KEY_MASK;
        rst[w.x] = p.kstate[r];
    }
    __syncthreads();
    if (ext) {
        // the roots of the "-" face nodes of the tiles of coordinate 0 along an
        // axis are that axis's candidates (cid = id + 2)
        const PTile t = ptile_of<DIM>(p, blockIdx.x);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            if (t.c[a] != 0) continue;
            const int n0 = base + face_off<DIM>(a, 0), nf = a == 0 ? PG<DIM>::F0 : a == 1 ? PG<DIM>::F1 : PG<DIM>::F2;
            for (int f = threadIdx.x; f < nf; f += MC::MT) {
                const int2 v = nload(p.node + n0 + f);
                if (v.x == NODE_NONE) continue;
                // a representative's parent is its root by now, another slot's its representative
                const int r = ((uint32_t)v.y & KEY_REP) ? v.x : pload(p.node + v.x);
                int32_t *c = p.cid + (size_t)r * DIM + a;
                if (gload(c) == 0 && atomicCAS(c, 0, 1) == 0)
                    *(volatile int32_t *)c = atomicAdd(p.ncand + a, 1) + 2;   // < F + 2: at most one per face site
            }
        }
    }
    // a slot that is not a representative (whose parent is still its own
    // representative in this tile) takes its cluster's new state too: the
    // neighbour's halo reads it with one load.  (Slots past the tile's sites
    // keep whatever they have: nobody reads them.)
#pragma unroll
    for (int qq = 0; qq < MC::NPT; ++qq)
        if (!is_rep[qq] && rep[qq] != NODE_NONE) rst[threadIdx.x + qq * MC::MT] = rst[rep[qq] - base];
    __syncthreads();
    for (int i = threadIdx.x; i < PG<DIM>::S / 16; i += MC::MT)
        reinterpret_cast<uint4 *>(p.nstate + base)[i] = reinterpret_cast<const uint4 *>(rst)[i];
    nroots = __reduce_add_sync(FULL, nroots);
    if (lane == 0 && nroots) atomicAdd(&obs[j].nclusters, (unsigned long long)nroots);
}

// ------------------------------------------------------------------- PCC
// The extension rule in d dimensions (Sec. III): a cluster spans axis a iff
// it occupies all L hyperplanes perpendicular to a.  Such a cluster holds a
// site of the hyperplane a = 0, on the - face of a tile of tile coordinate 0
// along a: the resolve kernel made those nodes' roots the candidates (cid of
// the root node, per axis: id + 2).  Here every border piece ORs the coordinates
// it occupies along a into its candidate root's coverage (L bits): in 3D, where a
// piece has one word an axis and the candidates of a face are many, the bits
// that were not there yet are added to the candidate's count, and a count of
// L spans; in 2D the last block checks the candidates' words (most fail at the
// first).  spans_x reports axis x, spans_y y, in 3D y or z.  Interior clusters
// touch no face and span nothing.  The last block to finish (a counter after a
// fence: no block waits) applies the feedback.
template <int DIM>
__global__ void __launch_bounds__(PMC<DIM>::CT) k_ppcc_cover(const PottsDev p, int j, uint64_t sweep0, DevObs *obs)
{
    using G = PG<DIM>;
    constexpr int CT = PMC<DIM>::CT;
    chain_wait();   // (the tile kernel starts when this one ends: sw_device.cuh)
    const int lt = blockIdx.x;
    const PTile t = ptile_of<DIM>(p, lt);
    const uint32_t W = ((uint32_t)p.L + 31u) / 32u;
    const int64_t F = DIM == 2 ? (int64_t)p.L : (int64_t)p.L * p.L;
    DevObs *o = obs + j;
    for (int s = threadIdx.x; s < G::S; s += CT) {
        const size_t n = (size_t)lt * G::S + s;
        const int2 v = nload(p.node + n);
        uint32_t m[G::PMW];
#pragma unroll
        for (int w = 0; w < G::PMW; ++w) m[w] = p.pmask[n * G::PMW + w];
        if (!((uint32_t)v.y & KEY_REP)) continue;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const int c = p.cid[(size_t)v.x * DIM + a];
            if (c < 2) continue;
            uint32_t *cov = p.cov + ((size_t)a * F + (size_t)(c - 2)) * W + (size_t)(t.o[a] >> 5);
            if constexpr (DIM == 2) {
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const uint32_t bits = a == 0 ? m[w] : w < 2 ? m[G::PMW - 2 + w] : 0u;
                    if (bits) atomicOr(cov + w, bits);
                }
            } else {
                // 32-site x words; 16-site y and z halves at an origin that is a
                // multiple of 16
                const uint32_t half = a == 0 ? m[0] : a == 1 ? (m[1] & 0xFFFFu) : (m[1] >> 16);
                const uint32_t bits = a == 0 ? half : half << (t.o[a] & 31);
                if (!bits) continue;
                const int fresh = __popc(bits & ~atomicOr(cov, bits));
                if (fresh && atomicAdd(p.ccount + a * F + (c - 2), fresh) + fresh == p.L)
                    atomicOr(a == 0 ? &o->spans_x : &o->spans_y, 1);
            }
        }
    }
    __shared__ int is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(p.ncand + 3, 1) == (int)gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!is_last) return;   // else: every other block's coverage and flags are visible
    if constexpr (DIM == 2) {
        for (int a = 0; a < 2; ++a) {
            const uint32_t *cov = p.cov + (size_t)a * F * W;
            const int nc = p.ncand[a];
            int span = 0;
            for (int id = threadIdx.x; id < nc; id += CT) {
                bool full = true;
                for (uint32_t w = 0; w < W && full; ++w) {
                    const uint32_t m = valid_mask((int)w, p.L);
                    full = (cov[(size_t)id * W + w] & m) == m;
                }
                span |= full;
            }
            span = __syncthreads_or(span);
            if (threadIdx.x == 0) (a == 0 ? o->spans_x : o->spans_y) = span;
        }
    }
    if (threadIdx.x != 0) return;
    p.ncand[3] = 0;
    const int flags = *(volatile int32_t *)&o->spans_x | *(volatile int32_t *)&o->spans_y;
    pcc_feedback(p.thr_dev, flags, sweep0 + (uint64_t)j);
}

// ------------------------------------------------------------ small kernels
__global__ void k_potts_hot_start(const PottsDev p)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.N) return;
    const U4 r = philox4x32_10((uint32_t)(i >> 2), 0u, 0u, STREAM_INIT, (uint32_t)p.seed, (uint32_t)(p.seed >> 32));
    p.spin[i] = potts_state(u4_word(r, (int)(i & 3)), p.q);
}

// Sets *bad if any of the n states is >= q.
__global__ void k_potts_check(const uint8_t *s, int64_t n, int q, int32_t *bad)
{
    int found = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        found |= s[i] >= q;
    if (__syncthreads_or(found) && threadIdx.x == 0) atomicOr(bad, 1);
}

// The tile kernels' dynamic shared-memory limit, raised once per device.
constexpr int PREP_DEVICES = 64;
cudaError_t potts_prepare()
{
    static std::mutex mu;
    static bool done[PREP_DEVICES] = {};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= PREP_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (done[dev]) return cudaSuccess;
    auto set = [&](auto... k) {
        ((err = err == cudaSuccess ? cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)std::max(ptile_smem<2>(true), ptile_smem<3>(true)))
                                   : err),
         ...);
    };
    set(k_ptile<2, 0, 1>, k_ptile<2, FEAT_TILE, 1>, k_ptile<2, 0, 2>, k_ptile<2, FEAT_TILE, 2>, k_ptile<2, 0, 4>,
        k_ptile<2, FEAT_TILE, 4>, k_ptile<3, 0, 1>, k_ptile<3, FEAT_TILE, 1>, k_ptile<3, 0, 2>, k_ptile<3, FEAT_TILE, 2>,
        k_ptile<3, 0, 4>, k_ptile<3, FEAT_TILE, 4>);
    if (err == cudaSuccess) done[dev] = true;
    return err;
}

bool all_shared(const PottsDev &p)
{
    return chain_all_shared(p.ntiles, (p.flags & RF_PCC) != 0, (p.flags & RF_WIND) != 0);
}

template <int DIM, int M>
cudaError_t launch_tile_cta(const PottsDev &p, int j, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st,
                            bool chained)
{
    const bool feat = (p.flags & (RF_PCC | RF_OPEN | RF_CSIZE | RF_WIND)) != 0;
    return launch_kernel(feat ? k_ptile<DIM, FEAT_TILE, M> : k_ptile<DIM, 0, M>, dim3((unsigned)p.ntiles), M * PG<DIM>::WT,
                         ptile_smem<DIM>((p.flags & RF_PCC) && !(p.flags & RF_WIND)), st, chained, all_shared(p), p, j,
                         nsweeps, sweep0, obs);
}

// M, the warps of a tile CTA by eights: a warp's rows in the labelling, its records and
// its codes are a chain that an SM with one or two CTAs cannot hide, and more warps
// have fewer rows each.  M = 4 up to two thirds of a CTA an SM (beyond, the blocks of
// the next kernels have no room beside one), M = 2 up to two CTAs an SM in 2D and four
// in 3D.  M = 1, 2 and 4, us a sweep at T_c: 2D, q=3, L=300 28.0, 24.3, 23.7; L=1024
// 32.9, 29.6, 30.7; L=1500 45.6, 38.9; L=1700 45.6, 50.8; 3D, q=2, L=50 41.4, 32.9,
// 30.6; L=96 50.8, 36.9, 38.1; L=128 71.3, 49.3; L=160 90.4, 83.9; L=200 136, 149; PCC
// by the topological rule in 3D, L=50 64.2, 52.1, 49.4.
template <int DIM>
cudaError_t launch_tile(const PottsDev &p, int j, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st,
                        bool chained)
{
    if (3 * p.ntiles <= 2 * FIRST_WAVE_SMS) return launch_tile_cta<DIM, 4>(p, j, nsweeps, sweep0, obs, st, chained);
    if (p.ntiles <= (DIM == 2 ? 2 : 4) * FIRST_WAVE_SMS)
        return launch_tile_cta<DIM, 2>(p, j, nsweeps, sweep0, obs, st, chained);
    return launch_tile_cta<DIM, 1>(p, j, nsweeps, sweep0, obs, st, chained);
}

template <int DIM>
cudaError_t launch_merge(const PottsDev &p, int j, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st,
                         bool chained)
{
    constexpr int MT = PMC<DIM>::MT;
    const bool pcc = (p.flags & RF_PCC) != 0, wind = (p.flags & RF_WIND) != 0;
    const dim3 tiles((unsigned)p.ntiles);
    cudaError_t e = cudaSuccess;
    auto go = [&](auto *k, dim3 grid, unsigned threads, auto... args) {
        if (e == cudaSuccess) e = launch_kernel(k, grid, threads, 0, st, chained, all_shared(p), args...);
    };
    const bool last = j == nsweeps - 1;
    if (wind) {
        go(k_pmerge_union<DIM, true>, tiles, PMC<DIM>::UT, p, j, obs);
        go(k_pmerge_resolve<DIM, true>, tiles, MT, p, j, last, sweep0, obs);
    } else {
        // no pointer-jumping round, here or above: after the unions'
        // single-swap links the walks are short, and the round cost more than it
        // saved (3D 2.99 -> 2.94 ms a sweep without it; the topological rule at
        // L=128 146 -> 135 us)
        go(k_pmerge_union<DIM, false>, tiles, PMC<DIM>::UT, p, j, obs);
        go(k_pmerge_resolve<DIM, false>, tiles, MT, p, j, last, sweep0, obs);
    }
    if (pcc && !wind) go(k_ppcc_cover<DIM>, tiles, PMC<DIM>::CT, p, j, sweep0, obs);
    return e;
}

}  // namespace

namespace swg {

void potts_geometry(int dim, int L, PottsGeometry *g)
{
    const int tx = dim == 2 ? PG<2>::TX : PG<3>::TX, ty = dim == 2 ? PG<2>::TY : PG<3>::TY;
    const int tz = dim == 2 ? PG<2>::TZ : PG<3>::TZ;
    g->ntx = (L + tx - 1) / tx;
    g->nty = (L + ty - 1) / ty;
    g->ntz = dim == 2 ? 1 : (L + tz - 1) / tz;
    g->ntiles = g->ntx * g->nty * g->ntz;
    g->sites_per_tile = dim == 2 ? PG<2>::NS : PG<3>::NS;
    g->slots = dim == 2 ? PG<2>::S : PG<3>::S;
    g->cross_words = dim == 2 ? PG<2>::CW : PG<3>::CW;
    g->pmask_words = dim == 2 ? PG<2>::PMW : PG<3>::PMW;
}

cudaError_t potts_enqueue_hot_start(const PottsDev &p, cudaStream_t st)
{
    cudaError_t e = potts_prepare();
    if (e != cudaSuccess) return e;
    k_potts_hot_start<<<(unsigned)((p.N + PT - 1) / PT), PT, 0, st>>>(p);
    return cudaGetLastError();
}

// Launch j of a call of nsweeps sweeps: the tile kernel (finishing sweep
// j-1, starting sweep j) ...
cudaError_t potts_enqueue_tile(const PottsDev &p, int j, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st,
                               bool chained)
{
    cudaError_t e = potts_prepare();
    if (e != cudaSuccess) return e;
    return p.dim == 2 ? launch_tile<2>(p, j, nsweeps, sweep0, obs, st, chained)
                      : launch_tile<3>(p, j, nsweeps, sweep0, obs, st, chained);
}

// ... and, for j < nsweeps, the merge of sweep j.
cudaError_t potts_enqueue_merge(const PottsDev &p, int j, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st,
                                bool chained)
{
    return p.dim == 2 ? launch_merge<2>(p, j, nsweeps, sweep0, obs, st, chained)
                      : launch_merge<3>(p, j, nsweeps, sweep0, obs, st, chained);
}

// The launches of one call of nsweeps sweeps: tile kernel j = 0 .. nsweeps,
// each but the last followed by the merge of sweep j.
cudaError_t potts_enqueue_sweeps(const PottsDev &p, int nsweeps, uint64_t sweep0, DevObs *obs, cudaStream_t st)
{
    for (int j = 0; j <= nsweeps; ++j) {
        cudaError_t e = potts_enqueue_tile(p, j, nsweeps, sweep0, obs, st, j > 0);
        if (e == cudaSuccess && j < nsweeps) e = potts_enqueue_merge(p, j, nsweeps, sweep0, obs, st, true);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t potts_enqueue_check(const uint8_t *s, int64_t n, int q, int32_t *bad, cudaStream_t st)
{
    const unsigned nb = (unsigned)std::min<int64_t>((n + 4095) / 4096, 4096);
    k_potts_check<<<nb > 0 ? nb : 1, PT, 0, st>>>(s, n, q, bad);
    return cudaGetLastError();
}

}  // namespace swg
