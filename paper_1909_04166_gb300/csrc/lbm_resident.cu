// Resident step kernel: a run of many time steps of a grid small enough to be held in the shared
// memory of the GPU's SMs, in one cooperative launch.
//
// Every block owns a strip of 64 columns and a range of rows and keeps their populations in
// shared memory for the whole run, with a ring of ghost nodes around them; the state buffer is
// read once at the start and written once at the end.  A time step of a block:
//   S  phi = sum f and p* = sum g-bar of every node and ghost node, into two arrays;
//   C  a warp takes a row (64 nodes, two per lane) or, where the block has at most half as many
//      rows as warps, half a row (32 nodes, one per lane): stencils, forces, both collisions in
//      registers, then, after a block barrier (every population of the round's rows is in
//      registers), the pushes in place, into the same array;
//   X  the populations that landed on the two outermost rings (the block's own boundary nodes
//      and its ghost nodes) go to the neighbouring blocks that hold the same nodes.
// With the ghost nodes' populations completed by their owners, the next S forms their phi and p*
// here, so a step needs one exchange, and no barrier over the grid: a message is a 16-byte word
// of two populations, each beside the number of the step, written straight into the receiver's
// mailbox and polled there until both halves carry the step's number (64-bit accesses are atomic,
// so a word validates itself and no fence is needed).  Mailboxes alternate with the step's parity:
// a block sends step t + 2 only after the messages of step t + 1 of all its neighbours have
// arrived, which those sent after reading step t's.
//
// A batch is taken in waves of cases whose blocks fit on the device together, one launch a wave for
// all the steps of a run: a case's neighbours are its own blocks, so cases never wait for each other.
//
// Per node the arithmetic is the paired march's of lbm_step.cu (F2, or F1 with the same
// roundings), the zeroth moments are summed in its orders (in plane order; in the halo's tree
// order for the columns next to a strip), and the 16-bit forms round every pushed population as
// it does (held as floats here: the rounded values are exact in FP32).  The state is the same
// bit for bit.
//
// What bounds it: on small grids the latency of a step, on the largest that fit the FP32 pipes (a
// packed operation takes two issue slots of a quarter SM).  One GB300, FP32, us a step over 200
// steps, this kernel against the faster of graph replays and the multi-step kernel, and in
// parentheses without the exchange (a timing probe): 64 x 64 2.3 against 3.8 (0.8), 51 x 201
// 2.4 against 4.3 (1.2), 161 x 481 3.7 against 6.7 (2.3), 512 x 256 4.1 against 7.3 (2.7),
// 256 x 1024 5.9 against 10.8 (4.6), the interface lattice alone 800 x 800 8.0 against 11.9
// (5.9); with BF16 storage 512 x 256 5.2 against 8.2 (3.6).  Of the exchange's 1.4 us about 0.5
// go into the sends (20 KB a block through its port), 0.75 into one read of the mailbox from L2
// and 0.25 into waiting.  Measured and not kept: a thread per ring node polling its messages and
// summing them directly (more polls in flight: 2.57 and 6.94 us at 64 x 64 and 256 x 1024 where
// this measured 2.33 and 6.3), two blocks of 8 warps per SM (3.2 and 8.2), a pause before or
// between the polls (no gain).
#include "lbm_device.cuh"
#include "lbm_resident.h"

#include <type_traits>
#include <vector>

namespace cmlbm {

namespace {

constexpr int NW = kResidentWarps;
constexpr int NT = NW * 32;
constexpr int RW = 66;   // floats of a plane of a row: west ghost, 64 columns, east ghost

// Polling bound: two seconds of the global timer (a neighbour's step takes microseconds).
constexpr unsigned long long kBoxWaitNs = 2000000000ull;

template <int V>
__host__ __device__ constexpr int row_floats() { return ((V & kVarShear) ? 9 : 18) * RW + 1; }   // odd: a column
                                                                           // walk hits all banks

__device__ __forceinline__ void st_box(ulonglong2* p, unsigned tag, float a, float b)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p),
                 "l"(t | __float_as_uint(a)), "l"(t | __float_as_uint(b))
                 : "memory");
}
__device__ __forceinline__ ulonglong2 ld_box(const ulonglong2* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
                 : "=l"(v.x), "=l"(v.y)
                 : "l"(p)
                 : "memory");
    return v;
}

// A lane's nodes: columns c and c + 32 of a row as F2, or column c alone as F1.
template <class T> struct Lane;
template <> struct Lane<F2> {
    static __device__ __forceinline__ F2 ld(const float* p) { return F2(p[0], p[32]); }
    static __device__ __forceinline__ F2 of(float a, float b) { return F2(a, b); }
    static __device__ __forceinline__ float half(F2 v, bool b) { return b ? v.v.y : v.v.x; }
};
template <> struct Lane<F1> {
    static __device__ __forceinline__ F1 ld(const float* p) { return F1(p[0]); }
    static __device__ __forceinline__ F1 of(float a, float) { return F1(a); }
    static __device__ __forceinline__ float half(F1 v, bool) { return v.v; }
};

// Value of a lane's pushed populations after 16-bit rounding, and their scaled rounding errors:
// the roundings of encode_word (lbm_step.cu).
template <typename S>
__device__ __forceinline__ float2 round16(float2 d)
{
    if constexpr (std::is_same<S, __half>::value) return __half22float2(__float22half2_rn(d));
    else return __bfloat1622float2(__float22bfloat162_rn(d));
}
template <typename S, bool ADJ>
__device__ __forceinline__ F2 encode_lane(F2 v, F2 z, float w, float scale, F2 adj, F2& stored)
{
    F2 d = fmad(F2(-w), z, v) * F2(scale);
    if constexpr (ADJ) d = d - adj;
    stored = F2(round16<S>(d.v));
    return stored - d;
}
template <typename S, bool ADJ>
__device__ __forceinline__ F1 encode_lane(F1 v, F1 z, float w, float scale, F1 adj, F1& stored)
{
    F1 d = fmad(F1(-w), z, v) * F1(scale);
    if constexpr (ADJ) d = d - adj;
    stored = F1(round16<S>(make_float2(d.v, 0.0f)).x);
    return stored - d;
}

// The halo order of a column's zeroth moment: the butterfly over lanes 0 .. 15 that march2 runs
// (plane q in lane q, Z in lane 9 of the 16-bit forms, zeros above), as one thread evaluates it.
__device__ __forceinline__ float tree_sum(const float v[9], float z)
{
    const float s0 = __fadd_rn(v[0], v[8]), s1 = __fadd_rn(v[1], z);
    float s[8] = {s0, s1};
#pragma unroll
    for (int q = 2; q < 8; ++q) s[q] = __fadd_rn(v[q], 0.0f);
    const float t0 = __fadd_rn(s[0], s[4]), t1 = __fadd_rn(s[1], s[5]);
    const float t2 = __fadd_rn(s[2], s[6]), t3 = __fadd_rn(s[3], s[7]);
    return __fadd_rn(__fadd_rn(t0, t2), __fadd_rn(t1, t3));
}

// One block's place in the grid.
struct Block {
    int strip, seg;
    int x0, w;    // first column, columns (1 .. 64)
    int y0, h;    // first row, rows
};
__device__ __forceinline__ int seg_start(int seg, int nseg, int ny)
{
    return (int)((long long)seg * ny / nseg);
}
__device__ __forceinline__ int seg_rows_of(int seg, int nseg, int ny)
{
    return seg_start(seg + 1, nseg, ny) - seg_start(seg, nseg, ny);
}
__device__ __forceinline__ int strip_cols(int strip, int nx) { return min(64, nx - strip * 64); }

// Mailbox index of population a of block-local node (r, c), r = 0 .. h + 1 and c = -1 .. w
// (ghosts included), of the two outermost rings: the two lowest and two highest rows whole, of
// the other rows the two columns at each side.
__device__ __forceinline__ int box_index(int r, int c, int a, int h, int w, int hmax)
{
    const int zr = r < 2 ? r : (r >= h ? 2 + r - h : -1);
    if (zr >= 0) return (zr * 9 + a) * RW + c + 1;
    const int ci = c <= 0 ? c + 1 : c - w + 3;
    return 36 * RW + (ci * 9 + a) * (hmax - 2) + r - 2;
}

// Where the population that lands on node (r, c) in plane a came from, in block-local
// coordinates: its upstream neighbour, or beyond a wall the node it was reflected from.
__device__ __forceinline__ void upstream(const Geometry& G, const Block& B, int r, int c, int a,
                                         int& sr, int& sc)
{
    constexpr int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
    constexpr int EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    sr = r - EY[a];
    sc = c - EX[a];
    const int gx = B.x0 + sc, gy = B.y0 + sr - 1;
    const bool ox = G.wall_x && (gx < 0 || gx >= G.nx);
    const bool oy = G.wall_y && (gy < 0 || gy >= G.ny);
    if (!ox && !oy) return;
    const bool slip_x = ox && ((G.slip >> (gx < 0 ? 0 : 1)) & 1);
    const bool slip_y = oy && ((G.slip >> (gy < 0 ? 2 : 3)) & 1);
    const bool bounce = (ox && !slip_x) || (oy && !slip_y) || (ox && oy);
    if (bounce || ox) sc = c;   // reflected along x: it came along the wall from the same column
    if (bounce || oy) sr = r;
}

// Exchange lists of a block: in global memory as the setup kernel leaves them, in shared memory
// during a run.
struct Lists {
    unsigned* node;          // row << 16 | column + 1 of the nodes of the two outermost rings
    unsigned short* sdst;    // where a send goes: the neighbour's code << box_bits | mailbox index
    unsigned short* soff;    // float offset of its g-bar population
    unsigned short* rbox;    // index in the own mailbox of a received entry
    unsigned short* roff;    // float offset of its g-bar population
};
__host__ __device__ inline int ring_nodes(int h) { return 4 * RW + 4 * (h - 2); }
__host__ __device__ inline size_t list_words(int hmax, int tab)
{
    return ring_nodes(hmax) + 2 * tab;
}
__device__ __forceinline__ Lists lists_at(void* p, int hmax, int tab)
{
    Lists T;
    T.node = static_cast<unsigned*>(p);
    T.sdst = reinterpret_cast<unsigned short*>(T.node + ring_nodes(hmax));
    T.soff = T.sdst + tab;
    T.rbox = T.soff + tab;
    T.roff = T.rbox + tab;
    return T;
}
// Ring node j of a block: the two lowest and the two highest rows whole (66 columns each), then
// of the other rows the two columns at each side.
constexpr unsigned kNoNode = 0xffffffffu;   // entry of one beyond a wall
__device__ __forceinline__ void ring_node(int j, int h, int w, int& r, int& c)
{
    if (j < 4 * RW) {
        const int zr = j / RW;
        r = zr < 2 ? zr : h + zr - 2;
        c = j % RW - 1;
    } else {
        const int k = j - 4 * RW, ci = k / (h - 2);
        r = 2 + k % (h - 2);
        c = ci < 2 ? ci - 1 : w + ci - 3;
    }
}
__device__ __forceinline__ Block block_of(const Geometry& G, const ResidentGrid& D)
{
    const int b = (int)blockIdx.x - D.block0;
    Block B;
    B.strip = b % D.nstrip;
    B.seg = b / D.nstrip;
    B.x0 = B.strip * 64;
    B.w = strip_cols(B.strip, G.nx);
    B.y0 = seg_start(B.seg, D.nseg, G.ny);
    B.h = seg_rows_of(B.seg, D.nseg, G.ny);
    return B;
}

// A neighbour of a block: dx strips (-2 .. 2) and dy segments (-1 .. 1) away.  The blocks beyond
// the next strip hold a common node with this one where that strip, the last of the grid, is a
// single column.
struct Neighbour {
    bool exists;
    int strip, seg;
    int dc, dr;   // its column 0 and row 0 in this block's coordinates
};
__device__ __forceinline__ Neighbour neighbour(const Geometry& G, const Block& B,
                                               const ResidentGrid& D, int dx, int dy)
{
    Neighbour N;
    N.strip = B.strip + dx;
    N.seg = B.seg + dy;
    N.exists = (dx || dy) && !(G.wall_x && (N.strip < 0 || N.strip >= D.nstrip)) &&
               !(G.wall_y && (N.seg < 0 || N.seg >= D.nseg));
    N.strip = (N.strip + 2 * D.nstrip) % D.nstrip;
    N.seg = (N.seg + D.nseg) % D.nseg;
    const int between = (B.strip + dx / 2 + D.nstrip) % D.nstrip;   // for dx = -2, 2
    if ((dx == 2 || dx == -2) && strip_cols(between, G.nx) != 1) N.exists = false;
    N.dc = dx > 0 ? B.w + (dx == 2 ? 1 : 0)
                  : (dx < 0 ? -strip_cols(N.strip, G.nx) - (dx == -2 ? 1 : 0) : 0);
    N.dr = dy > 0 ? B.h : (dy < 0 ? -seg_rows_of(N.seg, D.nseg, G.ny) : 0);
    return N;
}
// The imposed-flow form (taller blocks, longer lists) has 13 bits for a mailbox index, and no
// single-column strips; the others 12.
template <int V> __host__ __device__ constexpr int reach() { return (V & kVarShear) ? 1 : 2; }
template <int V> __host__ __device__ constexpr int box_bits() { return (V & kVarShear) ? 13 : 12; }
template <int V>
__host__ __device__ constexpr int neighbour_code(int dx, int dy)   // below 1 << (16 - box_bits)
{
    const int k = (dy + 1) * (2 * reach<V>() + 1) + dx + reach<V>();
    return (V & kVarShear) && k > 4 ? k - 1 : k;
}

// Setup, once per plan: the exchange lists of every block, in the order of the mailbox
// (consecutive threads take consecutive columns; any order would do), after the numbers of
// sends and receives.
template <int V>
__device__ void build_lists(const Geometry& G, const ResidentGrid& D, const ResidentLaunch& L)
{
    __shared__ int count[2];
    const Block B = block_of(G, D);
    int* out = L.lists + blockIdx.x * (2 + list_words(L.hmax, L.tab));
    const Lists T = lists_at(out + 2, L.hmax, L.tab);
    if (threadIdx.x < 2) count[threadIdx.x] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < ring_nodes(B.h); j += NT) {
        int r, c;
        ring_node(j, B.h, B.w, r, c);
        const int gx = B.x0 + c, gy = B.y0 + r - 1;
        // (a single column of a side row would be there twice)
        bool ok = c <= B.w && !(B.w == 1 && j >= 4 * RW + 2 * (B.h - 2) && c == 0);
        if (G.wall_x && (gx < 0 || gx >= G.nx)) ok = false;
        if (G.wall_y && (gy < 0 || gy >= G.ny)) ok = false;
        T.node[j] = ok ? (unsigned)r << 16 | (unsigned)(c + 1) : kNoNode;
    }
    constexpr int ROWF = row_floats<V>();
    const int lane = threadIdx.x & 31;
    const int E = 36 * RW + 36 * max(L.hmax - 2, 0);
    for (int i0 = (threadIdx.x >> 5) * 32; i0 < E; i0 += NT) {
        const int i = i0 + lane;
        int r = -1, c = 0, a = 0;
        bool ok = i < E;
        if (ok) {
            if (i < 36 * RW) {
                const int zr = i / (9 * RW);
                a = i / RW % 9;
                c = i % RW - 1;
                r = zr < 2 ? zr : B.h + zr - 2;
            } else {
                const int k = i - 36 * RW, ci = k / (9 * (L.hmax - 2));
                a = k / (L.hmax - 2) % 9;
                r = 2 + k % (L.hmax - 2);
                c = ci < 2 ? ci - 1 : B.w + ci - 3;
            }
            ok = r <= B.h + 1 && c <= B.w && box_index(r, c, a, B.h, B.w, L.hmax) == i;
            const int gx = B.x0 + c, gy = B.y0 + r - 1;
            if (G.wall_x && (gx < 0 || gx >= G.nx)) ok = false;
            if (G.wall_y && (gy < 0 || gy >= G.ny)) ok = false;
        }
        int sr = 0, sc = 0;
        if (ok) upstream(G, B, r, c, a, sr, sc);
        const bool mine = sr >= 1 && sr <= B.h && sc >= 0 && sc < B.w;
        const unsigned short off = (unsigned short)(r * ROWF + a * RW + c + 1);
        auto append = [&](bool has, int which) {   // position in list `which`, one atomic a warp
            const unsigned m = __ballot_sync(FULL, has);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&count[which], __popc(m));
            base = __shfl_sync(FULL, base, 0);
            const int at = base + __popc(m & ((1u << lane) - 1));
            return has && at < L.tab ? at : -1;
        };
        const int ar = append(ok && !mine, 1);
        if (ar >= 0) {
            T.roff[ar] = off;
            T.rbox[ar] = (unsigned short)i;
        }
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -reach<V>(); dx <= reach<V>(); ++dx) {
                const Neighbour N = neighbour(G, B, D, dx, dy);
                const int c2 = c - N.dc, r2 = r - N.dr;
                const int w2 = strip_cols(N.strip, G.nx), h2 = seg_rows_of(N.seg, D.nseg, G.ny);
                const int as = append(ok && mine && N.exists && c2 >= -1 && c2 <= w2 && r2 >= 0 &&
                                          r2 <= h2 + 1,
                                      0);
                if (as >= 0) {
                    T.soff[as] = off;
                    T.sdst[as] = (unsigned short)(neighbour_code<V>(dx, dy) << box_bits<V>() |
                                                  box_index(r2, c2, a, h2, w2, L.hmax));
                }
            }
    }
    __syncthreads();
    if (threadIdx.x < 2) out[threadIdx.x] = count[threadIdx.x];
}

template <int V>
__global__ void __launch_bounds__(NT) resident_lists_kernel(Geometry G, ResidentGrid D,
                                                            ResidentLaunch L)
{
    build_lists<V>(G, D, L);
}
template <int V>
__global__ void __launch_bounds__(NT)
resident_batch_lists_kernel(const ResidentCase* __restrict__ cases,
                            const int* __restrict__ case_of, ResidentLaunch L)
{
    const ResidentCase& c = cases[case_of[blockIdx.x]];
    build_lists<V>(c.G, c.D, L);
}

// 16-byte accesses to the tiles of a block's rows: flat index -> (row, tile, access) and where its
// first element sits: plane p and column c (a 16-bit tile starts with its two Z planes, p = -2 and
// -1, in floats).
template <typename S, int V>
struct TileVec {
    static constexpr bool SHEAR = (V & kVarShear) != 0;
    static constexpr int TE = Tile<S>::ELEMS;
    static constexpr int EV = 16 / (int)sizeof(S);             // elements of an access
    static constexpr int TV0 = SHEAR ? 9 * 32 / EV : 0;        // first one of a tile that is needed
    static constexpr int TV = TE / EV - TV0;                   // and how many follow
    struct At { int r, t, q, p, c; };
    static __device__ __forceinline__ At at(int ntiles, int i)
    {
        At a;
        a.r = i / (ntiles * TV);
        const int k = i - a.r * (ntiles * TV);
        a.t = k / TV;
        a.q = k - a.t * TV + TV0;
        constexpr int ZV = Tile<S>::ZBYTES / 16;               // 8 accesses a Z plane
        if (a.q < ZV) {
            a.p = a.q / 8 - 2;
            a.c = 32 * a.t + a.q % 8 * 4;
        } else {
            a.p = (a.q - ZV) * EV / 32 - (SHEAR ? 9 : 0);
            a.c = 32 * a.t + (a.q - ZV) * EV % 32;
        }
        return a;
    }
};

__device__ __forceinline__ bool row_exists(const Geometry& G, const Block& B, int r)
{
    const int gy = B.y0 + r - 1;
    return !(G.wall_y && (gy < 0 || gy >= G.ny));
}
template <typename S>
__device__ __forceinline__ S* global_row(const Geometry& G, const Block& B, S* state, int r)
{
    return state + (long long)map_row(B.y0 + r - 1, G) * G.nstrips * Tile<S>::ELEMS;
}

// Load a block and its ghost ring: the tiles of every row 16 bytes at a time, several loads of a
// thread in flight, then the two ghost columns.  (Not inlined: the registers of the time loop.)
template <typename S, int V>
__device__ __noinline__ void load_block(S* state, Geometry G, Block B, float* pop, float* sps,
                                        float* sph, float* gz)
{
    using VA = TileVec<S, V>;
    constexpr bool SHEAR = VA::SHEAR, NARROW = Narrow<S>::value;
    constexpr int PL = SHEAR ? 9 : 18, ROWF = row_floats<V>();
    const int tid = threadIdx.x, h = B.h, w = B.w, ntiles = (w + 31) / 32;
    {
        constexpr int U = 4;
        const int total = (h + 2) * ntiles * VA::TV;
        for (int i0 = tid; i0 < total; i0 += U * NT) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const typename VA::At a = VA::at(ntiles, min(i0 + u * NT, total - 1));
                if (row_exists(G, B, a.r))
                    v[u] = *reinterpret_cast<const uint4*>(
                        global_row(G, B, state, a.r) + (long long)(B.x0 / 32 + a.t) * VA::TE + a.q * VA::EV);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (i0 + u * NT >= total) break;
                const typename VA::At a = VA::at(ntiles, i0 + u * NT);
                if (!row_exists(G, B, a.r)) continue;
                if (NARROW && a.p < 0) {
                    const float* z = reinterpret_cast<const float*>(&v[u]);
                    float* d = (a.p == -2 ? sps : sph) + a.r * RW + a.c + 1;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (a.c + e < w) d[e] = z[e];
                } else {
                    const S* q = reinterpret_cast<const S*>(&v[u]);
                    float* d = pop + a.r * ROWF + a.p * RW + a.c + 1;
#pragma unroll
                    for (int e = 0; e < VA::EV; ++e)
                        if (a.c + e < w) d[e] = narrow_to_f_or_self(q[e]);
                }
            }
        }
        constexpr int GP = PL + (NARROW ? 2 : 0);            // planes of a ghost column
        for (int i = tid; i < (h + 2) * 2 * GP; i += NT) {
            const int r = i / (2 * GP), side = i / GP % 2, p = i % GP;
            const int c = side ? w : -1, gx = B.x0 + c;
            if (!row_exists(G, B, r) || (G.wall_x && (gx < 0 || gx >= G.nx))) continue;
            const int x = map_col(gx, G);
            const S* tile = global_row(G, B, state, r) + (long long)(x >> 5) * VA::TE;
            if (p >= PL)
                gz[r * 4 + 2 * side + p - PL] =
                    reinterpret_cast<const float*>(tile)[32 * (p - PL) + (x & 31)];
            else
                pop[r * ROWF + p * RW + c + 1] = narrow_to_f_or_self(
                    tile[Tile<S>::P0 + (p + (SHEAR ? 9 : 0)) * 32 + (x & 31)]);
        }
    }
}

// Write a block's own nodes back (FP32 storage; the padding columns of a row's last tile stay as
// they are).
template <int V>
__device__ __noinline__ void store_block(float* state, Geometry G, Block B, const float* pop)
{
    using VA = TileVec<float, V>;
    constexpr int ROWF = row_floats<V>();
    const int w = B.w, ntiles = (w + 31) / 32, total = B.h * ntiles * VA::TV;
    for (int i = threadIdx.x; i < total; i += NT) {
        typename VA::At a = VA::at(ntiles, i);
        ++a.r;
        float* to = global_row(G, B, state, a.r) + (long long)(B.x0 / 32 + a.t) * VA::TE + a.q * 4;
        const float* q = pop + a.r * ROWF + a.p * RW + a.c + 1;
        if (a.c + 4 <= w) *reinterpret_cast<float4*>(to) = make_float4(q[0], q[1], q[2], q[3]);
        else
            for (int e = 0; a.c + e < w; ++e) to[e] = q[e];
    }
}

// A run of L.nsteps steps of this block.
template <typename S, int V, class T>
__device__ __forceinline__ void resident_body(S* __restrict__ state, const Geometry& G,
                                              const Consts<float>& K, const ResidentGrid& D,
                                              const ResidentLaunch& L)
{
    constexpr bool SRT = (V & kVarSRT) != 0;
    constexpr bool SHEAR = (V & kVarShear) != 0;
    constexpr bool LANGMUIR = (V & kVarLangmuir) != 0;
    constexpr bool NARROW = Narrow<S>::value;
    constexpr int P = std::is_same<T, F2>::value ? 2 : 1;   // nodes per lane
    constexpr int PL = SHEAR ? 9 : 18;
    constexpr int FO = SHEAR ? 0 : 9 * RW;                  // first f plane of a row
    constexpr int ROWF = row_floats<V>();
    using LN = Lane<T>;

    extern __shared__ __align__(16) float sm[];
    const int rows = L.hmax + 2;
    float* pop = sm;                              // [rows][ROWF]
    float* carry = pop + rows * ROWF;             // [2][ROWF]: pushes into a later round's row
    float* sps = carry + 2 * ROWF;                // [rows][RW] p*
    float* sph = sps + (SHEAR ? 0 : rows * RW);   // [rows][RW] phi
    float* zold = sph + rows * RW;                // 16-bit forms: [rows][2][64] Z of the nodes
    float* gz = zold + (NARROW ? rows * 128 : 0); // and [rows][4] Z of the ghost columns
    float* swirl = gz + (NARROW ? rows * 4 : 0);  // imposed flow: [rows][2] sin, cos of the rows
    const Lists tb = lists_at(swirl + (SHEAR ? rows * 2 : 0), L.hmax, L.tab);
    __shared__ int dead;
    __shared__ int nbox[16];                      // first mailbox entry of the neighbours

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Block B = block_of(G, D);
    const int h = B.h, w = B.w;
    if (tid == 0) dead = 0;
    if (tid < 15) {
        const int dx = tid % 5 - 2, dy = tid / 5 - 1;
        if (dx >= -reach<V>() && dx <= reach<V>() && (dx || dy)) {
            const Neighbour N = neighbour(G, B, D, dx, dy);
            nbox[neighbour_code<V>(dx, dy)] =
                (D.block0 + N.seg * D.nstrip + N.strip) * L.box_entries;
        }
    }
    const int words = (int)list_words(L.hmax, L.tab);
    const int* lists = L.lists + blockIdx.x * (2 + (size_t)words);
    const int nsend = lists[0], nrecv = lists[1], nring = ring_nodes(h);
    if (nsend > L.tab || nrecv > L.tab) {   // never: list_capacity holds every list
        if (tid == 0) atomicCAS(L.err, 0, 4);
        return;
    }
    for (int i = tid; i < words; i += NT) tb.node[i] = lists[2 + i];

    load_block<S, V>(state, G, B, pop, sps, sph, gz);
    if constexpr (SHEAR)
        for (int r = 1 + tid; r <= h; r += NT)
            sincospif(float(B.y0 + r - 1) * K.inv_ny - 0.5f, &swirl[2 * r], &swirl[2 * r + 1]);
    __syncthreads();
    const bool xwall = G.wall_x && (B.strip == 0 || B.strip == D.nstrip - 1);
    const int cl = lane + (P == 1 ? 32 * (warp & 1) : 0);   // the lane's (first) column
    const bool actA = cl < w, actB = P == 2 && cl + 32 < w;
    const bool full = P == 2 ? w == 64 : w >= 32 * ((warp & 1) + 1);   // warp-uniform
    const T xf = LN::of(float(B.x0 + cl), float(B.x0 + cl + 32));
    const T omega_phi(K.omega_phi);
    T sxl(0.0f), cxl(0.0f);
    if constexpr (SHEAR) {
        float sa, ca, sb, cb;
        sincospif(float(B.x0 + cl) * K.inv_nx - 0.5f, &sa, &ca);
        sincospif(float(B.x0 + cl + 32) * K.inv_nx - 0.5f, &sb, &cb);
        sxl = LN::of(sa, sb);
        cxl = LN::of(ca, cb);
    }
    const float u0s = float(L.flow_sign) * K.u0pi;
    // column whose moment stands beyond the strip's west / east end: a ghost, or at a wall the
    // end column itself
    const int cwest = G.wall_x && B.strip == 0 ? 0 : -1;
    const int ceast = G.wall_x && B.strip == D.nstrip - 1 ? w - 1 : w;
    constexpr int RPR = P == 2 ? NW : NW / 2;               // rows of a round

    auto in_domain = [&](int r) { return row_exists(G, B, r); };
    // S for row r: phi and p* of its columns c0 .. c1 and, with `ends`, of the columns beyond its
    // ends (lane 0, 1 west p*, phi; lane 2, 3 east p*, phi)
    auto row_sums = [&](int r, int c0, int c1, bool ends) {
        const float* q = pop + r * ROWF + lane + 1;
        F2 ps(0.0f), ph = Lane<F2>::ld(q + FO);
        if (!SHEAR) ps = Lane<F2>::ld(q);
#pragma unroll
        for (int a = 1; a < 9; ++a) {
            if (!SHEAR) ps += Lane<F2>::ld(q + a * RW);
            ph += Lane<F2>::ld(q + FO + a * RW);
        }
        float* dps = sps + r * RW + lane + 1;
        float* dph = sph + r * RW + lane + 1;
        const int side = (lane >> 1) & 1, lat = lane & 1;
        const bool edge = ends && lane < 4 && (!SHEAR || lat == 1);
        const int ce = side ? ceast : cwest;
        float tree = 0.0f, seq = 0.0f, zg = 0.0f;
        if (edge) {
            const float* e = pop + r * ROWF + (lat ? FO : 0) + ce + 1;
            float v[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) v[a] = e[a * RW];
            if constexpr (NARROW) {
                const float inv = lat ? K.st_inv[1] : K.st_inv[0];
                // at a wall the end column itself stands there, its Z still in the sums' array
                const bool ghost = ce < 0 || ce == w;
                zg = ghost ? gz[r * 4 + 2 * side + lat] : (lat ? sph : sps)[r * RW + ce + 1];
                seq = v[0];
#pragma unroll
                for (int a = 1; a < 9; ++a) seq = __fadd_rn(seq, v[a]);
                seq = __fmaf_rn(seq, inv, zg);
#pragma unroll
                for (int a = 0; a < 9; ++a) v[a] = __fmul_rn(v[a], inv);
            }
            tree = tree_sum(v, zg);
        }
        const bool doA = lane >= c0 && lane <= c1, doB = lane + 32 >= c0 && lane + 32 <= c1;
        if constexpr (NARROW) {
            const F2 zps = Lane<F2>::ld(dps), zph = Lane<F2>::ld(dph);
            ps = fmad(ps, F2(K.st_inv[0]), zps);
            ph = fmad(ph, F2(K.st_inv[1]), zph);
            float* zo = zold + r * 128 + lane;
            if (doA) { zo[0] = zps.v.x; zo[64] = zph.v.x; }
            if (doB) { zo[32] = zps.v.y; zo[96] = zph.v.y; }
            __syncwarp();   // the end columns' Z are read before they are replaced
            if (edge) gz[r * 4 + 2 * side + lat] = seq;
        }
        if (doA) {
            if (!SHEAR) dps[0] = ps.v.x;
            dph[0] = ph.v.x;
        }
        if (doB) {
            if (!SHEAR) dps[32] = ps.v.y;
            dph[32] = ph.v.y;
        }
        if (edge) (lat ? sph : sps)[r * RW + (side ? w + 1 : 0)] = tree;
    };
    // 16-bit forms: S of ring node (r, c), lattice lat (the sum replaces the Z it starts from)
    auto ring_sum = [&](int r, int c, int lat) {
        const float* o = pop + r * ROWF + (lat ? FO : 0) + c + 1;
        float* d = (lat ? sph : sps) + r * RW + c + 1;
        const bool ghost = c < 0 || c == w;   // a column beyond the strip: tree order
        const float inv = lat ? K.st_inv[1] : K.st_inv[0];
        float* zp = ghost ? gz + r * 4 + (c < 0 ? 0 : 2) + lat : d;
        const float z = *zp;
        float q[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) q[a] = o[a * RW];
        float sum = q[0];
#pragma unroll
        for (int a = 1; a < 9; ++a) sum = __fadd_rn(sum, q[a]);
        sum = __fmaf_rn(sum, inv, z);
        if (ghost) *zp = sum;
        else zold[r * 128 + 64 * lat + c] = z;
#pragma unroll
        for (int a = 0; a < 9; ++a) q[a] = __fmul_rn(q[a], inv);
        if (ghost) {
            d[0] = tree_sum(q, z);
            return;
        }
        d[0] = sum;
        if (c == cwest) d[-1] = tree_sum(q, z);   // at a wall the end column itself
        if (c == ceast) d[1] = tree_sum(q, z);
    };

    for (int r = warp; r < h + 2; r += NW)
        if (in_domain(r)) row_sums(r, 0, w - 1, true);
    __syncthreads();

    for (int s = 0; s < L.nsteps; ++s) {
        // ---- C: collide and push, RPR rows a round -------------------------------------------
        for (int q = 0, rnd = 0; q < h; q += RPR, ++rnd) {
            const int r = 1 + q + (P == 2 ? warp : warp >> 1);
            const bool live = r <= h;                       // warp-uniform
            const int y = B.y0 + r - 1;
            T g[9], f[9];
            Win<T> ph, ps;
            if (live) {
                // mirror ghosts of the stencils at walls
                const int rS = G.wall_y && y == 0 ? r : r - 1;
                const int rN = G.wall_y && y == G.ny - 1 ? r : r + 1;
                auto window = [&](const float* m, Win<T>& v) {
                    const float* ms = m + rS * RW + cl;
                    const float* mc = m + r * RW + cl;
                    const float* mn = m + rN * RW + cl;
                    v.sw = LN::ld(ms); v.s = LN::ld(ms + 1); v.se = LN::ld(ms + 2);
                    v.w = LN::ld(mc);  v.c = LN::ld(mc + 1); v.e = LN::ld(mc + 2);
                    v.nw = LN::ld(mn); v.n = LN::ld(mn + 1); v.ne = LN::ld(mn + 2);
                };
                window(sph, ph);
                if constexpr (!SHEAR) window(sps, ps);
                const float* o = pop + r * ROWF + cl + 1;
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    if (!SHEAR) g[a] = LN::ld(o + a * RW);
                    f[a] = LN::ld(o + FO + a * RW);
                }
                if constexpr (NARROW) {   // q_a = w_a Z + d_a / s
                    const T zg = LN::ld(zold + r * 128 + cl);
                    const T zf = LN::ld(zold + r * 128 + 64 + cl);
                    const T ig(K.st_inv[0]), ifl(K.st_inv[1]);
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        const T wa(float(d2q9_w(a)));
                        g[a] = fmad(g[a], ig, wa * zg);
                        f[a] = fmad(f[a], ifl, wa * zf);
                    }
                }
                Macro<T> m;
                if constexpr (SHEAR) {
                    m.ux = T(-u0s * swirl[2 * r]) * cxl;
                    m.uy = T(u0s * swirl[2 * r + 1]) * sxl;
                    interface_flux<T>(ph, K, m.jx, m.jy);
                } else {
                    const T jgx = ((g[1] - g[3]) + (g[5] - g[6])) - (g[7] - g[8]);
                    const T jgy = ((g[2] - g[4]) + (g[5] + g[6])) - (g[7] + g[8]);
                    node_macro<T, LANGMUIR>(ph, ps, jgx, jgy, xf, T(float(y)), K, m);
                    if constexpr (SRT) collide_fluid_srt<T>(g, ps.c, m);
                    else collide_fluid<T>(g, ps.c, m);
                }
                if constexpr (SRT) collide_ace_srt<T>(f, ph.c, m, omega_phi);
                else collide_ace<T>(f, ph.c, m, omega_phi);
            }
            __syncthreads();   // every population of the round's rows is in registers
            if (rnd > 0) {     // the previous round's pushes into this round's first row
                constexpr int PLN[3] = {2, 5, 6};
                const float* from = carry + ((rnd - 1) & 1) * ROWF;
                float* to = pop + (1 + q) * ROWF;
                for (int k = tid; k < (PL / 3) * RW; k += NT) {
                    const int j = k / RW;
                    const int p = (j >= 3 ? 9 : 0) + (j % 3 == 0 ? PLN[0] : j % 3 == 1 ? PLN[1] : PLN[2]);
                    if (SHEAR && !carry_fills(p, k % RW - 1, w,
                                              G.wall_x && B.strip == 0 && !(G.slip & 1),
                                              G.wall_x && B.strip == D.nstrip - 1 && !(G.slip & 2)))
                        continue;
                    to[p * RW + k % RW] = from[p * RW + k % RW];
                }
                if (!SHEAR && xwall && carry_meets_pushes(G.slip)) __syncthreads();
            }
            if (!live) continue;
            float* rC = pop + r * ROWF + cl + 1;
            float* rS = rC - ROWF;
            float* rN = rC + ROWF;
            if (r == q + RPR && r < h) rN = carry + (rnd & 1) * ROWF + cl + 1;
            constexpr int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
            constexpr int EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
            const bool bys = y == 0 && G.wall_y, byn = y == G.ny - 1 && G.wall_y;
            if (!(bys || byn) && !xwall) {
                auto put = [&](int a, int fo, T v) {
                    float* o = (EY[a] < 0 ? rS : (EY[a] > 0 ? rN : rC)) + fo + a * RW + EX[a];
                    if (full || actA) o[0] = LN::half(v, false);
                    if (P == 2 && (full || actB)) o[32] = LN::half(v, true);
                };
                if constexpr (NARROW) {
                    T eg(0.0f), ef(0.0f), st;
#pragma unroll
                    for (int a = 1; a < 9; ++a) {
                        const float wa = float(d2q9_w(a));
                        eg += encode_lane<S, false>(g[a], win_at(ps, EX[a], EY[a]), wa,
                                                    K.st_scale[0], T(0.0f), st);
                        put(a, 0, st);
                        ef += encode_lane<S, false>(f[a], win_at(ph, EX[a], EY[a]), wa,
                                                    K.st_scale[1], T(0.0f), st);
                        put(a, FO, st);
                    }
                    const float w0 = float(d2q9_w(0));
                    encode_lane<S, true>(g[0], ps.c, w0, K.st_scale[0], eg, st);
                    put(0, 0, st);
                    encode_lane<S, true>(f[0], ph.c, w0, K.st_scale[1], ef, st);
                    put(0, FO, st);
                } else {
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        if (!SHEAR) put(a, 0, g[a]);
                        put(a, FO, f[a]);
                    }
                }
                continue;
            }
            // rows and strips at a wall, node by node: a population crossing a no-slip wall
            // returns reversed (half-way bounce-back), one crossing only free-slip walls has its
            // normal components reversed and stays on this side of them (specular reflection)
            constexpr int OPP[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
            constexpr int MX[9] = {0, 3, 2, 1, 4, 6, 5, 8, 7};
            constexpr int MY[9] = {0, 1, 4, 3, 2, 8, 7, 6, 5};
#pragma unroll
            for (int b = 0; b < P; ++b) {
                const int c = cl + 32 * b;
                if (c >= w) continue;
                const int x = B.x0 + c;
                const bool bxw = x == 0 && G.wall_x, bxe = x == G.nx - 1 && G.wall_x;
                float eg = 0.0f, ef = 0.0f, e;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const int a = k == 8 ? 0 : k + 1;   // the rest population last
                    const int ex = EX[a], ey = EY[a];
                    const bool cx = (ex < 0 && bxw) || (ex > 0 && bxe);
                    const bool cy = (ey < 0 && bys) || (ey > 0 && byn);
                    const bool sx = ((G.slip >> (ex < 0 ? 0 : 1)) & 1) != 0;
                    const bool sy = ((G.slip >> (ey < 0 ? 2 : 3)) & 1) != 0;
                    const bool bounce = (cx && !sx) || (cy && !sy) || (cx && cy);
                    const int plane = bounce ? OPP[a] : (cx ? MX[a] : (cy ? MY[a] : a));
                    float* row = bounce || cy ? rC : (ey > 0 ? rN : (ey < 0 ? rS : rC));
                    float* o = row + 32 * b + plane * RW + (bounce || cx ? 0 : ex);
                    float vg = SHEAR ? 0.0f : LN::half(g[a], b), vf = LN::half(f[a], b);
                    if constexpr (NARROW) {
                        auto landing = [&](const Win<T>& z) {
                            return bounce ? LN::half(z.c, b)
                                   : cx   ? LN::half(win_at(z, 0, ey), b)
                                   : cy   ? LN::half(win_at(z, ex, 0), b)
                                          : LN::half(win_at(z, ex, ey), b);
                        };
                        const float zg = landing(ps), zf = landing(ph), wa = float(d2q9_w(a));
                        if (a != 0) {
                            vg = narrow_to_f(encode_err<S, false>(vg, zg, wa, K.st_scale[0],
                                                                  0.0f, e));
                            eg += e;
                            vf = narrow_to_f(encode_err<S, false>(vf, zf, wa, K.st_scale[1],
                                                                  0.0f, e));
                            ef += e;
                        } else {
                            vg = narrow_to_f(encode_err<S, true>(vg, zg, wa, K.st_scale[0], eg, e));
                            vf = narrow_to_f(encode_err<S, true>(vf, zf, wa, K.st_scale[1], ef, e));
                        }
                    }
                    if (!SHEAR) o[0] = vg;
                    o[FO] = vf;
                }
            }
        }
        __syncthreads();

        // ---- X: exchange the two outermost rings ----------------------------------------------
        const bool last = s + 1 == L.nsteps;
        const unsigned tag = L.tag0 + 1u + (unsigned)s;
        ulonglong2* box = L.box + (size_t)(tag & 1u) * gridDim.x * L.box_entries;
        for (int i0 = tid; i0 < nsend; i0 += 4 * NT) {   // four entries read, then four sent
            int to[4];
            float a[4], b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = min(i0 + k * NT, nsend - 1);
                const float* o = pop + tb.soff[i];
                const unsigned d = tb.sdst[i];
                to[k] = nbox[d >> box_bits<V>()] + (int)(d & ((1u << box_bits<V>()) - 1));
                a[k] = o[0];
                b[k] = o[FO];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i0 + k * NT < nsend) st_box(box + to[k], tag, a[k], b[k]);
        }
        // while the messages travel: the sums of the nodes that need none of them
        if (!last)
            for (int r = 2 + warp; r < h; r += NW) row_sums(r, 1, w - 2, false);
        const ulonglong2* own = box + (size_t)blockIdx.x * L.box_entries;
        for (int i0 = tid; i0 < nrecv; i0 += 4 * NT) {
            const ulonglong2* from[4];
            ulonglong2 v[4];
            unsigned m = 0;      // entries still due
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                from[k] = own + tb.rbox[min(i0 + k * NT, nrecv - 1)];
                m |= i0 + k * NT < nrecv ? 1u << k : 0u;
            }
            unsigned long long t0 = 0;
            for (unsigned it = 1;; ++it) {
#pragma unroll
                for (int k = 0; k < 4; ++k)   // all in flight together
                    if ((m >> k) & 1) v[k] = ld_box(from[k]);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!((m >> k) & 1) || (unsigned)(v[k].x >> 32) != tag ||
                        (unsigned)(v[k].y >> 32) != tag)
                        continue;
                    m &= ~(1u << k);
                    float* o = pop + tb.roff[i0 + k * NT];
                    if (!SHEAR) o[0] = __uint_as_float((unsigned)v[k].x);
                    o[FO] = __uint_as_float((unsigned)v[k].y);
                }
                if (m == 0) break;
                // another block failed, this one did, or the wait runs out (the timer is read
                // every 256 polls; the poll count bounds it should the timer stand still)
                if ((it & 255u) == 0) {
                    const unsigned long long t = global_ns();
                    if (t0 == 0) t0 = t;
                    if (*(volatile int*)L.err != 0 || *(volatile int*)&dead || it > (1u << 27) ||
                        t - t0 > kBoxWaitNs) {
                        atomicCAS(L.err, 0, 4);
                        dead = 1;
                        break;
                    }
                }
            }
        }
        __syncthreads();
        if (dead) return;   // block-uniform; the state of this run is invalid
        if (last) break;
        // ---- S of the two outermost rings: the two outer rows at each end by a warp each, beside
        // them the columns at and beyond the ends of all rows by a thread each; in the 16-bit forms
        // a thread a node, so that nobody reads a Z that another replaces
        if constexpr (!NARROW) {
            if (warp < 4) {
                const int r = warp < 2 ? warp : h + warp - 2;
                if (in_domain(r)) row_sums(r, 0, w - 1, false);
            } else {
                // ends: 4 tree sums a row (h + 2 rows), 4 end-column sums a row (h - 2 rows)
                for (int i = tid - 128; i < 4 * (h + 2) + 4 * (h - 2); i += NT - 128) {
                    const bool tr = i < 4 * (h + 2);
                    const int k = tr ? i : i - 4 * (h + 2);
                    const int r = tr ? k >> 2 : 2 + (k >> 2), side = (k >> 1) & 1, lat = k & 1;
                    if (!in_domain(r) || (SHEAR && lat == 0)) continue;
                    const int c = tr ? (side ? ceast : cwest) : (side ? w - 1 : 0);
                    const float* o = pop + r * ROWF + (lat ? FO : 0) + c + 1;
                    float q[9];
#pragma unroll
                    for (int a = 0; a < 9; ++a) q[a] = o[a * RW];
                    float sum = q[0];
#pragma unroll
                    for (int a = 1; a < 9; ++a) sum = __fadd_rn(sum, q[a]);
                    const float t = tree_sum(q, 0.0f);
                    (lat ? sph : sps)[r * RW + (tr ? (side ? w + 1 : 0) : c + 1)] = tr ? t : sum;
                }
            }
        } else {
            for (int j = tid; j < 2 * nring; j += NT) {
                const int lat = j >= nring;
                const unsigned n = tb.node[lat ? j - nring : j];
                if (n != kNoNode) ring_sum(n >> 16, (int)(n & 0xffff) - 1, lat);
            }
        }
        __syncthreads();
    }

    // write the block back; every neighbour has read its ghost ring (it has sent a message since)
    if constexpr (NARROW) {   // (in 16-byte accesses the whole time loop came out 14 % slower)
        constexpr int TE = Tile<S>::ELEMS;
        for (int k = warp; k < h * PL; k += NW) {
            const int r = 1 + k / PL, p = k % PL;
            for (int c = lane; c < w; c += 32) {
                const int x = B.x0 + c;
                S* tile = global_row(G, B, state, r) + (x >> 5) * TE;
                tile[Tile<S>::P0 + p * 32 + (x & 31)] =
                    f_to_narrow<S>(pop[r * ROWF + p * RW + c + 1]);
                if (p < 2)   // the zeroth moments of the level before
                    reinterpret_cast<float*>(tile)[32 * p + (x & 31)] =
                        (p ? sph : sps)[r * RW + c + 1];
            }
        }
    } else {
        store_block<V>(state, G, B, pop);
    }
}

template <typename S, int V, class T>
__global__ void __launch_bounds__(NT, 1)
resident_kernel(S* __restrict__ state, Geometry G, Consts<float> K, ResidentGrid D,
                ResidentLaunch L)
{
    resident_body<S, V, T>(state, G, K, D, L);
}

// Many grids in one launch: block b runs its part of case case_of[b].
template <typename S, int V>
__global__ void __launch_bounds__(NT, 1)
resident_batch_kernel(S* __restrict__ base, const ResidentCase* __restrict__ cases,
                      const int* __restrict__ case_of, int parity, ResidentLaunch L)
{
    __shared__ Consts<float> K;
    const ResidentCase& c = cases[case_of[blockIdx.x]];
    for (int i = threadIdx.x; i < (int)(sizeof(K) / 4); i += NT)
        reinterpret_cast<int*>(&K)[i] = reinterpret_cast<const int*>(&c.K)[i];
    __syncthreads();
    const Geometry G = c.G;
    resident_body<S, V, F2>(base + c.off[parity], G, K, c.D, L);
}

template <typename S, int V>
size_t resident_smem(int hmax, int tab)
{
    const size_t rows = (size_t)hmax + 2;
    size_t f = (rows + 2) * row_floats<V>() + ((V & kVarShear) ? 1 : 2) * rows * RW;
    if (Narrow<S>::value) f += rows * (128 + 4);
    if (V & kVarShear) f += rows * 2;
    return (f + list_words(hmax, tab)) * 4;
}

template <typename S, int V>
const void* resident_fn(int hmax)
{
    // half a row per warp where every row of the block then has its own two warps; in the forms
    // where the compiler fuses no packed product with a sum (elsewhere F1's bits may differ)
    if constexpr (V == 0 || V == kVarLangmuir)
        if (2 * hmax <= NW) return (const void*)resident_kernel<S, V, F1>;
    return (const void*)resident_kernel<S, V, F2>;
}

// Entries of a block's send or receive list: nine populations of each node of the two outermost
// rings with a source (or a taker) on the other side, three more a side row towards the block
// beyond a single-column strip, and the corners.
template <int V>
constexpr int list_capacity(int hmax)
{
    return (9 * (2 * (64 + 2) + 2 * (hmax + 2)) + (reach<V>() == 2 ? 6 * (hmax + 2) : 0) + 128 +
            3) & ~3;
}
constexpr int mailbox_entries(int hmax) { return 36 * RW + 36 * (hmax > 2 ? hmax - 2 : 0); }

// Dynamic shared memory a block may have (the current device), and whether `fn` may be launched
// with it.
int most_smem()
{
    int dev = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return most - 1024;   // the static part and the system's own
}
bool can_launch(const void* fn, size_t smem, int most)
{
    int nb = 0;
    const bool ok =
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, NT, smem) == cudaSuccess && nb >= 1;
    cudaGetLastError();
    return ok;
}

// Blocks of at most `hmax` rows fit in shared memory and in the lists' 16-bit offsets.
template <typename S, int V>
bool rows_fit(int hmax, int most)
{
    return resident_smem<S, V>(hmax, list_capacity<V>(hmax)) <= (size_t)most &&
           (hmax + 2) * row_floats<V>() <= 65535 &&
           mailbox_entries(hmax) <= 1 << box_bits<V>();
}

// A grid's split needs two rows in every block, and strips whose reach the neighbour list covers.
template <int V>
bool grid_splits(const Geometry& G, int nstrip)
{
    const int last = G.nx - (nstrip - 1) * 64;
    return G.ny >= 2 && (last >= 2 || (last == 1 && nstrip >= 2 && reach<V>() == 2));
}

template <typename S, int V>
void fill_sizes(int nblocks, int hmax, ResidentSizes* z)
{
    z->nblocks = nblocks;
    z->hmax = hmax;
    z->tab = list_capacity<V>(hmax);
    z->box_entries = mailbox_entries(hmax);
    z->smem = resident_smem<S, V>(hmax, z->tab);
    z->box_bytes = (size_t)2 * nblocks * z->box_entries * sizeof(ulonglong2);
    z->list_bytes = (size_t)nblocks * (2 + list_words(hmax, z->tab)) * 4;
}

ResidentLaunch launch_args(const ResidentSizes& z, void* box, void* lists, int nsteps, int flow_sign,
                           unsigned tag0, int* err)
{
    ResidentLaunch L = {};
    L.hmax = z.hmax;
    L.tab = z.tab;
    L.box_entries = z.box_entries;
    L.nsteps = nsteps;
    L.flow_sign = flow_sign;
    L.tag0 = tag0;
    L.box = static_cast<ulonglong2*>(box);
    L.lists = static_cast<int*>(lists);
    L.err = err;
    return L;
}

}  // namespace

// Most rows of a block; 0 if not even two fit.
template <typename S, int V>
int most_rows(int most)
{
    int h = 0;
    while (rows_fit<S, V>(h + 1, most)) ++h;
    return h < 2 ? 0 : h;
}

template <typename S, int V>
bool resident_plan(const Geometry& G, int nsm, bool shared, ResidentPlan* out)
{
    const int nstrip = (G.nx + 63) / 64, most = most_smem(), fit = most_rows<S, V>(most);
    if (!grid_splits<V>(G, nstrip) || nstrip > nsm) return false;
    const GridSize size = {G.nx, G.ny};
    constexpr Form form = (V & kVarShear) ? Form::Flow : Narrow<S>::value ? Form::Narrow : Form::Fp32;
    const int nseg = shared ? shared_segments(size, nsm, fit, form) : most_segments(size, nsm);
    if (nseg < 1) return false;
    const int hmax = (G.ny + nseg - 1) / nseg;
    if (hmax > fit) return false;
    out->D = {nstrip, nseg, 0};
    fill_sizes<S, V>(nstrip * nseg, hmax, &out->Z);
    return can_launch(resident_fn<S, V>(hmax), out->Z.smem, most);
}

template <typename S, int V>
cudaError_t prepare_resident(const Geometry& G, const ResidentPlan& P, void* box, void* lists,
                             cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(box, 0, P.Z.box_bytes, st);
    if (e != cudaSuccess) return e;
    resident_lists_kernel<V><<<P.Z.nblocks, NT, 0, st>>>(
        G, P.D, launch_args(P.Z, box, lists, 0, 1, 0, nullptr));
    return cudaGetLastError();
}

cudaError_t mute_resident(const ResidentPlan& P, void* lists, cudaStream_t st)
{
    const size_t pitch = (2 + list_words(P.Z.hmax, P.Z.tab)) * sizeof(int);   // a block's; its sends first
    return cudaMemset2DAsync(lists, pitch, 0, sizeof(int), P.Z.nblocks, st);
}

template <typename S, int V>
cudaError_t launch_resident(void* state, const Geometry& G, const Consts<float>& K,
                            const ResidentPlan& P, int nsteps, int flow_sign, unsigned tag0,
                            void* box, void* lists, int* err, cudaStream_t st)
{
    ResidentLaunch L = launch_args(P.Z, box, lists, nsteps, flow_sign, tag0, err);
    S* s = static_cast<S*>(state);
    Geometry g = G;
    Consts<float> k = K;
    ResidentGrid d = P.D;
    void* args[] = {(void*)&s, (void*)&g, (void*)&k, (void*)&d, (void*)&L};
    return cudaLaunchCooperativeKernel(resident_fn<S, V>(P.Z.hmax), dim3(P.Z.nblocks), dim3(NT),
                                       args, P.Z.smem, st);
}

template <typename S, int V>
bool resident_batch_plan(const Geometry* G, int ncases, int nsm, std::vector<ResidentWave>* waves,
                         double* step_us)
{
    const int most = most_smem(), fit = most_rows<S, V>(most);
    if (fit < 2) return false;
    for (int c = 0; c < ncases; ++c)
        if (!grid_splits<V>(G[c], (G[c].nx + 63) / 64)) return false;
    std::vector<GridSize> grids;
    for (int c = 0; c < ncases; ++c) grids.push_back({G[c].nx, G[c].ny});
    const std::vector<Wave> plan = batch_waves(grids, nsm, fit);
    if (plan.empty()) return false;
    *step_us = waves_us(plan, Narrow<S>::value);
    for (const Wave& b : plan) {
        ResidentWave W;
        int nblocks = 0;
        for (const WavePart& p : b) {
            W.cases.push_back(p.c);
            W.D.push_back({p.nstrip, p.nseg, nblocks});
            nblocks += p.nstrip * p.nseg;
        }
        fill_sizes<S, V>(nblocks, tallest(b), &W.Z);
        if (!can_launch((const void*)resident_batch_kernel<S, V>, W.Z.smem, most)) return false;
        waves->push_back(W);
    }
    return true;
}

template <typename S, int V>
cudaError_t prepare_resident_batch(const ResidentSizes& Z, const ResidentCase* cases,
                                   const int* case_of, void* lists, cudaStream_t st)
{
    resident_batch_lists_kernel<V><<<Z.nblocks, NT, 0, st>>>(
        cases, case_of, launch_args(Z, nullptr, lists, 0, 1, 0, nullptr));
    return cudaGetLastError();
}

template <typename S, int V>
cudaError_t launch_resident_batch(void* base, const ResidentSizes& Z, const ResidentCase* cases,
                                  const int* case_of, int parity, int nsteps, unsigned tag0,
                                  void* box, void* lists, int* err, cudaStream_t st)
{
    ResidentLaunch L = launch_args(Z, box, lists, nsteps, 1, tag0, err);
    S* s = static_cast<S*>(base);
    void* args[] = {(void*)&s, (void*)&cases, (void*)&case_of, (void*)&parity, (void*)&L};
    return cudaLaunchCooperativeKernel((const void*)resident_batch_kernel<S, V>, dim3(Z.nblocks),
                                       dim3(NT), args, Z.smem, st);
}

#define CMLBM_INSTANTIATE_RESIDENT(S, V)                                                          \
    template bool resident_plan<S, V>(const Geometry&, int, bool, ResidentPlan*);               \
    template cudaError_t prepare_resident<S, V>(const Geometry&, const ResidentPlan&, void*,    \
                                                void*, cudaStream_t);                           \
    template cudaError_t launch_resident<S, V>(void*, const Geometry&, const Consts<float>&,    \
                                               const ResidentPlan&, int, int, unsigned, void*,  \
                                               void*, int*, cudaStream_t);
#define CMLBM_INSTANTIATE_RESIDENT_BATCH(S, V)                                                    \
    template bool resident_batch_plan<S, V>(const Geometry*, int, int,                          \
                                            std::vector<ResidentWave>*, double*);               \
    template cudaError_t prepare_resident_batch<S, V>(const ResidentSizes&,                     \
                                                      const ResidentCase*, const int*, void*,   \
                                                      cudaStream_t);                            \
    template cudaError_t launch_resident_batch<S, V>(void*, const ResidentSizes&,               \
                                                     const ResidentCase*, const int*, int, int, \
                                                     unsigned, void*, void*, int*,              \
                                                     cudaStream_t);
CMLBM_INSTANTIATE_RESIDENT(float, 0)
CMLBM_INSTANTIATE_RESIDENT(float, 1)
CMLBM_INSTANTIATE_RESIDENT(float, 2)
CMLBM_INSTANTIATE_RESIDENT(float, 3)
CMLBM_INSTANTIATE_RESIDENT(float, 4)
CMLBM_INSTANTIATE_RESIDENT(float, 5)
CMLBM_INSTANTIATE_RESIDENT(__half, 0)
CMLBM_INSTANTIATE_RESIDENT(__nv_bfloat16, 0)
CMLBM_INSTANTIATE_RESIDENT_BATCH(float, 0)
CMLBM_INSTANTIATE_RESIDENT_BATCH(float, 1)
CMLBM_INSTANTIATE_RESIDENT_BATCH(float, 4)
CMLBM_INSTANTIATE_RESIDENT_BATCH(float, 5)
CMLBM_INSTANTIATE_RESIDENT_BATCH(__half, 0)
CMLBM_INSTANTIATE_RESIDENT_BATCH(__nv_bfloat16, 0)
#undef CMLBM_INSTANTIATE_RESIDENT
#undef CMLBM_INSTANTIATE_RESIDENT_BATCH

}  // namespace cmlbm
