// Algorithm 1's passes in the circle colouring's order, spread over the GPU as a systolic
// array (schedule 1).
//
// The order.  With P = n rounded up to even, minus 1 (odd), class c pairs a and b when
// a + b = c (mod P); for even n the last node, "the odd one", meets a in class 2a mod P.
// Write the edges below P as the upper triangle of a matrix, row a < column b.  Cell (a, b)
// then depends only on (a, b - 1) (row a's previous partner) and (a - 1, b) (column b's
// previous partner): a class is an antidiagonal, and the pass is a wavefront.  A node is a
// column first (rows 0 .. y - 1 from the top), turns into row y at the diagonal, where it meets
// the odd one, runs to the right edge, and enters the next lap as a column.  Classes above
// and below a + b = P belong to the same wave (mod P), so the passes of a call follow one
// another without a barrier: a pass boundary is only a cut along the antidiagonal a + b = P.
//
// The array.  A tile is 32 consecutive rows, one per lane of a warp, with the row's load in a
// register.  Columns stream through the lanes: at step s lane i holds column s - i (counted
// from the tile's first row) and updates its row against it, then hands the column to lane
// i + 1 by a shuffle.  Lane 0 takes the column the previous tile's last lane gave out.  So every
// update of a pass is in program order inside a warp, or passed on as a value: no barrier, no
// load gathers, no bank conflicts, and a class costs one step of the array however many
// edges it has.  The updates are the staged sweep's, operation for operation, so splits and
// loads come out the same bit for bit.
//
// Tiles and the odd one.  Low tile k holds rows 32k .. below h = (P + 1)/2, high tile k rows
// h + 32k ..; both cross their diagonals in the same 64 classes, the low rows in the even ones and
// the high rows in the odd ones.  A block runs a few such pairs, a warp per tile.  For even n the
// low warp keeps the odd one's load in registers and moves it past the high rows too (they send
// their load and limits ahead), so it never travels back; rows without an edge to it skip that.
//
// Streams between tiles.  An entry is 16 bytes, (hi, tag), (lo, tag): the tag (lap and column)
// tells the reader that the value beside it is there, so no fence is needed.  Inside a
// block the streams are rings of 128 entries in shared memory (the reader publishes how far
// it got); between blocks they are arrays in global memory, and an import warp polls them and
// refills the ring.  Rows that leave at the right edge enter the top tile through such an
// array.  One cooperative launch runs all passes; every wait is bounded, and on expiry the
// warp sets an error bit and leaves, and the others follow.
//
// The splits sit in a dense array, 32 lanes per step (128 bytes), staged through shared memory by
// cp.async a chunk of 32 steps ahead and written back as they are updated; cells without an edge
// hold -1 (unit weights) or weight 0 and change nothing.  A graph whose cells all fit one block's
// shared memory keeps them there for the launch.
//
// What bounds it: a chain of P steps per pass, not bandwidth (DRAM 0.3 TB/s on the scale-22 R-MAT
// core).  A step's own chain is a shuffle and a transfer; on the critical path, about 230 cycles a
// step, lie the steps at the diagonal and the right edge, a lag of about three steps per tile, since
// inputs are checked four at a time, and the way between blocks.
// Measured (GB300, per pass, against the one-CTA sweep of one barrier per class): scale-22 R-MAT core, n
// 9,109, 6.49 M edges 1,027 us (2,705); n 9,110 at density 0.156 1,898 (2,890); n 4,047 at 0.126 437
// (701); n 6,193 weighted at 0.08 718 (1,189); n 307 27 (111); n 71 7.4 (22).
#include "ctx.cuh"
#include "prims.cuh"
#include "async.cuh"

#include <vector>

using namespace lowd;

namespace {

constexpr int kT = 256;
inline unsigned grid_for(int64_t n) { return lowd_grid_for(n, kT); }

constexpr int kPairs = 4;             // most pairs of tiles per block of several (two warps per scheduler)
constexpr int kPairsOdd = 2;          // odd n, while the SMs hold a block each
constexpr int kMaxW = 5;              // the most, in a block alone
constexpr int kPad = 96;              // steps of a lap beyond P: drained lanes, read-ahead, tags
constexpr size_t kSmemMost = 226 * 1024;   // dynamic shared memory of a block (227 KB less the static part)
constexpr uint32_t kOddBytes = 16u + 4u * 16u + 4u * 32u;   // of a pair: way in, low to high, high to low
constexpr int kRing = 128;            // entries of a stream ring (a reader tells how far it is every 32)
constexpr int kChunk = 32;            // steps per staged chunk
constexpr int kSlots = 2;             // staged chunks
constexpr int kAhead = kSlots - 1;    // chunks in flight
constexpr int kDiag = 64 / kChunk;    // chunks of a tile's diagonal
constexpr uint32_t kChunkBytes = kChunk * 128u;
constexpr uint32_t kCellBytes = kSlots * kChunkBytes;   // staged cells of one array of a tile
constexpr uint32_t kSpinSmem = 1u << 21;    // bounded waits: polls of shared memory
constexpr uint32_t kSpinGlobal = 1u << 20;  // polls of global memory

// Tile geometry.  Low tile k holds rows 32k .. of [0, h), high tile k rows h + 32k .. of
// [h, P).  A tile's cells are rounded up so that their offsets have a closed form.
struct Geo {
    int32_t n, P, h, KL, KU;
    int32_t A, B;        // steps of low tile 0 / high tile 0, less 32, multiples of 32
    __host__ __device__ int64_t low(int32_t k) const { return (int64_t)k * (A + 32) - 16ll * k * (k - 1); }
    __host__ __device__ int64_t high(int32_t k) const {
        return low(KL) + (int64_t)k * (B + 32) - 16ll * k * (k - 1);
    }
    __host__ __device__ int64_t steps() const { return high(KU); }
    // cell of the edge a < b (b == P: the odd one)
    __device__ __forceinline__ int64_t cell(int32_t a, int32_t b) const {
        const bool up = a >= h;
        const int32_t r = up ? a - h : a;
        const int32_t k = r >> 5, i = r & 31;
        const int32_t s = b == P ? 2 * i : b - a + 2 * i;
        return (((up ? high(k) : low(k)) + s) << 5) + i;
    }
};

Geo make_geo(int32_t n) {
    Geo g;
    g.n = n;
    g.P = n + (n & 1) - 1;
    g.h = (g.P + 1) / 2;
    g.KL = (g.h + 31) / 32;
    g.KU = (g.h - 1 + 31) / 32;
    g.A = (g.P + 64 + 31) / 32 * 32;   // a lap's last chunk may run up to 31 steps past its end
    g.B = (g.P - g.h + 64 + 31) / 32 * 32;
    return g;
}

struct SysArgs {
    Geo g;
    int32_t W;           // pairs per block
    int32_t T;           // passes
    int32_t odd;         // 1: n is even, node P is the odd one
    uint32_t tag0;       // tag base of this launch
    float* cs;
    const float* cw;
    float* l;
    float* l_lo;
    ulonglong2* in_low;       // [grid][P + kPad] streams into each block's first low tile (block 0: the wrap)
    ulonglong2* in_high;      // [grid][P + kPad]
    ulonglong2* in_odd;       // [grid] the odd one's load
    int32_t* err;        // kWaveExpired: a wait expired (every warp then leaves)
    uint32_t spin_shift; // the waits' limits are divided by 2 to this power
};

// A stream entry: (hi, tag), (lo, tag).  Each 8-byte half is written and read as one access and
// carries the tag, so a reader that sees the tag in both (single FP32 loads: in the first) has
// the whole value; the two halves need not arrive together.
struct Entry {
    unsigned long long a, b;
    __device__ __forceinline__ float2 value() const {
        return make_float2(__uint_as_float((uint32_t)a), __uint_as_float((uint32_t)b));
    }
    template <bool PAIR>
    __device__ __forceinline__ bool is(uint32_t tag) const {
        return PAIR ? ((((uint32_t)(a >> 32) ^ tag) | ((uint32_t)(b >> 32) ^ tag)) == 0u) : (uint32_t)(a >> 32) == tag;
    }
};
__device__ __forceinline__ unsigned long long half_of(float x, uint32_t tag) {
    return (unsigned long long)__float_as_uint(x) | ((unsigned long long)tag << 32);
}
template <bool PAIR>
__device__ __forceinline__ Entry ldg_entry(const ulonglong2* p) {
    Entry e;
    e.b = 0ull;
    if (PAIR) asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(e.a), "=l"(e.b) : "l"(p) : "memory");
    else asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(e.a) : "l"(p) : "memory");
    return e;
}
template <bool PAIR>
__device__ __forceinline__ void stg_entry(ulonglong2* p, float2 v, uint32_t tag) {
    if (PAIR)
        asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};"
                     ::"l"(p), "l"(half_of(v.x, tag)), "l"(half_of(v.y, tag)) : "memory");
    else asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(half_of(v.x, tag)) : "memory");
}
template <bool PAIR>
__device__ __forceinline__ Entry lds_entry(uint32_t p) {
    Entry e;
    e.b = 0ull;
    if (PAIR) asm volatile("ld.relaxed.cta.shared::cta.v2.b64 {%0, %1}, [%2];" : "=l"(e.a), "=l"(e.b) : "r"(p) : "memory");
    else asm volatile("ld.relaxed.cta.shared::cta.b64 %0, [%1];" : "=l"(e.a) : "r"(p) : "memory");
    return e;
}
template <bool PAIR>
__device__ __forceinline__ void sts_entry(uint32_t p, float2 v, uint32_t tag) {
    if (PAIR)
        asm volatile("st.relaxed.cta.shared::cta.v2.b64 [%0], {%1, %2};"
                     ::"r"(p), "l"(half_of(v.x, tag)), "l"(half_of(v.y, tag)) : "memory");
    else asm volatile("st.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(p), "l"(half_of(v.x, tag)) : "memory");
}
// The same to a generic address, where `on` is not 0 (predicated, no branch).
template <bool PAIR>
__device__ __forceinline__ void st_entry_if(uint32_t on, unsigned long long p, float2 v, uint32_t tag) {
    if (PAIR)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.relaxed.gpu.v2.b64 [%1], {%2, %3};\n\t}"
                     ::"r"(on), "l"(p), "l"(half_of(v.x, tag)), "l"(half_of(v.y, tag)) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.relaxed.gpu.b64 [%1], %2;\n\t}"
                     ::"r"(on), "l"(p), "l"(half_of(v.x, tag)) : "memory");
}
// ... where x < lim (unsigned)
template <bool PAIR>
__device__ __forceinline__ void st_entry_below(uint32_t x, uint32_t lim, unsigned long long p, float2 v, uint32_t tag) {
    if (PAIR)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %0, %1;\n\t@q st.relaxed.gpu.v2.b64 [%2], {%3, %4};\n\t}"
                     ::"r"(x), "r"(lim), "l"(p), "l"(half_of(v.x, tag)), "l"(half_of(v.y, tag)) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %0, %1;\n\t@q st.relaxed.gpu.b64 [%2], %3;\n\t}"
                     ::"r"(x), "r"(lim), "l"(p), "l"(half_of(v.x, tag)) : "memory");
}
// to shared memory where x == y: an entry, and a row with its limits (two entries, always both halves)
template <bool PAIR>
__device__ __forceinline__ void sts_entry_at(int32_t x, int32_t y, uint32_t p, float2 v, uint32_t tag) {
    if (PAIR)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.eq.s32 q, %0, %1;\n\t@q st.relaxed.cta.shared::cta.v2.b64 [%2], {%3, %4};\n\t}"
                     ::"r"(x), "r"(y), "r"(p), "l"(half_of(v.x, tag)), "l"(half_of(v.y, tag)) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.eq.s32 q, %0, %1;\n\t@q st.relaxed.cta.shared::cta.b64 [%2], %3;\n\t}"
                     ::"r"(x), "r"(y), "r"(p), "l"(half_of(v.x, tag)) : "memory");
}
__device__ __forceinline__ void sts_row_at(int32_t x, int32_t y, uint32_t p, float2 row, float2 lim, uint32_t tag) {
    sts_entry_at<true>(x, y, p, row, tag);
    sts_entry_at<true>(x, y, p + 16u, lim, tag);
}
__device__ __forceinline__ unsigned long long generic_of_shared(uint32_t a) {
    unsigned long long g;
    asm("{\n\t.reg .u64 x;\n\tcvt.u64.u32 x, %1;\n\tcvta.shared.u64 %0, x;\n\t}" : "=l"(g) : "r"(a));
    return g;
}
__device__ __forceinline__ uint32_t lds_word(uint32_t p) {
    uint32_t v;
    asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void sts_word(uint32_t p, uint32_t v) {
    asm volatile("st.relaxed.cta.shared::cta.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ float lds_f32(uint32_t p) {
    float v;
    asm volatile("ld.shared::cta.f32 %0, [%1];" : "=f"(v) : "r"(p));
    return v;
}
__device__ __forceinline__ float lds_f32v(uint32_t p) {
    float v;
    asm volatile("ld.volatile.shared::cta.f32 %0, [%1];" : "=f"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Algorithm 1's update on loads A (the row, f_e(A) = s) and B: with PAIR the loads are
// unevaluated pairs hi + lo and the transfer is moved by Knuth's TwoSum, so no update rounds a
// load.  The weight moved from A to B is half the difference, clipped to [nb, ca]: ca = s may
// leave A, -nb = w - s may leave B (both 0 without an edge).
template <bool PAIR>
__device__ __forceinline__ float transfer(float2& A, float2& B, float ca, float nb, float s, float w) {
    const float diff = PAIR ? (A.x - B.x) + (A.y - B.y) : A.x - B.x;
    const float dd = fminf(fmaxf(diff * 0.5f, nb), ca);
    if (PAIR) {
        const float ta = A.x - dd, ba = ta - A.x;
        A.y += (A.x - (ta - ba)) + (-dd - ba);
        A.x = ta;
        const float tb = B.x + dd, bb = tb - B.x;
        B.y += (B.x - (tb - bb)) + (dd - bb);
        B.x = tb;
    } else {
        A.x -= dd;
        B.x += dd;
    }
    return fminf(s - dd, w);
}

constexpr int kGroup = 4;             // steps per check of the input streams
// A group awaits the inputs of all its steps, so a low tile runs up to three classes behind the
// tile before it for the sake of entries it does not need yet.  With an odd one, the top tile's
// last inputs come from the last high tile, whose diagonal runs beside the last low tile's,
// which hangs on the top tile again through all KL low tiles: there the low tiles await their
// inputs step by step, or they would wait for one another.  A hop back goes one class back
// there and two forward elsewhere, so the last w classes of a lap do with w > 2 (KL - w) + 32:
// w = 3/4 KL + kFine.
constexpr int kFine = 64;

// One tile of a warp: the row and column loads of its lanes, its cells and its streams.
struct Tile {
    float2 R, C;
    Entry e[kGroup];       // input entries read ahead
    float* gs;             // global splits of step 0, this lane
    const float* src_s;    // global splits and weights of step 0, this lane's 16 bytes
    const float* src_w;
    uint32_t cells, wofs;  // staged splits (shared address, this lane); weights wofs further on
    int32_t c_end;         // chunks of this lap
    uint32_t ring, rmask, in_off;  // input entry of step s: slot (s + in_off) & rmask
    uint32_t cons;         // word where this tile publishes how far it read
    bool tell;             // false: its inputs are read again
    int32_t base, cnt;     // first row, rows
    int32_t in_end;        // steps with an input column: P - base
    uint32_t tag;          // tag of step 0 in the current lap
    int32_t live_from, live_to;   // columns (from the tile's first row) that are updated: [from, to)
    int32_t exit;          // the step after which this lane's row ends its lap (-1: no row)
    uint32_t exit_tag;     // tag of its entry in the lap it enters then
    unsigned long long exit_to;   // where it goes (generic address)
    // output stream: after step s entry q = s - off of the next tile, q < lim, from one lane, to
    // slot s & omask
    int32_t off, lim;
    uint32_t mine;         // lim in the lane that gives the columns out, 0 in the others
    unsigned long long out;   // generic address of slot 0
    uint32_t omask;        // ring mask (all ones: an array)
    uint32_t out_cons;     // the reader's published word (0: no ring to wait for)
    uint32_t seen;         // its value when last looked at
    uint32_t otag;         // tag of the reader's step 0 in the lap it will read in
    bool turns;            // the reader has a ring for every other lap
    // the odd one (even n): slots (shared addresses) where the low warp hands it to the high one, and
    // the high one its rows to the low one, the k-th of a lap in slot k mod 4 (the fourth after it
    // is only written when it was read); tag of row 0 in this lap
    uint32_t odd_slots, row_slots, odd_tag;
    uint32_t odd_low, odd_high;   // rows of the pair's low and high tile that have an edge to it (bit i)
    int32_t odd_at;        // the step at which this lane's row meets it (-1: never)
};

struct Bad {
    const SysArgs* a;
    volatile int32_t* flag;   // block-wide
    __device__ __forceinline__ bool expired(uint32_t spins, uint32_t limit) const {
        if ((spins & 255u) != 255u) return false;
        if (*flag) return true;
        if (spins >= (limit >> a->spin_shift) || *(volatile int32_t*)a->err != 0) {
            *flag = 1;
            atomicOr(a->err, kWaveExpired);
            return true;
        }
        return false;
    }
};

// A warp that polls shared memory holds up the shuffles of the warps that work: after a few polls
// it sleeps between them.
__device__ __forceinline__ void poll_pause(uint32_t spins) {
    if (spins > 8u) __nanosleep(spins > 64u ? 200u : 40u);
}

template <bool PAIR>
__device__ __forceinline__ void read_ahead(Tile& t, int32_t s) {
#pragma unroll
    for (int j = 0; j < kGroup; ++j) t.e[j] = lds_entry<PAIR>(t.ring + ((((uint32_t)(s + j) + t.in_off) & t.rmask) << 4));
}

// 0 if the entries of steps s + j0 .. s + j1 - 1 are in t.e
template <bool PAIR>
__device__ __forceinline__ uint32_t missing(const Tile& t, int32_t s, int j0, int j1) {
    uint32_t acc = 0u;
#pragma unroll
    for (int j = 0; j < kGroup; ++j) {
        if (j < j0 || j >= j1) continue;
        const uint32_t tag = t.tag + (uint32_t)(s + j);
        acc |= (uint32_t)(t.e[j].a >> 32) ^ tag;
        if (PAIR) acc |= (uint32_t)(t.e[j].b >> 32) ^ tag;
    }
    return acc;
}

// the columns one lane on; lane 0 takes `in`
template <bool PAIR>
__device__ __forceinline__ float2 shifted(float2 C, bool first_lane, float2 in) {
    float2 r = C;
    const float x = __shfl_up_sync(0xffffffffu, C.x, 1);
    r.x = first_lane ? in.x : x;
    if (PAIR) {
        const float y = __shfl_up_sync(0xffffffffu, C.y, 1);
        r.y = first_lane ? in.y : y;
    }
    return r;
}

// column C goes out after step s (slot: address of the slot of step s - j)
template <bool PAIR, bool RANGED>
__device__ __forceinline__ void emit(const Tile& t, unsigned long long slot, int32_t s, int j, float2 C) {
    const uint32_t q = (uint32_t)(s - t.off);
    if (RANGED) st_entry_below<PAIR>(q, t.mine, slot + 16u * (uint32_t)j, C, t.otag + q);
    else st_entry_if<PAIR>(t.mine, slot + 16u * (uint32_t)j, C, t.otag + q);
}
__device__ __forceinline__ unsigned long long out_slot(const Tile& t, int32_t s) {
    return t.out + ((unsigned long long)((uint32_t)s & t.omask) << 4);
}

// rows whose lap ended in steps s .. s + k - 1 (they do not change after it)
template <bool PAIR>
__device__ __forceinline__ void leave(const Tile& t, int32_t s, uint32_t k) {
    st_entry_below<PAIR>((uint32_t)(t.exit - s), k, t.exit_to, t.R, t.exit_tag);
}

// Offset of a chunk in the staged cells: all of a tile's cells stay in shared memory (RES), or the
// last kSlots chunks.
template <bool RES>
__device__ __forceinline__ uint32_t chunk_slot(int32_t c) {
    return (uint32_t)(RES ? c : (c & (kSlots - 1))) * kChunkBytes;
}

template <bool WEIGHTED, bool RES>
__device__ __forceinline__ void fetch_chunk(const Tile& t, int32_t c, int lane) {
    const uint32_t d = t.cells + chunk_slot<RES>(c) + 12u * (uint32_t)lane;   // cells is this lane's, 4 bytes each
    const float* ps = t.src_s + (int64_t)c * (kChunk * 32);
#pragma unroll
    for (int i = 0; i < kChunk / 4; ++i) cp_async16(d + 512u * i, ps + 128 * i);
    if (WEIGHTED) {
        const float* pw = t.src_w + (int64_t)c * (kChunk * 32);
#pragma unroll
        for (int i = 0; i < kChunk / 4; ++i) cp_async16(d + t.wofs + 512u * i, pw + 128 * i);
    }
}

// room in the reader's ring for everything emitted up to step s_last
__device__ __forceinline__ void await_room(Tile& t, int32_t s_last, const Bad& w, bool& bad) {
    const int32_t q = min(s_last - t.off, t.lim - 1);
    const int32_t back = q - (kRing - 1);
    if (t.out_cons == 0u || q < 0 || (back <= 0 && t.turns)) return;
    const uint32_t need = t.otag + (uint32_t)max(back, 0);
    uint32_t spins = 0;
    while ((int32_t)(t.seen - need) < 0 && !bad) {
        t.seen = lds_word(t.out_cons);
        if ((int32_t)(t.seen - need) < 0) {
            if (w.expired(++spins, kSpinSmem)) bad = true;
            poll_pause(spins);
        }
    }
    bad = __any_sync(0xffffffffu, bad);
}

// What comes before the steps of chunk c: tell how far the inputs were read, have the chunk's cells
// and the next fetch under way, and room for what the chunk gives out.
template <bool WEIGHTED, bool RES>
__device__ __forceinline__ void begin_chunk(Tile& t, int32_t c, int lane, const Bad& w, bool& bad) {
    if (lane == 0 && t.tell) sts_word(t.cons, t.tag + (uint32_t)(c * kChunk));
    if (!RES) {
        cp_wait<kAhead - 1>();
        __syncwarp();
        if (c + kAhead < t.c_end) fetch_chunk<WEIGHTED, false>(t, c + kAhead, lane);
        cp_commit();
    }
    await_room(t, c * kChunk + kChunk - 1, w, bad);
}

template <bool RES>
__device__ __forceinline__ void store_split(const Tile& t, int32_t s, uint32_t slot_off, float ns, bool edge) {
    if (RES) {
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared::cta.f32 [%1], %2;\n\t}"
                     ::"r"(edge ? 1u : 0u), "r"(t.cells + slot_off), "f"(ns) : "memory");
    } else if (edge) {
        t.gs[(int64_t)s << 5] = ns;
    }
}

// until the entry of step s is in the ring: polls it alone
template <bool PAIR>
__device__ __forceinline__ void poll_entry(const Tile& t, int32_t s, const Bad& w, bool& bad) {
    const uint32_t at = t.ring + ((((uint32_t)s + t.in_off) & t.rmask) << 4);
    uint32_t spins = 0;
    while (__any_sync(0xffffffffu, !lds_entry<PAIR>(at).template is<PAIR>(t.tag + (uint32_t)s)) && !bad) {
        if (w.expired(++spins, kSpinSmem)) bad = true;
        bad = __any_sync(0xffffffffu, bad);
        poll_pause(spins);
    }
}

// until the entries j0 .. j1 - 1 of the group at step s0 are in t.e.  They mostly come in order, so the last
// one is polled; but the wrap's come from the warps of different tiles, and nothing orders those: where the
// group is not whole then, its entries are polled one after the other.  (An entry that every lane has seen
// stays until this tile has told that it read it.)  Without a loop around the polls, each of which is
// bounded, a group costs least: n 9,109 at density 0.156 1,014 us a pass (a counted loop 1,061, or 1,090 where
// the clipping below was part of it), 6,193 weighted 714 (746, 775).
template <bool PAIR>
__device__ __forceinline__ void await_group(Tile& t, int32_t s0, int j0, int j1, const Bad& w, bool& bad) {
    if (__all_sync(0xffffffffu, missing<PAIR>(t, s0, j0, j1) == 0u)) return;
    poll_entry<PAIR>(t, s0 + j1 - 1, w, bad);
    read_ahead<PAIR>(t, s0);
    if (__all_sync(0xffffffffu, missing<PAIR>(t, s0, j0, j1) == 0u)) return;
#pragma unroll 1
    for (int j = j0; j < j1 - 1; ++j) poll_entry<PAIR>(t, s0 + j, w, bad);
    read_ahead<PAIR>(t, s0);
}

// the same, for those of the entries that exist (EDGE: the inputs may run out inside the group)
template <bool PAIR, bool EDGE>
__device__ __forceinline__ void await_entries(Tile& t, int32_t s0, int j0, int j1, const Bad& w, bool& bad) {
    if (EDGE && s0 + j1 > t.in_end) {
        if (s0 + j0 < t.in_end) await_group<PAIR>(t, s0, j0, t.in_end - s0, w, bad);
        return;
    }
    await_group<PAIR>(t, s0, j0, j1, w, bad);
}

// an entry in a slot of the odd exchange
template <bool PAIR>
__device__ __forceinline__ float2 await_slot(uint32_t at, uint32_t want, const Bad& w, bool& bad) {
    // (16-byte reads are served a quarter warp at a time, so lanes may see different states: the
    // warp goes on when all of them have the entry)
    Entry v = lds_entry<PAIR>(at);
    uint32_t spins = 0;
    while (!__all_sync(0xffffffffu, v.template is<PAIR>(want)) && !bad) {
        if ((++spins & 255u) == 255u) {
            if (w.expired(spins, kSpinSmem)) bad = true;
            bad = __any_sync(0xffffffffu, bad);
            __nanosleep(40);
        }
        v = lds_entry<PAIR>(at);
    }
    return v.value();
}

// Chunks [c0, c1) of a tile, whole steps only.  Straight-line groups of four steps without a
// branch: the group's cells are read first and its input entries are checked together; a step's
// columns are handed on before its results are stored, so that the chain of a step is one
// shuffle and one transfer.  DIAG: the first 64 steps, where a column that reaches its own row
// becomes that row, after meeting the odd one (ODD).  EDGE: rows may end and inputs run out
// (steps past the end change nothing).  FINE: inputs are awaited step by step (see kFine).
template <bool PAIR, bool WEIGHTED, bool RES, bool DIAG, int ODD, bool EDGE, bool FINE, bool LIVE>
__device__ __forceinline__ void run_chunks(Tile& t, int32_t c0, int32_t c1, int lane, float2& odd, const Bad& w,
                                           bool& bad) {
#pragma unroll 1
    for (int32_t c = c0; c < c1; ++c) {
        begin_chunk<WEIGHTED, RES>(t, c, lane, w, bad);
        if (bad) return;
        uint32_t slot = chunk_slot<RES>(c);
#pragma unroll 1
        for (int32_t s0 = c * kChunk; s0 < c * kChunk + kChunk; s0 += kGroup, slot += 128u * kGroup) {
            float sv[kGroup], wv[kGroup];
#pragma unroll
            for (int j = 0; j < kGroup; ++j) {
                sv[j] = lds_f32(t.cells + slot + 128u * j);
                wv[j] = WEIGHTED ? lds_f32(t.cells + t.wofs + slot + 128u * j) : 1.0f;
            }
            float* gs = t.gs + ((int64_t)s0 << 5);
            const unsigned long long os = out_slot(t, s0);
            await_entries<PAIR, EDGE>(t, s0, 0, FINE ? 1 : kGroup, w, bad);
            // past the last column: a spent entry, which meets no edge
            t.C = shifted<PAIR>(t.C, lane == 0, t.e[0].value());
#pragma unroll
            for (int j = 0; j < kGroup; ++j) {
                const int32_t s = s0 + j;
                const float x = sv[j], y = wv[j];
                bool ed = WEIGHTED ? y > 0.0f : x >= 0.0f;
                if (LIVE) ed = ed && s - lane >= t.live_from && s - lane < t.live_to;
                const float ca = LIVE ? (ed ? x : 0.0f) : (WEIGHTED ? x : fmaxf(x, 0.0f));
                const float nb = LIVE || !WEIGHTED ? (ed ? x - y : 0.0f) : x - y;
                float2 A = t.R, B = t.C;
                float ns;
                if (DIAG && (j & 1) == 0) {
                    const bool self = 2 * lane == s && lane < t.cnt;
                    const int32_t i = s >> 1;   // the row at the diagonal
                    float2 o = odd;
                    if (ODD == 2 && ((t.odd_high >> (i & 31)) & 1u) && i < 32) {
                        // high row i: its load and limits to the low warp, which moves the odd one past
                        // it; the odd one's load before that comes back
                        const uint32_t k = (uint32_t)__popc(t.odd_high & ((1u << i) - 1u)) & 3u;
                        const uint32_t at = t.row_slots + 32u * k;
                        sts_row_at(s, t.odd_at, at, B, make_float2(ca, nb), t.odd_tag + (uint32_t)i);
                        o = await_slot<PAIR>(t.odd_slots + 16u * k, t.odd_tag + (uint32_t)i, w, bad);
                    }
                    A.x = self ? B.x : A.x;
                    B.x = self ? o.x : B.x;
                    if (PAIR) {
                        A.y = self ? B.y : A.y;
                        B.y = self ? o.y : B.y;
                    }
                    ns = transfer<PAIR>(A, B, ca, nb, x, y);   // a column that became a row is not read again
                    if (ODD == 1 && i < 32) {   // (i is the warp's, and so are the branches)
                        if ((t.odd_low >> i) & 1u) {
                            odd.x = __shfl_sync(0xffffffffu, B.x, i);
                            if (PAIR) odd.y = __shfl_sync(0xffffffffu, B.y, i);
                        }
                        if ((t.odd_high >> i) & 1u) {   // the high row's turn: the same update as in its own warp
                            const uint32_t k = (uint32_t)__popc(t.odd_high & ((1u << i) - 1u)) & 3u;
                            sts_entry_at<PAIR>(lane, 0, t.odd_slots + 16u * k, odd, t.odd_tag + (uint32_t)i);
                            const uint32_t at = t.row_slots + 32u * k;
                            const float2 lim = await_slot<true>(at + 16u, t.odd_tag + (uint32_t)i, w, bad);
                            float2 r = await_slot<true>(at, t.odd_tag + (uint32_t)i, w, bad);
                            transfer<PAIR>(r, odd, lim.x, lim.y, 0.0f, 1.0f);
                        }
                    }
                } else {
                    ns = transfer<PAIR>(A, B, ca, nb, x, y);
                }
                t.R = A;
                if (FINE && j + 1 < kGroup) await_entries<PAIR, EDGE>(t, s0, j + 1, j + 2, w, bad);
                t.C = j + 1 < kGroup ? shifted<PAIR>(B, lane == 0, t.e[(j + 1) & (kGroup - 1)].value()) : B;
                if (j == kGroup - 2) read_ahead<PAIR>(t, s0 + kGroup);
                if (!DIAG || EDGE || j == kGroup - 1) emit<PAIR, DIAG || EDGE>(t, os, s, j, B);   // a whole tile's first is after step 63
                // once a group, but where the steps to come may hang on a row that ended
                if (EDGE && (DIAG || FINE)) leave<PAIR>(t, s, 1u);
                else if (EDGE && j == kGroup - 1) leave<PAIR>(t, s0, kGroup);
                if (RES) store_split<true>(t, s, slot + 128u * j, ns, ed);
                else if (ed) gs[j << 5] = ns;
            }
        }
        if (bad) return;
    }
}

// One step of a tile, any position: the ends of a segment at a cut.
template <bool PAIR, bool WEIGHTED, bool RES>
__device__ __forceinline__ void step_any(Tile& t, int32_t s, bool shift, bool diag, int lane, const Bad& w, bool& bad) {
    if (shift) {
        Entry e;
        e.a = e.b = 0ull;
        if (s < t.in_end) {
            const uint32_t want = t.tag + (uint32_t)s;
            uint32_t spins = 0;
            do {
                e = lds_entry<PAIR>(t.ring + ((((uint32_t)s + t.in_off) & t.rmask) << 4));
                if (!e.template is<PAIR>(want) && w.expired(++spins, kSpinSmem)) bad = true;
            } while (!e.template is<PAIR>(want) && !bad);
            bad = __any_sync(0xffffffffu, bad);
        }
        t.C = shifted<PAIR>(t.C, lane == 0, e.value());
    }
    const uint32_t slot = chunk_slot<RES>(s / kChunk) + 128u * (uint32_t)(s & (kChunk - 1));
    const float x = lds_f32(t.cells + slot);
    const float y = WEIGHTED ? lds_f32(t.cells + t.wofs + slot) : 1.0f;
    const bool ed = (WEIGHTED ? y > 0.0f : x >= 0.0f) && s - lane >= t.live_from && s - lane < t.live_to;
    const bool self = diag && 2 * lane == s && lane < t.cnt;   // the column is this lane's own row
    float2 A = self ? t.C : t.R;   // (without an odd one: with one the diagonal is never ragged)
    float2 B = t.C;
    const float ns = transfer<PAIR>(A, B, ed ? x : 0.0f, ed ? x - y : 0.0f, x, y);
    t.R = A;
    t.C = B;
    emit<PAIR, true>(t, out_slot(t, s), s, 0, B);
    leave<PAIR>(t, s, 1u);
    store_split<RES>(t, s, slot, ns, ed);
}

template <bool PAIR, bool WEIGHTED, bool RES>
__global__ void __launch_bounds__(64 * kMaxW, 1) k_sweep_systolic(const SysArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ volatile int32_t bad_flag;
    const Geo g = a.g;
    const int W = a.W;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int32_t P = g.P;
    const uint32_t lapt = (uint32_t)(P + kPad);      // tags per lap
    const bool single = gridDim.x == 1;
    const bool duo = a.odd != 0;
    // shared memory: the cells (RES: all of them; else two tiles' stages per pair), per pair 2
    // rings (and a second one for high tile 0), the odd exchange's slots and 2 published words; one
    // block alone keeps the wrap array here too
    const uint32_t sb = smem_u32(smem);
    const uint32_t cell_tile = WEIGHTED ? 2u * kCellBytes : kCellBytes;
    const uint32_t all_cells = (uint32_t)g.steps() << 7;   // RES only: one array's bytes
    const uint32_t rings = sb + (RES ? (WEIGHTED ? 2u : 1u) * all_cells : 2u * (uint32_t)W * cell_tile);
    const uint32_t odds = rings + (uint32_t)(W * 2 + 1) * kRing * 16u;
    const uint32_t words = odds + (uint32_t)W * kOddBytes;
    const uint32_t wrap_sm = words + (uint32_t)W * 16u;
    auto ring_of = [&](int pr, int high) -> uint32_t { return rings + (uint32_t)(pr * 2 + high) * kRing * 16u; };
    auto word_of = [&](int pr, int high) -> uint32_t { return words + (uint32_t)(pr * 2 + high) * 4u; };
    auto odd_of = [&](int pr) -> uint32_t { return odds + (uint32_t)pr * kOddBytes; };
    {   // clear the rings, slots and the wrap; nothing read yet
        const uint32_t end = single ? wrap_sm + (lapt << 4) : wrap_sm;
        for (uint32_t x = rings + 4u * threadIdx.x; x < end; x += 4u * blockDim.x) sts_word(x, 0u);   // no tag is 0
        __syncthreads();
        if ((int)threadIdx.x < 2 * W)
            sts_word(word_of(threadIdx.x >> 1, threadIdx.x & 1), a.tag0 + ((threadIdx.x & 1) ? lapt : 0u));
        if (threadIdx.x == 0) bad_flag = 0;
    }
    __syncthreads();
    Bad bw{&a, &bad_flag};
    bool bad = false;
    const int64_t pitch = (int64_t)P + kPad;
    const int32_t T = a.T;
    // lap x of this launch (-1 .. T) has tags tag0 + (x + 1) lapt + step
    auto lap_tag = [&](int32_t lap) -> uint32_t { return a.tag0 + (uint32_t)(lap + 1) * lapt; };

    if (warp >= 2 * W) {
        // ---------------- import warps: refill the rings of the block's first pair
        if (single) return;
        const int high = warp - 2 * W;
        const int32_t p0 = (int32_t)blockIdx.x * W;
        if (high ? p0 >= g.KU : p0 >= g.KL) return;
        const int32_t base = (high ? g.h : 0) + 32 * p0;
        const ulonglong2* src = (high ? a.in_high : a.in_low) + (int64_t)blockIdx.x * pitch;
        const uint32_t ring = ring_of(0, high), word = word_of(0, high);
        for (int32_t lap = high ? 0 : -1; lap < T; ++lap) {
            int32_t s = 0, e = P - base;
            if (!high && lap < 0) s = P - 2 * base + 1;
            if (!high && lap == T - 1) e = min(e, P - 2 * base);
            const uint32_t tg = lap_tag(lap);
            uint32_t spins = 0;
            while (s < e) {
                const int32_t q = s + lane;
                const Entry v = ldg_entry<PAIR>(src + min(q, e - 1));
                const bool ok = q < e && v.template is<PAIR>(tg + (uint32_t)q);
                const unsigned miss = __ballot_sync(0xffffffffu, !ok);
                const int got = miss ? __ffs(miss) - 1 : 32;
                if (got == 0) {
                    if (bw.expired(++spins, kSpinGlobal)) bad = true;
                    if (__any_sync(0xffffffffu, bad)) return;
                    continue;
                }
                spins = 0;
                const int32_t back = s + got - kRing;    // the slot of the last entry must have been read
                const uint32_t need = tg + (uint32_t)(back > 0 ? back : 0);
                uint32_t sp2 = 0;
                while ((int32_t)(lds_word(word) - need) < 0 && !bad)
                    if (bw.expired(++sp2, kSpinSmem)) bad = true;
                if (__any_sync(0xffffffffu, bad)) return;
                if (lane < got) sts_entry<PAIR>(ring + (((uint32_t)q & (kRing - 1)) << 4), v.value(), tg + (uint32_t)q);
                s += got;
            }
        }
        return;
    }
    // ---------------- tiles: warp 2 w runs the low tile of the block's pair w, warp 2 w + 1 the high one
    const int wp = warp >> 1;
    const int high = warp & 1;
    const int32_t p = (int32_t)blockIdx.x * W + wp;
    if (p >= (high ? g.KU : g.KL)) return;
    const bool last = p == g.KL - 1;
    const bool next_here = !last && wp + 1 < W;
    const int64_t step0 = high ? g.high(p) : g.low(p);
    Tile t;
    t.R = t.C = make_float2(0.0f, 0.0f);
    for (int j = 0; j < kGroup; ++j) t.e[j].a = t.e[j].b = 0ull;
    t.base = (high ? g.h : 0) + 32 * p;
    t.cnt = min(32, (high ? P : g.h) - t.base);
    t.in_end = P - t.base;
    const int32_t row = t.base + lane;
    t.gs = a.cs + (step0 << 5) + lane;
    t.src_s = a.cs + (step0 << 5) + 4 * lane;
    t.src_w = WEIGHTED ? a.cw + (step0 << 5) + 4 * lane : nullptr;
    t.cells = sb + (RES ? (uint32_t)step0 << 7 : (uint32_t)warp * cell_tile) + 4u * (uint32_t)lane;
    t.wofs = RES ? all_cells : kCellBytes;
    t.c_end = 0;
    t.ring = ring_of(wp, high);
    t.rmask = kRing - 1;
    t.in_off = 0u;       // entries from the import warp; from a tile of this block: its steps
    if (wp > 0) t.in_off = 63u;
    else if (single && high) t.in_off = (uint32_t)(2 * (g.h - 32 * (g.KL - 1)) - 1);
    t.cons = word_of(wp, high);
    t.tell = true;
    t.live_from = INT32_MIN;
    t.live_to = INT32_MAX;
    t.exit = lane < t.cnt ? P - 1 - t.base + lane : -1;
    t.exit_to = (single ? generic_of_shared(wrap_sm) : (unsigned long long)a.in_low) + ((unsigned long long)(uint32_t)row << 4);
    t.off = 63;
    t.lim = 0;           // no reader
    t.out = 0ull;
    t.omask = kRing - 1;
    t.out_cons = 0u;
    t.seen = 0u;
    t.turns = false;
    if (high ? p + 1 < g.KU : !last) {   // the same tile of the next pair
        t.lim = P - t.base - 32;
        if (next_here) {
            t.out = generic_of_shared(ring_of(wp + 1, high));
            t.out_cons = word_of(wp + 1, high);
        } else {
            t.out = (unsigned long long)((high ? a.in_high : a.in_low) + ((int64_t)blockIdx.x + 1) * pitch - 63);
            t.omask = 0xffffffffu;
        }
    } else if (!high && g.KU > 0) {      // the last low tile feeds the first high one, a lap later
        t.off = 2 * t.cnt - 1;
        t.lim = P - g.h;
        if (single) {
            t.out_cons = word_of(0, 1);
            t.turns = true;
        } else {
            t.out = (unsigned long long)(a.in_high - t.off);
            t.omask = 0xffffffffu;
        }
    }
    t.lim = max(t.lim, 0);
    t.mine = lane == (!high && last ? t.cnt - 1 : 31) ? (uint32_t)t.lim : 0u;
    // The odd one meets low row i, high row i, low row i + 1, ... of a pair, then goes to the next pair
    // (after the last to pair 0's next lap).  The low warp keeps it in registers and moves it past
    // the high rows too, as the high warp does for its own rows: both do the same update, so a
    // value crosses between the warps once, and nothing is sent back.
    t.odd_slots = odd_of(wp) + 16u;
    t.row_slots = odd_of(wp) + 80u;
    t.odd_at = lane < t.cnt ? 2 * lane : -1;
    t.odd_low = t.odd_high = 0u;
    if (duo) {   // rows without an edge to the odd one let it pass: nothing is exchanged for them
        auto edge_at = [&](int64_t first, bool is) -> bool {   // row `lane`'s cell with it: step 2 lane
            const int64_t c = ((first + 2 * lane) << 5) + lane;
            return is && (WEIGHTED ? a.cw[c] > 0.0f : a.cs[c] >= 0.0f);
        };
        t.odd_low = __ballot_sync(0xffffffffu, edge_at(g.low(p), 32 * p + lane < g.h));
        if (p < g.KU) t.odd_high = __ballot_sync(0xffffffffu, edge_at(g.high(p), g.h + 32 * p + lane < P));
    }
    float2 odd = make_float2(0.0f, 0.0f);

    // loads at the cut a + b = P: low rows in place, each row's next column P - row beside it
    if (!high && lane < t.cnt) {
        const float x = a.l[row], y = a.l_lo[row];
        t.R = PAIR ? make_float2(x, y) : make_float2(x + y, 0.0f);
        const int32_t col = P - row;
        if (col >= g.h && col < P) {
            const float cx = a.l[col], cy = a.l_lo[col];
            t.C = PAIR ? make_float2(cx, cy) : make_float2(cx + cy, 0.0f);
        }
    }
    const int32_t sLap = P - t.base + t.cnt - 1;            // steps of a whole lap
    const int32_t cLap = (sLap + kChunk - 1) / kChunk;
    const int32_t eC = (P - 1 - t.base) / kChunk;           // from here on rows end and inputs run out
    if (RES) {   // the tile's cells, for the whole launch
        for (int32_t c = 0; c < cLap; ++c) fetch_chunk<WEIGHTED, true>(t, c, lane);
        cp_commit();
        cp_wait<0>();
        __syncwarp();
    }
    for (int32_t lap = high ? 0 : -1; lap < T && !bad; ++lap) {
        // steps [sB, sE): the first and the last lap of a low tile are cut at the pass boundary
        const int32_t sB = lap < 0 ? P - 2 * t.base : 0;
        const int32_t sE = !high && lap == T - 1 ? P - 2 * t.base : sLap;
        t.tag = lap_tag(lap);
        t.otag = lap_tag(last && !high ? lap + 1 : lap);
        t.exit_tag = lap_tag(high ? lap : lap + 1) + (uint32_t)row;
        t.odd_tag = lap_tag(lap);
        if (single) {
            // The last low tile feeds high tile 0 a lap ahead, and must not wait there for the lap
            // before to be read (its own high tile's rows could then not leave): the laps take
            // turns on two rings.
            const uint32_t second = (uint32_t)(2 * W - 1) * kRing * 16u;
            if (high && p == 0) t.ring = ring_of(0, 1) + ((lap & 1) ? second : 0u);
            if (!high && last && g.KU > 0)
                t.out = generic_of_shared(ring_of(0, 1) + (((lap + 1) & 1) ? second : 0u));
            if (!high && p == 0) { t.ring = wrap_sm; t.rmask = 0xffffffffu; t.in_off = 0u; }
        }
        const int32_t cB = sB / kChunk, cE = (sE + kChunk - 1) / kChunk;
        t.c_end = cE;
        if (!RES) {
            // the splits this warp wrote in the lap before, by any lane, come before the copies below
            __threadfence();
            __syncwarp();
            for (int32_t c = cB; c < cB + kAhead; ++c) {
                if (c < cE) fetch_chunk<WEIGHTED, false>(t, c, lane);
                cp_commit();
            }
        }
        if (lap < 0) st_entry_if<PAIR>(row == 0 ? 1u : 0u, t.exit_to, t.R, lap_tag(0));   // row 0 ends at the cut
        if (!high && lap >= 0 && duo) {   // the odd one's way in: the loads, the pair before, or its block
            if (p == 0 && lap == 0) {
                const float x = a.l[P], y = a.l_lo[P];
                odd = PAIR ? make_float2(x, y) : make_float2(x + y, 0.0f);
            } else if (wp > 0 || single) {
                odd = await_slot<PAIR>(odd_of(wp), t.odd_tag, bw, bad);
            } else {
                Entry v;
                uint32_t spins = 0;
                do {
                    v = ldg_entry<PAIR>(a.in_odd + blockIdx.x);
                    if (!v.template is<PAIR>(t.odd_tag) && bw.expired(++spins, kSpinGlobal)) bad = true;
                    bad = __any_sync(0xffffffffu, bad);
                } while (__any_sync(0xffffffffu, !v.template is<PAIR>(t.odd_tag)) && !bad);
                odd = v.value();
            }
        }
        auto odd_out = [&]() {
            if (lane != 0) return;
            if (!last) {
                if (next_here) sts_entry<PAIR>(odd_of(wp + 1), odd, lap_tag(lap));
                else stg_entry<PAIR>(a.in_odd + blockIdx.x + 1, odd, lap_tag(lap));
            } else if (lap < T - 1) {
                if (single) sts_entry<PAIR>(odd_of(0), odd, lap_tag(lap + 1));
                else stg_entry<PAIR>(a.in_odd, odd, lap_tag(lap + 1));
            }
        };
        // whole chunks run straight-line; the ragged ones at a cut go step by step.  [f0, fe) are
        // whole (past a lap's end steps change nothing); [n0, n1) is the last part of a lap, where
        // low tiles await their inputs step by step
        const int32_t f0 = lap < 0 ? (sB + 1 + kChunk - 1) / kChunk : 0;
        const int32_t fe = !high && lap == T - 1 ? sE / kChunk : cE;
        const int32_t n0 = duo && !high ? max(0, (P - g.KL * 3 / 4 - kFine - 64 * p) / kChunk) : 0x7fffffff;
        const int32_t n1 = duo && !high ? max(0, (P - 64 * p + kChunk - 1) / kChunk) : 0x7fffffff;
        int32_t dg = lap >= 0 ? kDiag : 0;
        if (lap >= 0 && duo && !high && last) {
            // The last low tile first runs its triangle alone (columns below h), which needs no later
            // input: the top tile's last inputs come from the last high tile, which hangs on this
            // triangle by the odd one, and so must not hang on the top tile again.
            const uint32_t mine = t.mine;
            const int32_t exit = t.exit;
            t.mine = 0u;
            t.exit = -1;
            t.tell = false;
            t.in_end = t.cnt;
            t.live_to = t.cnt;
            t.c_end = min(cE, kDiag);
            run_chunks<PAIR, WEIGHTED, RES, true, 1, true, false, true>(t, 0, (2 * t.cnt - 1 + kChunk - 1) / kChunk, lane, odd,
                                                                      bw, bad);
            odd_out();
            t.mine = mine;
            t.exit = exit;
            t.tell = true;
            t.in_end = P - t.base;
            t.live_to = INT32_MAX;
            t.live_from = t.cnt;
            t.c_end = cE;
            dg = 0;
            if (!RES) {
                cp_wait<0>();
                __syncwarp();
                fetch_chunk<WEIGHTED, false>(t, 0, lane);
                cp_commit();
            }
        }
        for (int32_t c = cB; c < cE && !bad;) {
            if (c < f0 || c >= fe) {
                begin_chunk<WEIGHTED, RES>(t, c, lane, bw, bad);
                const int32_t lo = max(c * kChunk, sB), hi = min(c * kChunk + kChunk, sE);
#pragma unroll 1
                for (int32_t s = lo; s < hi && !bad; ++s)
                    step_any<PAIR, WEIGHTED, RES>(t, s, !(lap < 0 && s == sB), dg > 0, lane, bw, bad);
                ++c;
            } else if (c < dg) {
                const int32_t c1 = c + 1;
                const bool edge = last || c >= eC;    // rows end, inputs run out or columns go out early
                const bool fine = c >= n0 && c < n1;
                if (!duo && !edge) run_chunks<PAIR, WEIGHTED, RES, true, 0, false, false, false>(t, c, c1, lane, odd, bw, bad);
                else if (!duo) run_chunks<PAIR, WEIGHTED, RES, true, 0, true, false, false>(t, c, c1, lane, odd, bw, bad);
                else if (high && !edge) run_chunks<PAIR, WEIGHTED, RES, true, 2, false, false, false>(t, c, c1, lane, odd, bw, bad);
                else if (high) run_chunks<PAIR, WEIGHTED, RES, true, 2, true, false, false>(t, c, c1, lane, odd, bw, bad);
                else if (!edge && !fine) run_chunks<PAIR, WEIGHTED, RES, true, 1, false, false, false>(t, c, c1, lane, odd, bw, bad);
                else run_chunks<PAIR, WEIGHTED, RES, true, 1, true, true, false>(t, c, c1, lane, odd, bw, bad);
                if (duo && !high && c1 == kDiag) odd_out();
                c = c1;
            } else if (c < kDiag && t.live_from >= 0) {
                run_chunks<PAIR, WEIGHTED, RES, false, 0, true, true, true>(t, c, c + 1, lane, odd, bw, bad);
                ++c;
            } else if (c >= n0 && c < n1) {
                const int32_t c1 = min(fe, n1);
                run_chunks<PAIR, WEIGHTED, RES, false, 0, true, true, false>(t, c, c1, lane, odd, bw, bad);
                c = c1;
            } else {
                int32_t c1 = c < n0 ? min(fe, n0) : fe;
                if (c < eC) {
                    c1 = min(c1, eC);
                    run_chunks<PAIR, WEIGHTED, RES, false, 0, false, false, false>(t, c, c1, lane, odd, bw, bad);
                } else {
                    run_chunks<PAIR, WEIGHTED, RES, false, 0, true, false, false>(t, c, c1, lane, odd, bw, bad);
                }
                c = c1;
            }
        }
        t.live_from = INT32_MIN;
        if (lane == 0) sts_word(t.cons, t.tag + lapt);
        cp_wait<0>();
    }
    if (RES)   // the splits back to their cells (a lane's own)
        for (int32_t s = 0; s < sLap; ++s) t.gs[(int64_t)s << 5] = lds_f32v(t.cells + 128u * (uint32_t)s);
    if (bad || high) return;
    // the cut after the last pass: rows in place, the column just updated is P - 1 - row
    auto put_load = [&](int32_t id, float2 v) {
        const float u = v.x + v.y;   // renormalise: l = fl(hi + lo), l_lo = exact remainder
        a.l[id] = u;
        a.l_lo[id] = PAIR ? v.y - (u - v.x) : 0.0f;
    };
    if (lane < t.cnt) {
        put_load(row, t.R);
        const int32_t col = P - 1 - row;
        if (col >= g.h) put_load(col, t.C);
    }
    if (duo && last && lane == 0) put_load(P, odd);
}

// ------------------------------------------------------------------ building and reading the cells

__global__ void k_fill_cells(float* __restrict__ x, int64_t n4, float val) {
    const float4 v = make_float4(val, val, val, val);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x)
        reinterpret_cast<float4*>(x)[i] = v;
}

// splits (equal, or the given canonical ones clamped to [0, w_e]) and weights into the cells;
// ids: the edges the array covers (null: all)
__global__ void k_cells_from_edges(Geo g, const int32_t* __restrict__ ids, int64_t k, const int32_t* __restrict__ u,
                                   const int32_t* __restrict__ v, const float* __restrict__ w,
                                   const float* __restrict__ s_canon, bool clamp, float* __restrict__ cs,
                                   float* __restrict__ cw) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = ids ? ids[i] : i;
        const int64_t c = g.cell(u[e], v[e]);
        const float we = w ? w[e] : 1.0f;
        float s = we * 0.5f;   // Algorithm 1: w_e / 2
        if (s_canon) s = clamp ? fminf(fmaxf(s_canon[e], 0.0f), we) : s_canon[e];
        cs[c] = s;
        if (cw) cw[c] = we;
    }
}

__global__ void k_cells_to_canonical(Geo g, const int32_t* __restrict__ ids, int64_t k, const int32_t* __restrict__ u,
                                     const int32_t* __restrict__ v, const float* __restrict__ cs,
                                     float* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = ids ? ids[i] : i;
        out[e] = cs[g.cell(u[e], v[e])];
    }
}

// FP64 loads from the splits: the edges are in canonical order, so the low ends of a warp form
// runs whose sums are added with one atomic each; the high ends take one each.
__global__ void k_cells_rederive(Geo g, const int32_t* __restrict__ ids, int64_t k, const int32_t* __restrict__ u,
                                 const int32_t* __restrict__ v, const float* __restrict__ w,
                                 const float* __restrict__ cs, double* __restrict__ L64) {
    const unsigned lane = lane_id();
    for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < k; b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = b0 + threadIdx.x;
        const bool ok = i < k;
        const int64_t e = ok ? (ids ? ids[i] : i) : 0;
        const int32_t a = ok ? u[e] : -1;
        double s = 0.0;
        if (ok) {
            const int32_t b = v[e];
            s = (double)cs[g.cell(a, b)];
            atomicAdd(&L64[b], (w ? (double)w[e] : 1.0) - s);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, s, o);
            const int32_t ay = __shfl_up_sync(0xffffffffu, a, o);
            if ((int)lane >= o && ay == a) s += y;
        }
        const int32_t an = __shfl_down_sync(0xffffffffu, a, 1);
        if (ok && (lane == 31 || an != a)) atomicAdd(&L64[a], s);
    }
}

__device__ __forceinline__ int32_t circle_colour(int32_t P, int32_t a, int32_t b) {
    if (b == P) a *= 2;
    else a += b;
    return a >= P ? a - P : a;   // a + b < 2P and 2a < 2P
}

// class sizes into cnt [0, P), the edges at the odd one into cnt [P]
__global__ void k_colour_counts(int32_t P, const int32_t* __restrict__ u, const int32_t* __restrict__ v, int64_t m,
                                int32_t* __restrict__ cnt) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        atomicAdd(&cnt[circle_colour(P, u[e], v[e])], 1);
        if (v[e] == P) atomicAdd(&cnt[P], 1);
    }
}

}  // namespace

// Class sizes of the circle colouring of edges (u, v) and, last, the edges at the odd one, into
// cnt_h [P + 1] (host).
lowd_status lowd_sys_class_sizes(lowd_ctx* h, const int32_t* u, const int32_t* v, int64_t m, int32_t* cnt_h) {
    const int32_t P = h->n + (h->n & 1) - 1;
    int32_t* cnt = nullptr;
    LOWD_TRY(dalloc(h, &cnt, (size_t)P + 1));
    cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * ((size_t)P + 1), h->st);
    if (m > 0) LOWD_LAUNCH(k_colour_counts, grid_for(m), kT, 0, h->st, P, u, v, m, cnt);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(cnt_h, cnt, sizeof(int32_t) * ((size_t)P + 1), cudaMemcpyDeviceToHost, h->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
    dfree(h, &cnt);
    return e == cudaSuccess ? LOWD_OK : h->fail(e);
}

// Whether the array serves a graph whose circle colouring has C classes that hold edges, the longest
// of `longest` edges (padded to 4), `odd_edges` of the edges at the odd one.
//
// The array walks all P steps of a pass, the one-CTA kernels the C classes, so what is compared is P
// times a step with C times a class.  Measured (GB300, random graphs of 71 to 10,002 nodes, ns):
//  - staged sweep (pair loads), a class: 92 to 105 with up to 128 edges in the longest class, 120 to 136
//    up to 256, 157 to 170 up to 384, 192 to 201 up to 512 (a warp more per scheduler each time), 222 at
//    560, 300 to 317 at 770 (weighted 370);
//  - register ring (single FP32 loads), a class: 290 to 335, above 340 from 64 edges on;
//  - array, a step, odd n: 107 to 116 with pair loads, 84 to 95 with single ones (168 at 25 nodes, 124
//    at 33, 110 at 67);
//  - array, a step, even n, pair loads: 140 with hardly an edge a class, about 175 from 64 edges a class
//    on (more rows with an update in a group), and up to 130 more as more rows meet the odd one (2,048
//    nodes of degree 800 198, 770 nodes of degree 640 284); single loads: 430 at 16 nodes, 310 at 32, 203
//    at 66, 140 at 308, 113 at 2,048 and up to 100 more for the odd one.
// 10,001 nodes with 300 edges (300 classes): 89 us a pass on the register ring, 930 on the array; with
// 2,500 edges 202 on the staged sweep, 1,100 on the array; 1,030 nodes with 400 edges a class 200 and 292.
//
// The cells grow with n^2.  Up to 2^20 of them (4 MB) they may be any number, above it at most 64 per
// edge, above 2^26 (268 MB, n about 11,500) at most 16: sparser graphs keep the class-major arrays,
// which grow with the edges.
bool lowd_sys_serves(int32_t n, int64_t m, int32_t C, int32_t longest, int64_t odd_edges, bool pair) {
    const Geo g = make_geo(n);
    const int64_t x = C > 0 ? m / C : 0;   // edges a class
    int64_t step, cls;
    if (pair) {
        cls = 62 + 34 * (((int64_t)longest + 127) / 128);
        step = (n & 1) ? 112 : 140 + 40 * (x < 64 ? x : 64) / 64 + 130 * odd_edges / n;
    } else {
        cls = 300;
        step = (n & 1) ? 90 + 1500 / n : 120 + 6000 / n + 100 * odd_edges / n;
    }
    return lowd_sys_may_serve(n, m) && (int64_t)g.P * step < (int64_t)C * cls;
}

// What is known before the classes are counted.  (With fewer than P / 3 edges there are fewer classes than
// that, at 300 ns each at most: a longer class is paid for by the classes its edges do not fill.)
bool lowd_sys_may_serve(int32_t n, int64_t m) {
    if (n < 9) return false;
    const Geo g = make_geo(n);
    const int64_t cells = g.steps() << 5;
    if (cells > ((int64_t)1 << 20) && cells > (cells > ((int64_t)1 << 26) ? 16 : 64) * m) return false;
    return g.KL <= lowd_device_sms() * kPairs && 3 * m >= g.P;
}

lowd_status lowd_sys_build(lowd_ctx* h, const int32_t* plain_ids, int64_t m_plain, const float* init_splits_canon) {
    cudaStream_t st = h->st;
    const Geo g = make_geo(h->n);
    const int64_t cells = g.steps() << 5;
    LOWD_TRY(dalloc(h, &h->sys_cs, (size_t)cells));
    if (h->w) LOWD_TRY(dalloc(h, &h->sys_cw, (size_t)cells));
    if (plain_ids) {
        LOWD_TRY(dalloc(h, &h->sys_ids, (size_t)m_plain));
        LOWD_CK(cudaMemcpyAsync(h->sys_ids, plain_ids, sizeof(int32_t) * (size_t)m_plain, cudaMemcpyDeviceToDevice, st));
    }
    if (h->w) {
        LOWD_CK(cudaMemsetAsync(h->sys_cs, 0, sizeof(float) * (size_t)cells, st));
        LOWD_CK(cudaMemsetAsync(h->sys_cw, 0, sizeof(float) * (size_t)cells, st));
    } else {
        LOWD_LAUNCH(k_fill_cells, grid_for(cells / 4), kT, 0, st, h->sys_cs, cells / 4, -1.0f);
    }
    h->sys_m = m_plain;
    if (m_plain > 0)
        LOWD_LAUNCH(k_cells_from_edges, grid_for(m_plain), kT, 0, st, g, h->sys_ids, m_plain, h->u, h->v, h->w,
                    init_splits_canon, true, h->sys_cs, h->sys_cw);
    LOWD_CK_LAUNCH();
    return LOWD_OK;
}

lowd_status lowd_sys_rederive(lowd_ctx* h, double* L64) {
    if (h->sys_m > 0)
        LOWD_LAUNCH(k_cells_rederive, grid_for(h->sys_m), kT, 0, h->st, make_geo(h->n), h->sys_ids, h->sys_m, h->u,
                    h->v, h->w, h->sys_cs, L64);
    LOWD_CK_LAUNCH();
    return LOWD_OK;
}

lowd_status lowd_sys_to_canonical(lowd_ctx* h, float* out) {
    if (h->sys_m > 0)
        LOWD_LAUNCH(k_cells_to_canonical, grid_for(h->sys_m), kT, 0, h->st, make_geo(h->n), h->sys_ids, h->sys_m, h->u,
                    h->v, h->sys_cs, out);
    LOWD_CK_LAUNCH();
    return LOWD_OK;
}

lowd_status lowd_sys_from_canonical(lowd_ctx* h, const float* in) {
    if (h->sys_m > 0)
        LOWD_LAUNCH(k_cells_from_edges, grid_for(h->sys_m), kT, 0, h->st, make_geo(h->n), h->sys_ids, h->sys_m, h->u,
                    h->v, h->w, in, false, h->sys_cs, h->sys_cw);
    LOWD_CK_LAUNCH();
    return LOWD_OK;
}

// T passes over the plain edges.
cudaError_t lowd_sys_passes(lowd_ctx* h, int32_t passes) {
    const Geo g = make_geo(h->n);
    const bool weighted = h->w != nullptr;
    const bool pair = h->sys_pair != 0;
    // One block when the pairs fit it (every stream then stays in shared memory).  Of several, two
    // pairs each for odd n while every SM holds one: fewer warps per SM are faster steps, more
    // blocks are more slow hops.  Two against four pairs: n 513 57 against 60 us, 1,031 111 (121),
    // 4,047 437 (469), 6,193 weighted 718 (756), 9,109 1,015 (1,074); one pair 6 to 10 % slower than
    // two.  Even n gains nothing (770: 238 against 232 us, 9,110: 1,828 against 1,829) and keeps four.
    const int several = (g.P == h->n && g.KL <= lowd_device_sms() * kPairsOdd) ? kPairsOdd : kPairs;
    const int W = g.KL <= (weighted ? kPairs : kMaxW) ? g.KL : several;
    const int grid = (g.KL + W - 1) / W;
    h->wave_blocks = grid;
    size_t smem = (size_t)(2 * W + 1) * kRing * 16u + (size_t)W * (kOddBytes + 16u);
    if (grid == 1) smem += (size_t)(g.P + kPad) * 16u;
    const size_t arrays = weighted ? 2u : 1u;
    // a block that holds all its cells in shared memory for the launch saves their traffic and the
    // wait for the first of them at every lap (n up to about 300)
    const size_t all = arrays * ((size_t)g.steps() << 7);
    const bool res = grid == 1 && smem + all <= kSmemMost;
    smem += res ? all : (size_t)W * 2u * arrays * kCellBytes;
    auto kern = res ? (pair ? (weighted ? k_sweep_systolic<true, true, true> : k_sweep_systolic<true, false, true>)
                            : (weighted ? k_sweep_systolic<false, true, true> : k_sweep_systolic<false, false, true>))
                    : (pair ? (weighted ? k_sweep_systolic<true, true, false> : k_sweep_systolic<true, false, false>)
                            : (weighted ? k_sweep_systolic<false, true, false> : k_sweep_systolic<false, false, false>));
    cudaError_t e = lowd_allow_smem(kern, kSmemMost);
    if (e != cudaSuccess) return e;
    const size_t pitch = (size_t)g.P + kPad;
    const size_t words = (size_t)grid * (2 * pitch + 1);
    if (!h->sys_streams) {
        if (dalloc(h, &h->sys_streams, words) != LOWD_OK) return cudaErrorMemoryAllocation;
        h->sys_tag = 0;
    }
    const uint32_t lapt = (uint32_t)pitch;
    const int64_t per = ((int64_t)1 << 30) / lapt - 4;   // passes whose tags fit a launch
    for (int32_t done = 0; done < passes && e == cudaSuccess;) {
        const int32_t k = (int32_t)(passes - done < per ? passes - done : per);
        // tags go on from launch to launch; when they would pass 2^31 the streams are cleared
        if (h->sys_tag == 0 || (uint64_t)h->sys_tag + (uint64_t)(k + 3) * lapt >= (1ull << 31)) {
            e = cudaMemsetAsync(h->sys_streams, 0, sizeof(ulonglong2) * words, h->st);
            if (e != cudaSuccess) break;
            h->sys_tag = lapt;
        }
        SysArgs a;
        a.g = g;
        a.W = W;
        a.T = k;
        a.odd = (h->n & 1) == 0 ? 1 : 0;
        a.tag0 = h->sys_tag;
        a.cs = h->sys_cs;
        a.cw = h->sys_cw;
        a.l = h->l;
        a.l_lo = h->l_lo;
        a.in_low = h->sys_streams;
        a.in_high = h->sys_streams + (size_t)grid * pitch;
        a.in_odd = h->sys_streams + 2 * (size_t)grid * pitch;
        a.err = h->d_i32 + 8;
        a.spin_shift = 0;
        void* args[] = {&a};
        e = cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(32 * (2 * W + (grid > 1 ? 2 : 0))), args, smem,
                                        h->st);
        lowd_note_launch();
        h->sys_tag += (uint32_t)(k + 2) * lapt;
        done += k;
    }
    return e;
}

// Two blocks of the nine that 1,031 nodes take, with short limits: the columns that the others would
// hand on never come, so the waits expire (the streams are as long as for all nine).
cudaError_t lowd_sys_selftest(int32_t* err_bits) {
    const Geo g = make_geo(1031);
    const size_t pitch = (size_t)g.P + kPad, cells = (size_t)g.steps() << 5;
    const size_t blocks = (size_t)(g.KL + kPairsOdd - 1) / kPairsOdd;
    const size_t streams = 2 * blocks * pitch + blocks;
    const size_t smem = (size_t)(2 * kPairsOdd + 1) * kRing * 16u + (size_t)kPairsOdd * (kOddBytes + 16u) +
                        (size_t)kPairsOdd * 2u * kCellBytes;
    unsigned char* d = nullptr;
    cudaError_t e = cudaMalloc((void**)&d, 16 * streams + 4 * (cells + 2 * (size_t)g.n + 1));
    if (e != cudaSuccess) return e;
    SysArgs a;
    a.g = g;
    a.W = kPairsOdd;
    a.T = 2;
    a.odd = 0;
    a.tag0 = (uint32_t)pitch;
    a.in_low = reinterpret_cast<ulonglong2*>(d);
    a.in_high = a.in_low + blocks * pitch;
    a.in_odd = a.in_low + 2 * blocks * pitch;
    a.cs = reinterpret_cast<float*>(d + 16 * streams);
    a.cw = nullptr;
    a.l = a.cs + cells;
    a.l_lo = a.l + g.n;
    a.err = reinterpret_cast<int32_t*>(a.l_lo + g.n);
    a.spin_shift = 7;
    void* args[] = {&a};
    auto kern = k_sweep_systolic<true, false, false>;
    e = cudaMemset(d, 0, 16 * streams + 4 * (cells + 2 * (size_t)g.n + 1));
    if (e == cudaSuccess) e = lowd_allow_smem(kern, kSmemMost);
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel((const void*)kern, dim3(2), dim3(32 * (2 * kPairsOdd + 2)), args, smem, nullptr);
    lowd_note_launch();
    if (e == cudaSuccess) e = cudaMemcpy(err_bits, a.err, sizeof(int32_t), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e;
}
