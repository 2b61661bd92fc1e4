// Many time steps per launch with the state kept on chip: the fused stream-collide step of
// arXiv 2509.22308, Sec. III, for lattices whose state fits the GPU's registers (FP32) or shared
// memory (FP64, double-float).
//
// What bounds small lattices otherwise is not arithmetic: a launch per step (or per two) costs
// 2 - 4 us in launch, fill and drain and in the state's way through L2, where the update of a
// 512^2 FP32 lattice needs 0.7 us.  Here one cooperative launch takes up to kResidentSteps steps;
// global memory sees the state at its first and last step only, and the thread blocks exchange
// what crosses their borders.  Measured on GB300, one handle, us per step, plain launches / here:
// FP32 64^2 2.3 / 0.72, 256^2 2.5 / 1.0, 384 x 300 2.9 / 1.05, 512^2 3.9 / 1.8, 600^2 4.7 / 2.9;
// FP64 64^2 4.6 / 2.35, 256^2 7.3 / 4.0, 512^2 17.5 / 14.75 (FP64 pipe 80 % busy);
// double-float 256^2 5.2 / 3.7.
//
// Messages between blocks are 16-byte stores to mailboxes in global memory (they stay in L2) that
// carry their values together with a sequence number: the reader polls the message itself, so no
// fence, flag or grid-wide barrier is needed (a message needs about 600 clocks from SM to SM on one
// die and 1000 across the two; a release and an acquire fence on top cost 2.5 us per exchange).
// A mailbox has two slots, used in turn: a sender overwrites a message after it has received the
// neighbour's following one, which the neighbour sent when it had read it.  Sequence numbers go on
// from launch to launch (a device word), so an old message is never taken for a new one.  Every wait
// is bounded (ResidentPlan::wait) and a warp that gives up reports kErrTimeout, which ends the others';
// the cooperative launch guarantees that all the blocks run at the same time.
//
// The per-site arithmetic is the one-step kernel's (moments / collide, update_pair for FP32), so every
// form gives the bits of one step per launch.  Accumulating launches store the fields of the
// contour's stencil sites per step into a staging buffer; a flush kernel adds them to the FP64 sums
// in time order afterwards.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "pair32.cuh"
#include "pairdf.cuh"
#include "resident.h"
#include "tma.cuh"

namespace lbmem {

namespace {

constexpr unsigned kFull = 0xffffffffu;

constexpr int MSGS = 2;  // 8-byte forms: 16-byte messages per border site

__device__ __forceinline__ df shfl_from(df v, int d) {  // d = -1: the lane to the left, +1: to the right
    const int src = ((int)threadIdx.x & 31) + d;
    return df(__shfl_sync(kFull, v.hi, src), __shfl_sync(kFull, v.lo, src));
}
template <typename T>
__device__ __forceinline__ T shfl_from(T v, int d) {
    return d < 0 ? __shfl_up_sync(kFull, v, 1) : __shfl_down_sync(kFull, v, 1);
}

// The values one column to the left (right) of this lane's; in: the border value of lane 0 (31).
template <typename T>
__device__ __forceinline__ T from_left(T v, T in, int lane) {
    const T l = shfl_from(v, -1);
    return lane == 0 ? in : l;
}
template <typename T>
__device__ __forceinline__ T from_right(T v, T in, int lane) {
    const T r = shfl_from(v, 1);
    return lane == 31 ? in : r;
}
// The lattice's last column keeps its own value (zero-gradient open edge).
template <typename T>
__device__ __forceinline__ T keep_last(T pulled, T own, bool a_last) { return a_last ? own : pulled; }
__device__ __forceinline__ f2 keep_last(f2 pulled, f2 own, bool a_last, bool b_last) {
    return pack2(a_last ? lo2(own) : lo2(pulled), b_last ? hi2(own) : hi2(pulled));
}

// A lane's values of a row in a state plane (zero outside the lattice).
template <typename T>
__device__ __forceinline__ T load_cols(const T *p, int xa, int nx) { return xa < nx ? p[xa] : T(0); }
__device__ __forceinline__ f2 load_cols(const float *p, int xa, int nx) {
    // xa is even and the pitch a multiple of 32 floats: 8-byte aligned, xa + 1 inside the pitch
    if (xa >= nx) return both(0.f);
    const float2 v = *reinterpret_cast<const float2 *>(p + xa);
    return pack2(v.x, xa + 1 < nx ? v.y : 0.f);
}
template <typename T>
__device__ __forceinline__ void store_cols(T *p, int xa, int nx, T v) {
    if (xa < nx) p[xa] = v;
}
__device__ __forceinline__ void store_cols(float *p, int xa, int nx, f2 v) {
    if (xa + 1 < nx)
        *reinterpret_cast<f2 *>(p + xa) = v;
    else if (xa < nx)
        p[xa] = lo2(v);
}

// ---- messages -----------------------------------------------------------------------------
// One 16-byte access each way.  Every word of a message has to be looked at by its receiver: where a word
// was not, the compiler narrowed the 128-bit load to two smaller ones, between which a message can arrive
// (seen as a value of the message before under the new sequence number).  So whoever takes a message apart
// (from_word, take_pair) uses all of its values, and all_there, get_row, get_site and watch_mail
// compare all of its sequence numbers: a value that is no longer needed must leave the message, not just
// go unused.
struct alignas(16) Msg {
    unsigned long long v, seq;
};
__device__ __forceinline__ Msg msg_load(const Msg *p) {
    Msg m;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(m.v), "=l"(m.seq)
                 : "l"(p)
                 : "memory");
    return m;
}
__device__ __forceinline__ void msg_store(Msg *p, unsigned long long v, unsigned long long seq) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(v),
                 "l"(seq)
                 : "memory");
}
__device__ __forceinline__ unsigned long long word_of(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long word_of(df v) { return pack2(v.hi, v.lo).v; }
// (both words of a message are used: see Msg)
__device__ __forceinline__ void from_word(unsigned long long w, double &v) { v = __longlong_as_double((long long)w); }
__device__ __forceinline__ void from_word(unsigned long long w, df &v) { v = df(lo2(f2{w}), hi2(f2{w})); }

// The two values of a border site (p[0 .. MSGS - 1]).
template <typename T>
__device__ __forceinline__ void send_site(Msg *p, T a, T b, unsigned seq) {
    msg_store(p, word_of(a), seq);
    msg_store(p + 1, word_of(b), seq);
}
// A lane's two values of a border row, in two messages at p[0] and p[32].
template <typename V>
__device__ __forceinline__ void send_row(Msg *p, V a, V b, unsigned seq) {
    msg_store(p, word_of(a), seq);
    msg_store(p + 32, word_of(b), seq);
}
// The same messages in shared memory (the blocks' inboxes).
__device__ __forceinline__ void msg_put(Msg *p, unsigned long long v, unsigned long long seq) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.cta.shared::cta.b128 [%0], t;\n\t}" ::"r"(
                     smem_u32(p)),
                 "l"(v), "l"(seq)
                 : "memory");
}
__device__ __forceinline__ Msg msg_get(const Msg *p) {
    Msg m;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.cta.shared::cta.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(m.v), "=l"(m.seq)
                 : "r"(smem_u32(p))
                 : "memory");
    return m;
}
template <typename T>
__device__ __forceinline__ void put_site(Msg *p, T a, T b, unsigned seq) {
    msg_put(p, word_of(a), seq);
    msg_put(p + 1, word_of(b), seq);
}
// True once the messages of sequence number seq are there (a and b are undefined before).
template <typename T>
__device__ __forceinline__ bool get_site(const Msg *p, T &a, T &b, unsigned seq) {
    const Msg m = msg_get(p), n = msg_get(p + 1);
    from_word(m.v, a);
    from_word(n.v, b);
    return m.seq == seq && n.seq == seq;
}
template <typename V>
__device__ __forceinline__ void put_row(Msg *p, V a, V b, unsigned seq) {
    msg_put(p, word_of(a), seq);
    msg_put(p + 32, word_of(b), seq);
}
template <typename V>
__device__ __forceinline__ bool get_row(const Msg *p, V &a, V &b, unsigned seq) {
    const Msg m = msg_get(p), n = msg_get(p + 32);
    from_word(m.v, a);
    from_word(n.v, b);
    return m.seq == seq && n.seq == seq;
}

// ---- site updates -------------------------------------------------------------------------
// One row of the lane's sites.  rw: what tells a runaway field (a flag, or in FP32 the largest
// |E/3| seen); f3: the fields of the Fourier sums in the form's type when ACC.
template <int POL, bool ACC, typename T>
__device__ __forceinline__ void update_row(Pop<T> &p, const MatT<T> &m, unsigned thr, bool in_lattice, bool &rw, T *f3) {
    bool bad;
    if constexpr (POL == POL_TM) {
        T E3, Hx, Hy, D;
        moments(p, m, &E3, &Hx, &Hy, &D);
        bad = field_runaway(E3, thr);
        if (ACC) {
            f3[0] = D * m.inv_eps;
            f3[1] = Hx;
            f3[2] = Hy;
        }
        collide(p, E3, Hx, Hy);
    } else {
        T Ey3, Ex3, Hz, Dy, Dx;
        moments_te(p, m, &Ey3, &Ex3, &Hz, &Dy, &Dx);
        bad = field_runaway(Ey3, thr) || field_runaway(Ex3, thr);
        if (ACC) {
            f3[0] = Hz;
            f3[1] = Dx * m.inv_eps;
            f3[2] = Dy * m.inv_eps;
        }
        collide_te(p, Ey3, Ex3, Hz);
    }
    rw |= bad && in_lattice;
}

template <typename T>
struct ResidentArgs {
    StepArgs<T> a;
    const T *fin;
    T *fout;
    const long long *t_in;
    long long *t_out;
    int strips, rows, segs, warps, comm, total, ctas, n;
    long long wait;   // clock cycles after which a wait gives up
    Msg *xm, *ym;
    unsigned *ctl;    // [0]: sequence number of the launch's start, [1]: blocks that have finished
    T *stage;
    int n_slots;
};

// Byte offsets of the block's shared memory.
struct ResidentSmem {
    size_t edge, table, src, flags, xin, yin, ids, slots, end;
};
template <typename T>
__host__ __device__ inline ResidentSmem resident_smem(int warps, int rows) {
    ResidentSmem o;
    o.edge = (size_t)warps * rows * NPLANES * 32 * 8;             // state
    o.table = o.edge + (size_t)2 * warps * 4 * 32 * 8;            // border rows, two steps
    o.src = o.table + 256 * sizeof(MatT<T>);
    o.flags = o.src + (size_t)kResidentSteps * 2 * sizeof(T);
    o.xin = o.flags + 2 * kResidentMaxWarps * sizeof(unsigned);
    o.yin = o.xin + (size_t)2 * warps * rows * 2 * MSGS * sizeof(Msg);
    o.ids = o.yin + (size_t)2 * 128 * sizeof(Msg);
    o.slots = o.ids + ((size_t)warps * rows * 32 + 15) / 16 * 16;
    o.end = o.slots + (size_t)warps * rows * 32 * sizeof(int);
    return o;
}

// Flags between the warps of a block: how many of its border rows of one side a warp has published.
__device__ __forceinline__ void flag_set(unsigned *f, unsigned v) {
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(f)), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned flag_get(const unsigned *f) {
    unsigned v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(f)) : "memory");
    return v;
}

// Up to r.wait clock cycles of failed attempts; true: give up (also once another warp has).  All lanes of
// the warp call it together.
struct Patience {
    long long c0 = 0;
    unsigned spin = 0;
    template <typename T>
    __device__ __forceinline__ bool over(const ResidentArgs<T> &r) {
        if (++spin == 1) c0 = clock64();
        if (spin & 63u) return false;
        return __any_sync(kFull, clock64() - c0 > r.wait || (*(const volatile unsigned *)r.a.err & kErrTimeout));
    }
};

// A border row that arrives from the neighbouring segment: through the edge buffer and flag of a warp
// of the same block, through the block's inbox otherwise.
template <typename V>
struct RowLink {
    bool exists, here;
    const unsigned *flag;  // here: the neighbour's count of published rows
    const V *buf;          // here: its edge rows of two steps
    const Msg *box;        // otherwise: the inbox (two slots of 128 messages)
};

// A communication warp (number cw of the block's): each lane watches up to kWatch mailboxes in global
// memory and copies every message that arrives to its place in shared memory (xin, and for the rows
// beyond the block's first and last row y_above, y_below), where the compute warps wait for it.  (A
// compute warp that polled global memory itself waited at least one L2 round trip per step and
// link.)  An inbox has two slots like the mailbox, and a slot is free for the message of step k + 2 when
// that arrives: the neighbour sent it after it had received what this block sent when it had used
// the message of step k.
constexpr int kWatch = 4;
template <typename T>
__device__ void watch_mail(const ResidentArgs<T> &r, unsigned base, int cw, int lane, Msg *xin, int xin_slot,
                           Msg *y_above, Msg *y_below, int yin_slot) {
    const int ny = r.a.ny, first = (int)blockIdx.x * r.warps, warps = min(r.warps, r.total - first);
    const int n_x = warps * r.rows * 2 * MSGS;
    const size_t xslot = (size_t)max(r.strips - 1, 0) * 2 * ny * MSGS, yslot = (size_t)r.ctas * 2 * 64;
    const Msg *src[kWatch];
    Msg *dst[kWatch];
    unsigned left[kWatch];  // messages still to come
    bool is_x[kWatch], any = false;
#pragma unroll
    for (int u = 0; u < kWatch; ++u) {
        int m = (u * r.comm + cw) * 32 + lane;
        src[u] = nullptr, dst[u] = nullptr, left[u] = 0u;
        is_x[u] = m < n_x;
        if (is_x[u]) {
            const int part = m % MSGS, side = m / MSGS % 2, i = m / (2 * MSGS) % r.rows;
            const int g = first + m / (2 * MSGS * r.rows), s = g / r.segs, sg = g - s * r.segs;
            const int y = (int)((long long)sg * ny / r.segs), n = (int)((long long)(sg + 1) * ny / r.segs) - y;
            if (i < n && (side == 0 ? s > 0 : s + 1 < r.strips)) {
                src[u] = r.xm + (((size_t)(side == 0 ? s - 1 : s) * 2 + side) * ny + y + i) * MSGS + part;
                dst[u] = xin + m;
                left[u] = (unsigned)r.n - 1u;
            }
        } else {
            m -= n_x;
            const int sg = (m < 64 ? first : first + warps - 1) % r.segs;
            if (m < 128 && (m < 64 ? sg > 0 : sg + 1 < r.segs)) {
                src[u] = r.ym + (size_t)blockIdx.x * 128 + m;
                dst[u] = m < 64 ? y_above + m : y_below + (m - 64);
                left[u] = (unsigned)r.n - 1u;
            }
        }
        any = any || left[u] > 0u;
    }
    Patience pt;
    while (__any_sync(kFull, any)) {
        Msg m[kWatch];
#pragma unroll
        for (int u = 0; u < kWatch; ++u) {
            const unsigned seq = base + (unsigned)r.n - left[u];
            if (left[u]) m[u] = msg_load(src[u] + (seq & 1u) * (is_x[u] ? xslot : yslot));
        }
        any = false;
        bool got = false;
#pragma unroll
        for (int u = 0; u < kWatch; ++u) {
            const unsigned seq = base + (unsigned)r.n - left[u];
            if (left[u] && m[u].seq == seq) {
                msg_put(dst[u] + (seq & 1u) * (is_x[u] ? xin_slot : yin_slot), m[u].v, m[u].seq);
                --left[u];
                got = true;
            }
            any = any || left[u] > 0u;
        }
        if (__any_sync(kFull, got)) {
            pt.spin = 0;
        } else if (pt.over(r)) {
            if (lane == 0) atomicOr(r.a.err, kErrTimeout);
            return;
        }
    }
}

// The last block to finish moves the sequence on for the next launch (every warp of a block has read
// it before the block's barrier).
template <typename T>
__device__ __forceinline__ void finish_block(const ResidentArgs<T> &r, unsigned base) {
    if (threadIdx.x == 0 && atomicAdd(r.ctl + 1, 1u) == gridDim.x - 1) {
        r.ctl[1] = 0u;
        r.ctl[0] = base + (unsigned)r.n + 2u;
    }
}

// The source values of every step, in blocks that hold column 0 (SRC_NONE: none).
template <typename T>
__device__ __forceinline__ void launch_source(const ResidentArgs<T> &r, long long t0, T *srcv) {
    if (r.a.src.kind == SRC_NONE || (int)blockIdx.x * r.warps >= r.segs) return;
    for (int k = threadIdx.x; k < r.n; k += blockDim.x) {
        double gq = 0.0, inc = 0.0;
        if (t0 + k >= 1) source_values(r.a.src, t0 + k, &gq, &inc);
        srcv[2 * k] = (T)gq;
        srcv[2 * k + 1] = (T)inc;
    }
}

// ---- FP32: overlapped tiles in registers --------------------------------------------------
// A block owns a tile of the lattice and holds it with a halo of H sites on every side where the
// lattice goes on: 64 columns (two per lane) and R rows per warp, 2 x 11 R registers a lane.  For H
// steps the block needs nobody (the halo's valid part shrinks by a site per step); then it publishes
// what lies in its neighbours' halos and receives its own.  Streaming along y inside a warp is a
// renaming of registers, along x four shuffles per row; adjacent warps exchange their border rows
// through shared memory with one block barrier per step.
//
// Why not an exchange per step, as the 8-byte forms do: a message needs about 600 clocks from SM to SM
// on one die and 1000 across the two, and an FP32 step of 30 rows per SM about 900; one exchange
// per step held the 512^2 lattice at 1.9 us per step.
//
// Halo sites travel as messages of three FP32 values and a sequence number (16 bytes, one access), eight
// for the 22 values of a pair of columns, received straight into the registers that need them: no
// fence, no flag and no staging (the same exchange with a release and an acquire fence per block and
// plain copies took 2.5 us against 0.8).  They lie in the two bands that a border is the middle of:
// xm[slot][strip border][row][pair of columns 0 .. H - 1][message] (the first half owned to the left,
// the second to the right) and ym[slot][row border][row 0 .. 2 H - 1][pair of columns of the
// lattice][message]; a tile's corners come with the column bands.  Two slots in turn: a tile
// publishes exchange x + 2 after it has received its neighbours' exchange x + 1, which they sent when
// they had received x.
constexpr int H = kResidentHalo, HP = H / 2, OW = 64 - 2 * H;  // halo, in pairs of columns, columns between halos
struct Resident32Smem {
    size_t src, edge, mats, slots, end;
};
__host__ __device__ inline Resident32Smem resident32_smem(int warps, int rows) {
    Resident32Smem o;
    o.src = 256 * sizeof(MatT<float>);
    o.edge = o.src + (size_t)kResidentSteps * 2 * sizeof(float);
    o.mats = o.edge + (size_t)2 * warps * 4 * 32 * sizeof(f2);
    o.slots = o.mats + (size_t)warps * rows * 4 * 32 * sizeof(f2);
    o.end = o.slots + (size_t)warps * rows * 64 * sizeof(int);
    return o;
}
// Warps per block that the registers of R rows leave room for: a multiple of four, because each
// quarter of the SM has a quarter of the registers (16 warps: 128 a thread, 12: 168).
__host__ __device__ constexpr int resident32_warps(int R) { return R <= 2 ? 16 : R <= 4 ? 12 : 8; }
// First row of tile b of nb: tiles of `height` rows spread evenly from row 0 to row ny - 1, any two
// adjacent ones with 2 H rows or a few more in common.  Tile b > 0 owns rows from its row H on (what it
// holds beyond H rows of halo on a side is computed and never used).
__host__ __device__ inline int tile_row(int b, int nb, int ny, int height) {
    return b == 0 ? 0 : (int)((long long)b * (ny - height) / (nb - 1));
}
// First column of strip s of n: every OW columns, the last one moved left so that it ends with the
// lattice (the right edge is then in lane 31 of every lattice at least 64 wide).
__host__ __device__ inline int strip_col(int s, int n, int nx) {
    return s == 0 ? 0 : s + 1 < n ? s * OW : (nx + 1) / 2 * 2 - 64;
}

constexpr int kHaloMsgs = 8;  // per pair of columns

template <typename F>
__device__ __forceinline__ void each_population(Pop<f2> &p, F f) {
    f(p.ez, 0);
    f(p.epx, 1);
    f(p.emx, 2);
    f(p.epy, 3);
    f(p.emy, 4);
    f(p.hxpx, 5);
    f(p.hxmx, 6);
    f(p.hxz, 7);
    f(p.hypy, 8);
    f(p.hymy, 9);
    f(p.hyz, 10);
}

// The 22 values of a lane's pair of columns as kHaloMsgs messages, and back.
__device__ __forceinline__ void send_pair(Msg *p, int stride, Pop<f2> &s, unsigned seq) {
    float v[24];
    v[22] = v[23] = __uint_as_float(seq);
    each_population(s, [&](f2 &q, int c) { v[2 * c] = lo2(q), v[2 * c + 1] = hi2(q); });
#pragma unroll
    for (int m = 0; m < kHaloMsgs; ++m)
        msg_store(p + m * stride, pack2(v[3 * m], v[3 * m + 1]).v, pack2(v[3 * m + 2], __uint_as_float(seq)).v);
}
__device__ __forceinline__ bool all_there(const Msg *m, unsigned seq) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < kHaloMsgs; ++i) ok = ok && (unsigned)(m[i].seq >> 32) == seq;
    return ok && (unsigned)(m[kHaloMsgs - 1].v >> 32) == seq && (unsigned)m[kHaloMsgs - 1].seq == seq;
}
// (every value of the messages is used: see Msg)
__device__ __forceinline__ void take_pair(const Msg *m, Pop<f2> &s) {
    float v[24];
#pragma unroll
    for (int i = 0; i < kHaloMsgs; ++i)
        v[3 * i] = lo2(f2{m[i].v}), v[3 * i + 1] = hi2(f2{m[i].v}), v[3 * i + 2] = lo2(f2{m[i].seq});
    each_population(s, [&](f2 &q, int c) { q = pack2(v[2 * c], v[2 * c + 1]); });
}

template <int POL, bool ACC, int R>
__global__ void __launch_bounds__(resident32_warps(R) * 32, 1)
    k_resident32(const __grid_constant__ ResidentArgs<float> r) {
    extern __shared__ __align__(16) unsigned char sm[];
    const StepArgs<float> &a = r.a;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int nx = a.nx, ny = a.ny, S = r.strips, NB = r.segs, np = (nx + 1) / 2;
    const Resident32Smem o = resident32_smem(r.warps, R);
    MatT<float> *const table = reinterpret_cast<MatT<float> *>(sm);
    float *const srcv = reinterpret_cast<float *>(sm + o.src);
    f2 *edge = reinterpret_cast<f2 *>(sm + o.edge) + warp * 128 + lane;  // this warp's of the current step
    f2 *const mats = reinterpret_cast<f2 *>(sm + o.mats) + warp * R * 128 + lane;
    int *const slots = reinterpret_cast<int *>(sm + o.slots) + warp * R * 64 + lane * 2;

    const long long t0 = *r.t_in;
    const unsigned base = *(volatile unsigned *)r.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) *r.t_out = t0 + r.n;

    // the tile: 64 columns from xs, height rows from ya; owned columns [own lanes], rows [yo0, yo1)
    const int s = (int)blockIdx.x / NB, b = (int)blockIdx.x - s * NB;
    const bool has_left = s > 0, has_right = s + 1 < S, has_up = b > 0, has_down = b + 1 < NB;
    const int xs = strip_col(s, S, nx), xa = xs + lane * 2;
    const int ls = has_left ? (s * OW - xs) / 2 : 0;  // first lane of the left halo (0 but in the last strip)
    const int height = r.warps * R, ya = tile_row(b, NB, ny, height), ynext = has_down ? tile_row(b + 1, NB, ny, height) : 0;
    const int yo0 = has_up ? ya + H : 0, yo1 = has_down ? ynext + H : ny;
    const int y0 = ya + warp * R;              // this warp's first row
    const bool below = warp + 1 < r.warps;     // another warp's rows follow
    const bool own_lane = (!has_left || lane >= ls + HP) && (has_right ? lane < 32 - HP : xa < nx);
    const size_t ps = a.pstride;

    for (int k = threadIdx.x; k < 256; k += blockDim.x) table[k] = a.mtab[k];
    if (a.src.kind != SRC_NONE && !has_left)
        for (int k = threadIdx.x; k < r.n; k += blockDim.x) {
            double gq = 0.0, inc = 0.0;
            if (t0 + k >= 1) source_values(a.src, t0 + k, &gq, &inc);
            srcv[2 * k] = (float)gq;
            srcv[2 * k + 1] = (float)inc;
        }
    __syncthreads();

    Pop<f2> st[R];
    int id0 = -1;
    bool uniform = true;
    unsigned own_rows = 0u;  // bit i: this lane's sites of row i are owned
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int y = y0 + i;
        const size_t row = (size_t)y * a.pitch;
        each_population(st[i], [&](f2 &v, int c) { v = load_cols(r.fin + c * ps + row, xa, nx); });
        const int ida = xa < nx ? a.mat[row + xa] : -1, idb = xa + 1 < nx ? a.mat[row + xa + 1] : -1;
        if (id0 < 0) id0 = ida;
        uniform = uniform && (ida < 0 || ida == id0) && (idb < 0 || idb == id0);
        const PairMat m = pair_mat(table[max(ida, 0)], table[max(idb, 0)]);
        mats[i * 128] = m.inv3, mats[i * 128 + 32] = m.cd, mats[i * 128 + 64] = m.nc3, mats[i * 128 + 96] = m.inv;
        const bool own = own_lane && y >= yo0 && y < yo1;
        if (own) own_rows |= 1u << i;
        if (ACC) {
            const bool in = own && y >= a.accp.y0 && y <= a.accp.y1;
            slots[i * 64] = in ? a.accp.slot[row + xa] : -1;
            slots[i * 64 + 1] = in && xa + 1 < nx ? a.accp.slot[row + xa + 1] : -1;
        }
    }
    // one material over all of the warp's sites: its constants stay in registers
    const int idw = __reduce_max_sync(kFull, id0);
    uniform = __all_sync(kFull, uniform && (id0 < 0 || id0 == idw)) && idw >= 0;
    PairMat m = pair_mat(table[max(idw, 0)], table[max(idw, 0)]);
    const bool a_last = xa == nx - 1, b_last = xa + 1 == nx - 1;
    const int other = 128 * r.warps;  // to the edges of the next step and back
    int toggle = other;
    float emax = 0.f;  // largest |E/3| seen (field_runaway())
    bool ok = true;

    const bool alone = S * NB == 1;
    const bool to_left = has_left && lane >= ls + HP && lane < ls + 2 * HP, from_left = has_left && lane >= ls && lane < ls + HP;
    const bool to_right = has_right && lane >= 32 - 2 * HP && lane < 32 - HP, from_right = has_right && lane >= 32 - HP;
    const unsigned xm_size = (unsigned)((S - 1) * ny * H * kHaloMsgs), ym_size = (unsigned)((NB - 1) * 2 * H * np * kHaloMsgs);

    edge[0] = st[0].emy, edge[32] = st[0].hymy, edge[64] = st[R - 1].epy, edge[96] = st[R - 1].hypy;
    __syncthreads();
    const int kind = !has_left ? a.src.kind : SRC_NONE;
    for (int k = 0;; ++k) {
        // the pairs from the rows above and below this warp's; at the tile's top and bottom the row's own (the
        // lattice's open edge, or a halo row that no longer counts)
        f2 c0 = st[0].epy, c1 = st[0].hypy, b0 = st[R - 1].emy, b1 = st[R - 1].hymy;
        if (warp > 0) c0 = edge[64 - 128], c1 = edge[96 - 128];
        if (below) b0 = edge[128], b1 = edge[128 + 32];
        const bool on = kind != SRC_NONE && t0 + k >= 1, open = on && kind == SRC_OPEN, hard = on && kind == SRC_HARD;
        float gq = 0.f;  // the source of this step
        if (on) gq = srcv[2 * k + (hard ? 1 : 0)];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            Pop<f2> &q = st[i];
            if (!uniform) {
                m.inv3 = mats[i * 128], m.cd = mats[i * 128 + 32], m.nc3 = mats[i * 128 + 64];
                if (ACC) m.inv = mats[i * 128 + 96];
            }
            const float le = __shfl_up_sync(kFull, hi2(q.epx), 1), lh = __shfl_up_sync(kFull, hi2(q.hxpx), 1);
            const float re = __shfl_down_sync(kFull, lo2(q.emx), 1), rh = __shfl_down_sync(kFull, lo2(q.hxmx), 1);
            f2 epx = pack2(le, lo2(q.epx)), hxpx = pack2(lh, lo2(q.hxpx));
            f2 emx = pack2(hi2(q.emx), re), hxmx = pack2(hi2(q.hxmx), rh);
            if (!has_left) {  // open edge and source at x = 0
                float e = lo2(q.epx), h = lo2(q.hxpx);
                if (open) e = __fadd_rn(e, gq);
                e = hard ? gq : e;
                h = hard ? 0.f : h;
                epx = pack2(lane == 0 ? e : le, lo2(q.epx));
                hxpx = pack2(lane == 0 ? h : lh, lo2(q.hxpx));
            }
            if (!has_right) {  // open edge at x = nx - 1
                emx = keep_last(emx, q.emx, a_last, b_last);
                hxmx = keep_last(hxmx, q.hxmx, a_last, b_last);
            }
            const f2 oe = q.epy, oh = q.hypy;
            q.epx = epx, q.hxpx = hxpx, q.emx = emx, q.hxmx = hxmx;
            q.epy = c0, q.hypy = c1;
            q.emy = i + 1 < R ? st[i + 1 < R ? i + 1 : i].emy : b0;
            q.hymy = i + 1 < R ? st[i + 1 < R ? i + 1 : i].hymy : b1;
            c0 = oe, c1 = oh;
            f2 e3, f3[3];
            update_pair<POL, ACC>(q, m, e3, f3);
            if (!has_right && !(xa + 1 < nx)) e3 = pack2(lo2(e3), 0.f);  // a column outside does not count
            if (own_rows & (1u << i)) emax = amax3(emax, lo2(e3), hi2(e3));
            if constexpr (ACC) {
                const int y = y0 + i;
                if (y >= a.accp.y0 && y <= a.accp.y1) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int sl = slots[i * 64 + c];
                        if (sl >= 0) {
                            float *g = r.stage + (size_t)(3 * k) * r.n_slots + sl;
#pragma unroll
                            for (int j = 0; j < 3; ++j) g[(size_t)j * r.n_slots] = c == 0 ? lo2(f3[j]) : hi2(f3[j]);
                        }
                    }
                }
            }
        }
        if (k + 1 == r.n) break;
        if (((k + 1) & (H - 1)) == 0 && !alone) {
            const unsigned seq = base + (unsigned)((k + 1) / H);
            Msg *const xm = r.xm + (seq & 1u) * xm_size, *const ym = r.ym + (seq & 1u) * ym_size;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int y = y0 + i;
                if (own_rows & (1u << i)) {
                    if (to_left || to_right)
                        send_pair(xm + ((to_left ? s - 1 : s) * ny + y) * kHaloMsgs * H + (to_left ? lane - ls : lane - (32 - 2 * HP)), H,
                                  st[i], seq);
                    if (has_up && y < yo0 + H) send_pair(ym + ((b - 1) * 2 * H + (y - ya)) * kHaloMsgs * np + xa / 2, np, st[i], seq);
                    if (has_down && y >= yo1 - H) send_pair(ym + (b * 2 * H + (y - ynext)) * kHaloMsgs * np + xa / 2, np, st[i], seq);
                }
            }
            // a row's eight messages are in flight together (two rows' at once gained nothing); the rows share
            // one limit, so that a warp that gives up does so after one wait, not after one per row
            Patience pt;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int y = y0 + i;
                const Msg *src = nullptr;
                int stride = np;
                if (!has_down || y < yo1 + H) {  // rows beyond the halo are never used
                    if (from_left || from_right)
                        src = xm + ((from_left ? s - 1 : s) * ny + y) * kHaloMsgs * H + (from_left ? lane - ls : lane - (32 - 2 * HP)), stride = H;
                    else if (own_lane && has_up && y < yo0)
                        src = ym + ((b - 1) * 2 * H + (y - ya)) * kHaloMsgs * np + xa / 2;
                    else if (own_lane && has_down && y >= yo1)
                        src = ym + (b * 2 * H + (y - ynext)) * kHaloMsgs * np + xa / 2;
                }
                bool need = src != nullptr;
                while (__any_sync(kFull, need)) {
                    if (need) {
                        Msg v[kHaloMsgs];
#pragma unroll
                        for (int j = 0; j < kHaloMsgs; ++j) v[j] = msg_load(src + j * stride);
                        if (all_there(v, seq)) {
                            take_pair(v, st[i]);
                            need = false;
                        }
                    }
                    if (pt.over(r)) {
                        ok = false;
                        break;
                    }
                }
            }
        }
        edge += toggle;
        toggle = -toggle;
        edge[0] = st[0].emy, edge[32] = st[0].hymy, edge[64] = st[R - 1].epy, edge[96] = st[R - 1].hypy;
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
    }

    if (!ok) {
        if (threadIdx.x == 0) atomicOr(a.err, kErrTimeout);
    } else {
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (own_rows & (1u << i))
                each_population(st[i], [&](f2 &v, int c) { store_cols(r.fout + c * ps + (size_t)(y0 + i) * a.pitch, xa, nx, v); });
        if (__any_sync(kFull, field_runaway(emax, a.runaway)) && lane == 0) atomicOr(a.err, kErrUnstable);
    }
    finish_block(r, base);
}

// ---- FP64 and double-float: rows in shared memory -----------------------------------------
// Every warp owns a strip of 32 columns and a segment of rows and keeps their populations in shared
// memory.  After every step it sends what crosses its borders, the two populations that move that way
// (streaming has no diagonal): up and down inside a block through an edge buffer and a flag, everything
// else through the mailboxes and the block's communication warps.  No site is computed twice, because
// the FP64 pipe is what bounds it: a FP64 warp instruction occupies a quarter of the SM for 64 clocks
// whatever its active lanes, 28 of them per row make 0.87 us, and a step of the 512^2 lattice needs
// 11.7 us.
template <typename T, int POL, bool ACC>
__global__ void __launch_bounds__(kResidentMaxWarps * 32, 1) k_resident(const __grid_constant__ ResidentArgs<T> r) {
    constexpr int W = 32;
    extern __shared__ __align__(16) unsigned char sm[];
    const StepArgs<T> &a = r.a;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    // This warp's place among the block's segments.  Warps 0, 4, 8, .. run on the same quarter of the SM and
    // share its FP64 pipe, so they take adjacent segments, whose sizes (they alternate where ny is not a
    // multiple of the segments) even out.
    const int per = r.warps >> 2, extra = r.warps & 3, quarter = warp & 3;
    const int loc = warp < r.warps ? quarter * per + min(quarter, extra) + (warp >> 2) : warp;
    const int nx = a.nx, ny = a.ny;
    const ResidentSmem o = resident_smem<T>(r.warps, r.rows);
    T *const st = reinterpret_cast<T *>(sm) + (size_t)loc * r.rows * NPLANES * 32 + lane;
    T *const edge = reinterpret_cast<T *>(sm + o.edge);
    MatT<T> *const table = reinterpret_cast<MatT<T> *>(sm + o.table);
    T *const srcv = reinterpret_cast<T *>(sm + o.src);
    unsigned *const flags = reinterpret_cast<unsigned *>(sm + o.flags);
    uint8_t *const ids = sm + o.ids + (size_t)loc * r.rows * W;
    int *const slots = reinterpret_cast<int *>(sm + o.slots) + (size_t)loc * r.rows * W;

    const long long t0 = *r.t_in;
    const unsigned base = *(volatile unsigned *)r.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) *r.t_out = t0 + r.n;

    // this warp's strip and rows (segment j of a strip starts at row j ny / segs)
    const int g = (int)blockIdx.x * r.warps + loc;
    const bool live = warp < r.warps && g < r.total;  // a compute warp with rows
    const int strip = live ? g / r.segs : 0, seg = live ? g - strip * r.segs : 0;
    const int x0 = strip * W, xa = x0 + lane;
    const int y0 = (int)((long long)seg * ny / r.segs);
    const int nrows = live ? (int)((long long)(seg + 1) * ny / r.segs) - y0 : 0;
    const bool has_left = strip > 0, has_right = strip + 1 < r.strips, has_up = seg > 0, has_down = seg + 1 < r.segs;
    const bool up_here = has_up && loc > 0, down_here = has_down && loc + 1 < r.warps;  // neighbour in this block
    const bool last_column = xa == nx - 1, inside = xa < nx;
    const int kind = a.src.kind;
    const size_t ps = a.pstride;

    // once per launch: material table, the source values of every step, the state, ids and slots
    for (int k = threadIdx.x; k < 256; k += blockDim.x) table[k] = a.mtab[k];
    if (threadIdx.x < 2 * kResidentMaxWarps) flags[threadIdx.x] = 0u;
    launch_source(r, t0, srcv);
    int id0 = -1;
    bool uniform = true;
    for (int i = 0; i < nrows; ++i) {
        const size_t row = (size_t)(y0 + i) * a.pitch;
#pragma unroll
        for (int p = 0; p < NPLANES; ++p) st[(i * NPLANES + p) * 32] = load_cols(r.fin + p * ps + row, xa, nx);
        const uint8_t id = inside ? a.mat[row + xa] : (uint8_t)0;
        ids[i * W + lane] = id;
        if (ACC)
            slots[i * W + lane] = inside && y0 + i >= a.accp.y0 && y0 + i <= a.accp.y1 ? a.accp.slot[row + xa] : -1;
        if (inside) {
            if (id0 < 0) id0 = id;
            uniform = uniform && id == id0;
        }
    }
    // one material over all of the warp's sites: its constants stay in registers
    const int idw = __reduce_max_sync(kFull, id0);
    uniform = __all_sync(kFull, uniform && (id0 < 0 || id0 == idw)) && idw >= 0;

    // Rows are taken downwards in even segments and upwards in odd ones, so that both sides of a
    // border between segments publish and need its rows at the same end of a step: first (A) or
    // last (B).  A border row is then needed about a whole step after it was published.
    const bool down = (seg & 1) == 0;
    // mailboxes: xm[slot][strip border][0: going right, 1: going left][row][message],
    // ym[slot][receiving block][0: from above, 1: from below][message][lane]; inboxes:
    // xin[slot][warp][row][0: from the left, 1: from the right][message], yin[slot][0, 1][message][lane]
    const size_t xslot = (size_t)max(r.strips - 1, 0) * 2 * ny * MSGS, yslot = (size_t)r.ctas * 2 * 64;
    const int xin_slot = r.warps * r.rows * 2 * MSGS;
    Msg *const xin = reinterpret_cast<Msg *>(sm + o.xin), *const yin = reinterpret_cast<Msg *>(sm + o.yin);
    Msg *const my_xin = xin + loc * r.rows * 2 * MSGS;
    const size_t bstep = (size_t)r.warps * 128;
    // nothing has arrived yet for the second step (shared memory holds what an earlier kernel left,
    // perhaps a message of this very number)
    for (int i = threadIdx.x; i < xin_slot; i += blockDim.x) msg_put(xin + ((base + 1u) & 1u) * xin_slot + i, 0ull, base);
    for (int i = threadIdx.x; i < 128; i += blockDim.x) msg_put(yin + ((base + 1u) & 1u) * 128 + i, 0ull, base);
    // what the first step receives, from the input state: as if step -1 had sent it
    if (live) {
        const bool mine = lane == 0 ? has_left : lane == 31 && has_right;
        if (mine)
            for (int i = 0; i < nrows; ++i) {
                const size_t at = (size_t)(y0 + i) * a.pitch + (lane == 0 ? x0 - 1 : x0 + W);
                put_site(my_xin + (base & 1u) * xin_slot + (i * 2 + (lane == 0 ? 0 : 1)) * MSGS,
                            r.fin[(lane == 0 ? P_EPX : P_EMX) * ps + at], r.fin[(lane == 0 ? P_HXPX : P_HXMX) * ps + at],
                            base);
            }
        if (has_up && !up_here) {
            const size_t row = (size_t)(y0 - 1) * a.pitch;
            put_row(yin + (base & 1u) * 128 + lane, load_cols(r.fin + P_EPY * ps + row, xa, nx),
                    load_cols(r.fin + P_HYPY * ps + row, xa, nx), base);
        }
        if (has_down && !down_here) {
            const size_t row = (size_t)(y0 + nrows) * a.pitch;
            put_row(yin + (base & 1u) * 128 + 64 + lane, load_cols(r.fin + P_EMY * ps + row, xa, nx),
                    load_cols(r.fin + P_HYMY * ps + row, xa, nx), base);
        }
        T *const e = edge + bstep + loc * 128 + lane;
        const T *const ql = st + (nrows - 1) * NPLANES * 32;
        e[0] = st[P_EMY * 32], e[32] = st[P_HYMY * 32], e[64] = ql[P_EPY * 32], e[96] = ql[P_HYPY * 32];
    }
    Msg *const x_send = r.xm + (((size_t)(lane == 0 ? strip - 1 : strip) * 2 + (lane == 0 ? 1 : 0)) * ny + y0) * MSGS;
    const bool sends_x = (lane == 0 && has_left) || (lane == 31 && has_right);
    Msg *const up_send = r.ym + ((size_t)blockIdx.x - 1) * 128 + 64 + lane;
    Msg *const down_send = r.ym + ((size_t)blockIdx.x + 1) * 128 + lane;
    const RowLink<T> up{has_up, up_here, flags + 2 * (loc - 1) + 1, edge + ((loc - 1) * 4 + 2) * 32 + lane, yin + lane};
    const RowLink<T> dn{has_down, down_here, flags + 2 * (loc + 1), edge + ((loc + 1) * 4) * 32 + lane,
                        yin + 64 + lane};
    __syncthreads();  // the only block barrier: from here on a warp waits for its neighbours alone

    if (warp >= r.warps) {
        watch_mail<T>(r, base, warp - r.warps, lane, xin, xin_slot, yin, yin + 64, 128);
        return;
    }
    if (!live) return;

    MatT<T> mu{};
    if (uniform) mu = table[idw];
    bool rw = false;  // a runaway field was seen
    const bool waits_x = lane == 0 ? has_left : lane == 31 && has_right;

    // The border row of step k - 1 from a neighbouring segment; false: gave up.
    auto receive = [&](const RowLink<T> &l, int k, T &v, T &h) -> bool {
        Patience pt;
        if (l.here) {
            // by a vote, like every wait here: over() needs all lanes, and each lane's own acquire orders its reads
            while (!__all_sync(kFull, (int)(flag_get(l.flag) - (unsigned)k) >= 0))
                if (pt.over(r)) return false;
            const T *const q = l.buf + ((k + 1) & 1) * bstep;
            v = q[0];
            h = q[32];
            return true;
        }
        const unsigned seq = base + (unsigned)k;
        const Msg *const q = l.box + (seq & 1u) * 128;
        while (!__all_sync(kFull, get_row(q, v, h, seq)))
            if (pt.over(r)) return false;
        return true;
    };

    // All steps of the warp, rows downwards or upwards.  Returns false after a wait gave up.  dir is a
    // constant in FP64, where it is compiled twice, and a value in double-float, whose two copies of the
    // long update would not fit the instruction cache.
    auto steps = [&](auto dir) -> bool {
        const bool DOWN = dir;
        // planes that come from the row taken before (carried) and from the row taken next
        const int PC0 = DOWN ? P_EPY : P_EMY, PC1 = DOWN ? P_HYPY : P_HYMY;
        const int PN0 = DOWN ? P_EMY : P_EPY, PN1 = DOWN ? P_HYMY : P_HYPY;
        const int RS = (DOWN ? 1 : -1) * NPLANES * 32;
        const RowLink<T> &la = DOWN ? up : dn, &lb = DOWN ? dn : up;
        const int ifirst = DOWN ? 0 : nrows - 1;
        for (int k = 0; k < r.n; ++k) {
            const unsigned seq = base + (unsigned)k, so = seq + 1u;
            const bool sends = k + 1 < r.n;
            const bool src_now = strip == 0 && kind != SRC_NONE && t0 + k >= 1, inner = has_left || has_right;
            T *q = st + ifirst * NPLANES * 32;
            // beyond the lattice's top and bottom: the border row's own values (zero-gradient open edge)
            T c0 = q[PC0 * 32], c1 = q[PC1 * 32];
            if (la.exists && !receive(la, k, c0, c1)) return false;
            T *const eout = edge + (k & 1) * bstep + loc * 128 + lane;
            Msg *const xs = x_send + (so & 1u) * xslot;
            // the pair that row i (at w) pulls from the row taken after it; false: gave up
            auto next = [&](const T *w, bool last, T &n0, T &n1) -> bool {
                if (!last) {
                    n0 = w[RS + PN0 * 32], n1 = w[RS + PN1 * 32];
                    return true;
                }
                n0 = w[PN0 * 32], n1 = w[PN1 * 32];
                return !lb.exists || receive(lb, k, n0, n1);
            };
            // row i (at w) pulled from its neighbours, and its own pair carried to the row taken after it
            auto pull = [&](const T *w, int i, T n0, T n1, Pop<T> &p) -> bool {
                // the border values from the left (lane 0) and the right (lane 31)
                T in0{}, in1{};
                if (inner) {
                    const Msg *const xr = my_xin + (seq & 1u) * xin_slot + (i * 2 + (lane == 0 ? 0 : 1)) * MSGS;
                    Patience pt;
                    while (!__all_sync(kFull, !waits_x || get_site<T>(xr, in0, in1, seq)))
                        if (pt.over(r)) return false;
                }
                const T epx = w[P_EPX * 32], emx = w[P_EMX * 32], hxpx = w[P_HXPX * 32], hxmx = w[P_HXMX * 32];
                p.ez = w[P_EZ * 32];
                p.hxz = w[P_HXZ * 32];
                p.hyz = w[P_HYZ * 32];
                p.epy = DOWN ? c0 : n0;
                p.hypy = DOWN ? c1 : n1;
                p.emy = DOWN ? n0 : c0;
                p.hymy = DOWN ? n1 : c1;
                c0 = w[PC0 * 32];
                c1 = w[PC1 * 32];
                if (strip == 0 && lane == 0) in0 = epx, in1 = hxpx;
                p.epx = from_left(epx, in0, lane);
                p.hxpx = from_left(hxpx, in1, lane);
                p.emx = from_right(emx, in0, lane);
                p.hxmx = from_right(hxmx, in1, lane);
                if (!has_right) {
                    p.emx = keep_last(p.emx, emx, last_column);
                    p.hxmx = keep_last(p.hxmx, hxmx, last_column);
                }
                if (src_now && lane == 0) inject_source_t<T>(kind, srcv[2 * k], srcv[2 * k + 1], p);
                return true;
            };
            // the updated row i (to w): its fields staged, its populations kept and sent
            auto put = [&](T *w, int i, const Pop<T> &p, const T *f3) {
                if constexpr (ACC) {
                    const int y = y0 + i;
                    if (y >= a.accp.y0 && y <= a.accp.y1) {
                        const int sl = slots[i * 32 + lane];
                        if (sl >= 0) {
                            T *s = r.stage + (size_t)(3 * k) * r.n_slots + sl;
#pragma unroll
                            for (int jj = 0; jj < 3; ++jj) s[(size_t)jj * r.n_slots] = f3[jj];
                        }
                    }
                }
                w[P_EZ * 32] = p.ez;
                w[P_EPX * 32] = p.epx;
                w[P_EMX * 32] = p.emx;
                w[P_EPY * 32] = p.epy;
                w[P_EMY * 32] = p.emy;
                w[P_HXPX * 32] = p.hxpx;
                w[P_HXMX * 32] = p.hxmx;
                w[P_HXZ * 32] = p.hxz;
                w[P_HYPY * 32] = p.hypy;
                w[P_HYMY * 32] = p.hymy;
                w[P_HYZ * 32] = p.hyz;
                if (!sends) return;
                if (sends_x)
                    send_site(xs + (size_t)i * 2, lane == 0 ? p.emx : p.epx, lane == 0 ? p.hxmx : p.hxpx, so);
                if (i == 0 && has_up) {
                    if (up_here) {
                        eout[0] = p.emy, eout[32] = p.hymy;
                        __syncwarp();
                        if (lane == 0) flag_set(flags + 2 * loc, (unsigned)k + 1u);
                    } else {
                        send_row(up_send + (so & 1u) * yslot, p.emy, p.hymy, so);
                    }
                }
                if (i == nrows - 1 && has_down) {
                    if (down_here) {
                        eout[64] = p.epy, eout[96] = p.hypy;
                        __syncwarp();
                        if (lane == 0) flag_set(flags + 2 * loc + 1, (unsigned)k + 1u);
                    } else {
                        send_row(down_send + (so & 1u) * yslot, p.epy, p.hypy, so);
                    }
                }
            };
            for (int j = 0, i = ifirst; j < nrows; ++j, i += DOWN ? 1 : -1, q += RS) {
                T n0, n1;
                Pop<T> p;
                T f3[3];
                if constexpr (std::is_same<T, df>::value) {
                    // two rows at a time as packed pairs (an odd last one with itself).  The first is sent no
                    // earlier than the second has what it needs of the step before, which waits for
                    // nothing of this step.
                    const bool pair = j + 1 < nrows;
                    const int i2 = pair ? i + (DOWN ? 1 : -1) : i;
                    if (!next(q, !pair, n0, n1) || !pull(q, i, n0, n1, p)) return false;
                    Pop<T> p2 = p;
                    if (pair && (!next(q + RS, j + 2 == nrows, n0, n1) || !pull(q + RS, i2, n0, n1, p2))) return false;
                    Pop<df2> v;
                    df2 g3[3];
                    each_of_pair(v, p, p2, [](df2 &o, df &u, df &w) { o = pack_df(u, w); });
                    rw |= update_pair<POL, ACC>(v, uniform ? mu : table[ids[i * 32 + lane]],
                                                uniform ? mu : table[ids[i2 * 32 + lane]], true, a.runaway, g3) &&
                          inside;
                    each_of_pair(v, p, p2, [](df2 &o, df &u, df &w) { u = first(o), w = second(o); });
                    if (ACC) f3[0] = first(g3[0]), f3[1] = first(g3[1]), f3[2] = first(g3[2]);
                    put(q, i, p, f3);
                    if (!pair) break;
                    if (ACC) f3[0] = second(g3[0]), f3[1] = second(g3[1]), f3[2] = second(g3[2]);
                    put(q + RS, i2, p2, f3);
                    ++j, i = i2, q += RS;
                } else {
                    if (!next(q, j + 1 == nrows, n0, n1) || !pull(q, i, n0, n1, p)) return false;
                    update_row<POL, ACC>(p, uniform ? mu : table[ids[i * 32 + lane]], a.runaway, inside, rw, f3);
                    put(q, i, p, f3);
                }
            }
        }
        return true;
    };
    bool ok;
    if constexpr (std::is_same<T, df>::value)
        ok = steps(down);
    else
        ok = down ? steps(std::true_type{}) : steps(std::false_type{});

    if (!ok) {
        if (lane == 0) atomicOr(a.err, kErrTimeout);
    } else {
        for (int i = 0; i < nrows; ++i) {
            const size_t row = (size_t)(y0 + i) * a.pitch;
#pragma unroll
            for (int p = 0; p < NPLANES; ++p) store_cols(r.fout + p * ps + row, xa, nx, st[(i * NPLANES + p) * 32]);
        }
        if (__any_sync(kFull, rw) && lane == 0) atomicOr(a.err, kErrUnstable);
    }
    finish_block(r, base);
}

// After an accumulating launch of n steps from time *t_in: every slot's staged fields into its
// Fourier sums (Sec. III), in time order, with the one-step kernel's expression.  One thread per
// slot and sum in blocks of one warp: the chain of n FP64 operations per sum bounds it, and a
// quarter of an SM issues one FP64 instruction per 64 clocks, so the warps are spread as far as they
// go (one thread per slot took 27 us for the 96 steps and 600 slots of a 512^2 period, this 7).
template <typename T>
__global__ void k_resident_flush(const T *__restrict__ stage, double *__restrict__ acc, int n_slots, int n,
                                 const double2 *__restrict__ cs, int period, const long long *__restrict__ t_in) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * n_slots) return;
    const int part = i / n_slots, slot = i - part * n_slots;  // part: 2 x component + (0: cos, 1: sin)
    const T *s = stage + (size_t)(part >> 1) * n_slots + slot;
    double *q = acc + 6 * (size_t)slot + part;
    double sum = *q;
    int ph = (int)(*t_in % (long long)period);
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const double2 c = cs[ph];
        if (++ph == period) ph = 0;
        sum += (double)s[(size_t)(3 * k) * n_slots] * ((part & 1) ? c.y : c.x);
    }
    *q = sum;
}

// Whether every tile of this height owns at least H rows and adjacent ones share at least 2 H.
bool owns_enough(int nb, int ny, int height) {
    for (int b = 0; b < nb; ++b) {
        const int y = tile_row(b, nb, ny, height), next = b + 1 < nb ? tile_row(b + 1, nb, ny, height) : 0;
        if (b + 1 < nb && y + height - next < 2 * H) return false;
        const int lo = b > 0 ? y + H : 0, hi = b + 1 < nb ? next + H : ny;
        if (hi - lo < H) return false;
    }
    return true;
}

template <int R>
const void *kernel32(int pol, bool acc) {
    if (pol == POL_TE) return acc ? (const void *)k_resident32<POL_TE, true, R> : (const void *)k_resident32<POL_TE, false, R>;
    return acc ? (const void *)k_resident32<POL_TM, true, R> : (const void *)k_resident32<POL_TM, false, R>;
}

template <typename T>
const void *kernel_of(int pol, bool acc, int rows) {
    if constexpr (std::is_same<T, float>::value) {
        switch (rows) {
            case 1: return kernel32<1>(pol, acc);
            case 2: return kernel32<2>(pol, acc);
            case 4: return kernel32<4>(pol, acc);
            case 5: return kernel32<5>(pol, acc);
            default: return kernel32<7>(pol, acc);
        }
    } else {
        if (pol == POL_TE) return acc ? (const void *)k_resident<T, POL_TE, true> : (const void *)k_resident<T, POL_TE, false>;
        return acc ? (const void *)k_resident<T, POL_TM, true> : (const void *)k_resident<T, POL_TM, false>;
    }
}

// Communication warps for `warps` compute warps of `rows` rows.
int comm_warps(int warps, int rows) {
    return (warps * rows * 2 * MSGS + 128 + 32 * kWatch - 1) / (32 * kWatch);
}

}  // namespace

constexpr size_t kSmemDefault = 48 * 1024;  // dynamic shared memory of a kernel that has not been given more

template <typename T>
cudaError_t resident_plan(int nx, int ny, int pol, ResidentPlan *plan) {
    *plan = ResidentPlan{};
    int dev = 0, sms = 0, coop = 0, smem_max = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess || !coop) return e;
    ResidentPlan p{};
    bool fits = false;
    if (std::is_same<T, float>::value) {
        p.strips = nx <= 64 ? 1 : (nx - 2 * H + 63 - 2 * H) / (64 - 2 * H);
        // as many tiles as SMs, as low as that allows, each owning at least H rows (R = 5 is for lattices of 25 rows
        // too wide for two tiles above one another, which no other height divides: 6000 x 25 takes 1.8
        // us per step, with plain launches 3.1)
        for (int R : {1, 2, 4, 5, 7}) {
            const int most = std::min(sms / std::max(p.strips, 1), resident32_warps(R) * R > 2 * H ? ny / H : 1);
            for (p.segs = most; p.segs >= 1; --p.segs) {
                // the last tile ends with the lattice: height = 2 H + what each owns, a multiple of R
                const int need = p.segs == 1 ? ny : 2 * H + std::max(H, (ny - 2 * H + p.segs - 1) / p.segs);
                p.warps = (need + R - 1) / R;
                const int height = p.warps * R;
                if (p.segs == 1 ? height == ny : height <= ny && owns_enough(p.segs, ny, height)) break;
            }
            p.rows = R;
            fits = p.segs >= 1 && p.warps <= resident32_warps(R);
            if (fits) p.smem = resident32_smem(p.warps, R).end;
            fits = fits && p.smem <= (size_t)smem_max;
            if (fits) break;
        }
        p.total = p.strips * p.segs * p.warps;
    } else {
        // as many warps per block as there are rows of strips per SM, fewer where they do not fit
        p.strips = (nx + 31) / 32;
        const long long units = (long long)p.strips * ny;  // rows of strips
        for (p.warps = (int)std::min<long long>((units + sms - 1) / sms, kResidentMaxWarps - 1); p.warps >= 1 && !fits; --p.warps) {
            p.segs = std::min((int)((long long)sms * p.warps / p.strips), ny);
            if (p.segs < 1) break;
            p.rows = (ny + p.segs - 1) / p.segs;
            p.total = p.strips * p.segs;
            p.comm = comm_warps(p.warps, p.rows);
            p.smem = resident_smem<T>(p.warps, p.rows).end;
            fits = p.warps + p.comm <= kResidentMaxWarps && p.rows <= kResidentMaxRows && p.smem <= (size_t)smem_max;
            if (fits) break;
        }
        // double-float (536 FP32 operations per site) is bound by their latency at the few warps that the
        // registers leave, so with more than one pair of rows per warp the one-step kernel is the faster one
        // (us per step here / there: 256^2 3.7 / 4.7, 320^2 4.0 / 4.8, 384^2 6.3 / 5.6, 512^2 9.0 / 8.0)
        if (std::is_same<T, df>::value && p.rows > 2) fits = false;
    }
    if (!fits) return cudaSuccess;
    p.ctas = (p.total + p.warps - 1) / p.warps;
    p.mail_x = (size_t)(p.strips - 1) * 2 * ny * MSGS;
    size_t mail_y = (size_t)p.ctas * 2 * 64;
    if (std::is_same<T, float>::value) {
        p.mail_x = (size_t)(p.strips - 1) * ny * H * kHaloMsgs;
        mail_y = (size_t)(p.segs - 1) * 2 * H * ((nx + 1) / 2) * kHaloMsgs;
    }
    p.mail_bytes = kControlBytes + 2 * (p.mail_x + mail_y) * sizeof(Msg);
    // (a block of at most the kernel's launch bounds and smem_max always fits an SM)
    for (int acc = 0; acc < 2 && e == cudaSuccess && p.smem > kSmemDefault; ++acc)
        e = cudaFuncSetAttribute(kernel_of<T>(pol, acc != 0, p.rows), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    p.wait = kWaitCycles;
    p.launch = p.ctas;
    if (e == cudaSuccess) *plan = p;
    return e;
}

template <typename T>
cudaError_t launch_resident(const StepArgs<T> &a, const T *fin, T *fout, const long long *t_in, long long *t_out,
                            const ResidentPlan &plan, void *mail, int n, bool accumulate, T *stage, int n_slots,
                            cudaStream_t s) {
    ResidentArgs<T> r{};
    r.a = a;
    r.fin = fin;
    r.fout = fout;
    r.t_in = t_in;
    r.t_out = t_out;
    r.strips = plan.strips;
    r.rows = plan.rows;
    r.segs = plan.segs;
    r.warps = plan.warps;
    r.comm = plan.comm;
    r.total = plan.total;
    r.ctas = plan.ctas;
    r.n = n;
    r.wait = plan.wait;
    r.ctl = (unsigned *)mail;
    r.xm = (Msg *)((char *)mail + kControlBytes);
    r.ym = r.xm + 2 * plan.mail_x;
    r.stage = stage;
    r.n_slots = n_slots;
    void *args[] = {&r};
    cudaError_t e = cudaLaunchCooperativeKernel(kernel_of<T>(a.pol, accumulate, plan.rows), dim3(plan.launch), dim3((plan.warps + plan.comm) * 32),
                                                args, plan.smem, s);
    if (e == cudaSuccess && accumulate && n_slots > 0) {
        k_resident_flush<T><<<(6 * n_slots + 31) / 32, 32, 0, s>>>(stage, a.accp.acc, n_slots, n, a.src.cs, a.src.period,
                                                                 t_in);
        e = cudaGetLastError();
    }
    return e;
}

#define LBMEM_RESIDENT(T)                                                                                            \
    template cudaError_t resident_plan<T>(int, int, int, ResidentPlan *);                                                \
    template cudaError_t launch_resident<T>(const StepArgs<T> &, const T *, T *, const long long *, long long *,     \
                                            const ResidentPlan &, void *, int, bool, T *, int, cudaStream_t);
LBMEM_RESIDENT(float)
LBMEM_RESIDENT(double)
LBMEM_RESIDENT(df)
#undef LBMEM_RESIDENT

}  // namespace lbmem
