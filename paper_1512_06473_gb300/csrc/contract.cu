// contract.cu -- the response of Eq. 5 / Eq. 7 with fp32 table entries, as a
// contraction on the tensor cores.
//
// Summing the look-ups of an output adds <x^(m)(p_s), D^(m)_k> over kernel
// offsets and sub-spaces, which is the dot product of the input patch with
// the row of sub-codewords that the codes select.  A look-up costs one
// shared-memory load per C'_s terms, 32 per SM and clock; the tensor cores
// do 4096 bf16 multiply-adds per SM and clock.  Taken three bf16 pieces per
// operand and the six products of order <= 2 (below), that is 683 fp32-grade
// terms per SM and clock: 170 look-ups at C'_s = 4, 85 at C'_s = 8, against at
// most 27 measured with tables in shared memory.  So where a call has columns
// (positions or images) enough to fill a tile, the sub-codewords are gathered
// once per tile into an operand of the tensor cores and no table is built.
//
// Split.  Every fp32 value v, times 2^16, is b0 + b1 + b2 with b0 = bf16(v), b1 =
// bf16(v - b0) cut off, b2 the rest: 24 bits, the differences exact.  Of the nine
// products of two such sums the six whose pieces' indices add up to at most 2
// are kept; the others are below 2^-24 of the product.  bf16 has fp32's exponent
// range but 16 bits less below its smallest normal number: without the factor the
// last piece of a value below 2^-110 would lose bits (2^-126 would keep eight),
// with it the last bit of a subnormal is one of bf16's.  A sum is divided by 2^32
// where it is rounded for the last time; from 2^96 on (or of values from 2^112
// on) it overflows before, and plain arithmetic takes over (plain_outputs).
//
// Accumulation.  tcgen05.mma adds into fp32 without rounding to nearest, so a
// long accumulation in tensor memory would drift.  Accumulators live there
// for kG steps of 16 terms only: the five small products of those steps are
// added first (while the sum is small), the kG large ones last, then the
// drain warps add the group's sum to fp32 registers with rounded additions,
// while the next group runs in the other half of the accumulator columns.
//
// Tile.  One CTA takes 128 output channels (rows, TMEM lanes) x NT columns.
// Columns are consecutive positions of a padded grid (as in conv.cu: one gap
// of `pad` zero columns between rows, here also `pad` zero rows between
// images), so kernel offset (dy, dx) is a plain shift: the columns' input
// vectors are staged once per 16 channels, K-major without swizzle (16-byte
// rows of 8 channels), and each kernel offset is the same operand at another
// start address.  Stride s: the s^2 phases of the input become channels of a
// stride-1 correlation with ceil(k / s) taps.  FC: the columns are images.
//
// Blocks.  A step contracts 16 terms: four quarters of four, a quarter being a
// sub-codeword of up to four components or half of a longer one, padded with
// zeros (C's 4 and 8 fill their quarters; 3 pads a quarter of the work).
//
// Roles (24 warps, one CTA per SM; registers moved between warpgroups):
//   0-7    gather sub-codewords by code and store them to TMEM as operand A
//          (8 columns per piece and step); one warpgroup per step of an
//          accumulation group;
//   8-9    stage inputs, sub-codebooks and codes in shared memory;
//   10-11  issue the MMAs, one accumulation group each in turn;
//   12-23  add up drained groups, 64 columns per warpgroup; epilogue.
// A warp alone issues an instruction every four to six clocks, and a group of
// 12 MMAs lasts 960 (NT = 160): the roles' inner loops advance by increments,
// without divisions or index arithmetic.  presplit_kernel splits inputs and
// codebooks once per call, into the workspace and in the layouts that the
// main kernel wants, so that staging is bulk copies and the gather only moves
// data.  (Splitting in the staging and gather warps instead saved the launch,
// but was slower from the smallest sizes on: 64x56x56 batch 1 18.5 against
// 14.9 us, AlexNet conv3 batch 128 336 against 151.)
// A from TMEM leaves shared memory's bandwidth to the B operand (6 KB per 96
// clocks at NT = 192, half of it) and the codeword gather.
#define QCNN_UNIT_RECORDS
#include "qcnn_internal.cuh"

#include <algorithm>
#include <climits>
#include <type_traits>

namespace qcnn {

namespace {

constexpr int kG = 2;          // 16-term steps per accumulation group (the MMA issue is written for 2)
constexpr int kGB = 2;         // groups of A operands in TMEM
constexpr int kNTMax = 192;    // columns per tile: two accumulators and A in 512
constexpr int kACols = 24;     // TMEM columns of one step's A: 3 pieces x 8
constexpr int kMT = 128;       // channels per tile
constexpr int kThreads = 768;
constexpr int kStageThreads = 64;  // warps 8-9
constexpr int kWgCols = 64;        // columns of a drain warpgroup
constexpr int kOutPitch = 33;      // ONE: floats from channel to channel of the outputs on their way out
// registers per thread: 6 warpgroups x 80 at launch = 3 x 64 + 3 x 96
constexpr int kRegsRoles = 64, kRegsDrain = 96;
static_assert(3 * kRegsRoles + 3 * kRegsDrain <= 6 * 80, "register pool");
constexpr int kStagesMax = 4;
constexpr size_t kSmemMax = 226 * 1024;  // dynamic
constexpr unsigned kPolls = 1u << 22;  // after which a wait gives up
static_assert(2 * kNTMax + kGB * kG * kACols <= 512, "tensor memory columns");

struct Args {
    const float *x;  // may be the output of the kernel before: coherent loads
    const float *__restrict__ D;
    const uint8_t *__restrict__ codes;
    const float *__restrict__ bias;
    float *y;        // outputs, or partial sums [splits][N][Ct][Ho*Wo]
    int N, Cs, H, W, Ct, kw, stride, pad, Csp, K, M, Ho, Wo, relu;
    int pitch, img, ndx, noff, dymin, dxmin;  // grid geometry
    int nph, mixed;  // stride phases; mixed: a block of 16 spans phases
    int ay[16], ax[16], dy0[16], dy1[16], dx0[16], dx1[16];  // per phase: taps
    // per kind of block (not mixed: its phase; mixed: b mod kinds), the taps
    // that any of its phases has
    int kinds, ry0[16], ry1[16], rx0[16], rx1[16];
    int steps;       // of a unit when splits == 1
    int cbp;         // not mixed: blocks per phase
    int nb;          // blocks
    int kbs;         // blocks per stage
    int n_stages, stages_per_split, splits;
    int S;           // stage buffers
    int NT, n_tiles, m_tiles, units;
    int rows, rpad;  // staged input vectors per block, and their padded count
    int xstage, dstage, cstage;  // bytes per stage buffer
    int taboff;      // mixed: valid quarters per tap [noff], after the codes
    int kstr0, kstr1;  // bytes per sub-codeword of a block's first two pieces
                       // and of its third, all quarters and copies
    int book;          // bytes of a block's codebook: (K + 1) x both
    const uint4 *xpre;  // inputs already split (presplit_kernel)
    const unsigned char *bpre;  // and codebooks, [mixed ? nb : cbp][book]
    long long qr;
    int code_m, code_pk;  // code address = m * code_m + pk * code_pk + ct
    int cbits;       // 0: byte codes, else bit-packed rows
    int crow;        // bytes per staged code row
    int cmis;        // how far a code row begins past the one before, mod 16
                     // (FC byte codes: Ct; else 0)
    int dvec;        // 1: sub-codewords read as float4 (C's 4 and 8)
    int xvec;        // 1: FC rows read as float4
    int early;       // 1: no kernel of this call writes D or the codes
};

// The range of one unit of work: 128 channels x NT columns x a stage range.
struct Unit {
    int mt, nt, q0, st0, st1, split;
};
__device__ __forceinline__ Unit unit_of(const Args &a, int u) {
    Unit r;
    const int t = u / a.m_tiles;  // (neighbouring CTAs share their columns)
    r.mt = u - t * a.m_tiles;
    r.split = t / a.n_tiles;
    r.nt = t - r.split * a.n_tiles;
    r.q0 = r.nt * a.NT;
    r.st0 = r.split * a.stages_per_split;
    r.st1 = min(a.n_stages, r.st0 + a.stages_per_split);
    return r;
}

// Quarters (of four terms) per sub-vector, and sub-vectors per block of 16.
__host__ __device__ constexpr int quarters_of(int csp) { return csp <= 4 ? 1 : 2; }
__host__ __device__ constexpr int block_vectors(int csp) { return 4 / quarters_of(csp); }

// Block b: its phase, first sub-vector (mixed: sub-vector x phase, phases
// innermost) and taps.
struct Blk {
    int ph, t0, y0, y1, x0, x1;
};
__device__ __forceinline__ Blk block_of(const Args &a, int b) {
    const int nv = block_vectors(a.Csp);
    Blk r;
    int kind = 0;
    if (a.mixed) {
        kind = b % a.kinds;
        r.ph = 0;
        r.t0 = b * nv;
    } else {
        if (a.nph > 1) kind = b / a.cbp;
        r.ph = kind;
        r.t0 = (b - kind * a.cbp) * nv;
    }
    r.y0 = a.ry0[kind];
    r.y1 = a.ry1[kind];
    r.x0 = a.rx0[kind];
    r.x1 = a.rx1[kind];
    return r;
}
__device__ __forceinline__ int unit_steps(const Args &a, const Unit &u) {
    if (a.splits == 1) return a.steps;
    const int b0 = u.st0 * a.kbs, b1 = min(a.nb, u.st1 * a.kbs);
    if (a.nph == 1) return (b1 - b0) * a.noff;
    int n = 0;
    for (int b = b0; b < b1; ++b) {
        const Blk k = block_of(a, b);
        n += (k.y1 - k.y0 + 1) * (k.x1 - k.x0 + 1);
    }
    return n;
}
// Barriers and flags of a CTA.
struct Shared {
    uint64_t x_full[kStagesMax], x_empty[kStagesMax];
    uint64_t ready[kGB], a_empty[kGB];  // ready: A written and D drained
    uint64_t d_full[kGB], done[kGB];
    unsigned tmem;
    int give_up;
    int staged[2];  // stages that each staging warp has gone through
};

// Bounded wait of one thread; false when it gave up or another of the CTA did.
__device__ __forceinline__ bool wait_one(Shared &s, uint64_t *bar, unsigned parity) {
    bool ok = mbar_wait_bounded(bar, parity, 64);
    for (unsigned i = 0; i < kPolls / 64 && !ok; ++i) {
        if (*reinterpret_cast<volatile int *>(&s.give_up)) return false;
        ok = mbar_wait_bounded(bar, parity, 64);
    }
    if (!ok) {
        *reinterpret_cast<volatile int *>(&s.give_up) = 1;
        QCNN_RECORD_IF(true, QCNN_CHECK_TIMEOUT);
    }
    return ok;
}
// The same for a whole warp, with one answer.
__device__ __forceinline__ bool wait_warp(Shared &s, uint64_t *bar, unsigned parity) {
    return __all_sync(0xffffffffu, wait_one(s, bar, parity));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
// Asynchronous contiguous copy, 16-byte aligned on both sides; its bytes are
// counted on the mbarrier.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes,
                                          uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
// One arrival when this thread's cp.async copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}

// Three bf16 pieces of two fp32 values (low half: the first), times 2^16.  b0
// rounded to nearest; the difference has at most 16 significant bits, so b1 is its
// upper half cut off and b2 the rest, exactly: b0 + b1 + b2 == 2^16 v.  (b0
// rounded: the signs of b1 and b2, and so of the products left out, are random.)
constexpr float kSplitScale = 65536.f, kSumScale = 1.f / (65536.f * 65536.f);
__device__ __forceinline__ void split3(float v0, float v1, unsigned &p0, unsigned &p1,
                                       unsigned &p2) {
    const float2 m1 = make_float2(-1.f, -1.f);
    v0 *= kSplitScale;
    v1 *= kSplitScale;
    p0 = pack_bf16x2(v0, v1);
    const float2 r = __ffma2_rn(
        make_float2(__uint_as_float(p0 << 16), __uint_as_float(p0 & 0xffff0000u)), m1,
        make_float2(v0, v1));
    const unsigned rx = __float_as_uint(r.x), ry = __float_as_uint(r.y);
    p1 = __byte_perm(rx, ry, 0x7632);
    const float2 s = __ffma2_rn(
        make_float2(__uint_as_float(rx & 0xffff0000u), __uint_as_float(ry & 0xffff0000u)), m1, r);
    p2 = __byte_perm(__float_as_uint(s.x), __float_as_uint(s.y), 0x7632);
}

// kind::f16 with bf16 operands, fp32 accumulators, both K-major, M = 128.
__host__ __device__ constexpr uint32_t idesc_bf16(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}
// One lane of a converged warp, always the same.  (MMAs issued under
// lane == 0 instead took 218 clocks each at any N: the compiler then loops
// over the lanes that might be active.  Issued under this they take N / 2 +
// 10: 106 at N = 192, 74 at 128, with any 16-byte start address.)
__device__ __forceinline__ bool elect_one() {
    unsigned p;
    asm volatile(
        "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(p));
    return p != 0;
}
// D[tmem] (+)= A[tmem] * B[smem], 128 x N x 16, issued by one thread.
__device__ __forceinline__ void mma_bf16_ts(unsigned d, unsigned a, uint64_t b, uint32_t idesc,
                                            bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"((unsigned)accumulate)
        : "memory");
}
// The five products of order 2 and 1 of one step (piece: descriptor units
// between the pieces of B; those of A are 8 columns apart).
__device__ __forceinline__ void issue_small(unsigned d, unsigned a, uint64_t b, uint64_t piece,
                                            uint32_t idesc, bool accumulate) {
    mma_bf16_ts(d, a + 16, b, idesc, accumulate);
    mma_bf16_ts(d, a + 8, b + piece, idesc, true);
    mma_bf16_ts(d, a, b + 2 * piece, idesc, true);
    mma_bf16_ts(d, a + 8, b, idesc, true);
    mma_bf16_ts(d, a, b + piece, idesc, true);
}
// 16 lanes x 8 or 16 columns: thread t has columns 2 (t % 4) and + 1 of each 8
// for lanes t / 4 (r[0], r[1]) and t / 4 + 8 (r[2], r[3]).
__device__ __forceinline__ void tmem_st_16x256(unsigned taddr, unsigned a, unsigned b, unsigned c,
                                               unsigned d) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(taddr),
                 "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void tmem_st_16x256(unsigned taddr, unsigned a, unsigned b, unsigned c,
                                               unsigned d, unsigned e, unsigned f, unsigned g,
                                               unsigned h) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(taddr),
        "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Code of channel ct in sub-space m at kernel offset pk (plain_outputs only).
__device__ unsigned load_code(const Args &a, int m, int pk, int ct) {
    if (a.cbits) {
        const uint8_t *row = a.codes + (size_t)m * a.code_m;
        const int bit = ct * a.cbits;
        unsigned w = row[bit >> 3];
        if ((bit & 7) + a.cbits > 8) w |= (unsigned)row[(bit >> 3) + 1] << 8;
        return (w >> (bit & 7)) & ((1u << a.cbits) - 1u);
    }
    return a.codes[(size_t)m * a.code_m + (size_t)pk * a.code_pk + ct];
}

// A unit's outputs that came out non-finite, again by plain fp32 arithmetic: those
// of a warp's 32 channels (from ch0) x cols columns (from col0), which are NaN in
// memory.  An infinite or NaN input (or one that bf16 rounds to infinity) makes
// NaN of the split products, and a channel padded with zero weights would spread
// it; the look-ups themselves give what this gives: an entry's terms in order,
// then the entries.  A lane has a column, and eight channels at a time, which
// share its inputs.  (Rare, and off everybody's path: a column of 2,304 look-ups
// takes a lane as many times some 1,000 clocks per eight channels.)
template <int CSP>
__device__ __noinline__ void plain_outputs(const Args &a, const Unit &u, int ch0, int col0,
                                           int cols) {
    const int lane = threadIdx.x & 31, HW = a.H * a.W;
    const int ct_end = min(ch0 + 32, a.Ct), b_end = min(a.nb, u.st1 * a.kbs);
    for (int c = lane; c < cols; c += 32) {
        const int q = u.q0 + col0 + c;
        const int n = q / a.img, rem = q - n * a.img;
        const int Y = rem / a.pitch, X = rem - Y * a.pitch;
        if (n >= a.N || Y >= a.Ho || X >= a.Wo) continue;
        const size_t hw = (size_t)a.Ho * a.Wo;
        float *const y = a.y + (((size_t)u.split * a.N + n) * a.Ct) * hw + (size_t)Y * a.Wo + X;
        for (int ct = ch0; ct < ct_end; ct += 8) {
            unsigned left = 0;  // channels to take
            for (int i = 0; i < min(8, ct_end - ct); ++i) {
                const float v = y[(size_t)(ct + i) * hw];
                if (v != v) left |= 1u << i;
            }
            if (!left) continue;
            const unsigned bad = left;
            float acc[8] = {};
            for (int b = u.st0 * a.kbs; b < b_end && left; ++b) {
                const Blk k = block_of(a, b);
                for (int t = k.t0; t < k.t0 + block_vectors(CSP); ++t) {
                    int ph = k.ph, m = t;
                    if (a.mixed) {
                        m = t / a.nph;
                        ph = t - m * a.nph;
                    }
                    if (m >= a.M) break;
                    for (int dy = a.dy0[ph]; dy <= a.dy1[ph]; ++dy)
                        for (int dx = a.dx0[ph]; dx <= a.dx1[ph]; ++dx) {
                            const int iy = (Y + dy + a.dymin) * a.stride + a.ay[ph];
                            const int ix = (X + dx + a.dxmin) * a.stride + a.ax[ph];
                            if (iy < 0 || iy >= a.H || ix < 0 || ix >= a.W) continue;
                            const int pk = ((dy + a.dymin) * a.stride + a.ay[ph] + a.pad) * a.kw +
                                           (dx + a.dxmin) * a.stride + a.ax[ph] + a.pad;
                            const float *x =
                                a.x + ((size_t)n * a.Cs + m * CSP) * HW + (size_t)iy * a.W + ix;
                            float xv[CSP];
#pragma unroll
                            for (int j = 0; j < CSP; ++j) xv[j] = x[(size_t)j * HW];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                if (!(left >> i & 1u)) continue;
                                const int code = min((int)load_code(a, m, pk, ct + i), a.K - 1);
                                const float *d = a.D + ((size_t)m * a.K + code) * CSP;
                                float e = 0.f;
#pragma unroll
                                for (int j = 0; j < CSP; ++j) e = fmaf(xv[j], d[j], e);
                                acc[i] += e;
                                if (acc[i] != acc[i]) left &= ~(1u << i);  // NaN stays NaN
                            }
                        }
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (!(bad >> i & 1u)) continue;
                float v = acc[i];
                if (a.splits == 1) {
                    if (a.bias) v += a.bias[ct + i];
                    if (a.relu) v = fmaxf(v, 0.f);
                }
                y[(size_t)(ct + i) * hw] = v;
            }
        }
    }
}

// A block's codebook: sub-codewords k of its four quarters side by side, as
// [k][copy][quarter] pieces 0 and 1 (16 bytes), then [k][copy][quarter] piece
// 2 (8 bytes); k = K is zero, for sub-vectors that are not there.  Copies so
// that the lanes of a shared-memory load phase (eight for 16 bytes: all
// quarters of two channels; sixteen for 8: of four) meet in no bank whatever
// their codes: without them a load of random 16-byte rows takes 10.4
// wavefronts instead of 4, and the gather as much of the shared memory's time
// as the MMAs' operand.  Item e = (k, quarter) of the block whose first
// sub-vector is t0:
template <int CSP>
__device__ __forceinline__ void book_item(const Args &a, int t0, int e, unsigned char *book) {
    const int quarter = e & 3, k = e >> 2;
    constexpr int QV = quarters_of(CSP);
    int m = t0 + quarter / QV;
    if (a.mixed) m /= a.nph;
    const int j0 = (quarter % QV) * 4;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (m < a.M && k < a.K) {
        const float *s = a.D + ((size_t)m * a.K + k) * CSP + j0;
        if ((CSP == 4 || CSP == 8) && a.dvec) {
            const float4 f = *reinterpret_cast<const float4 *>(s);
            v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + j < CSP) v[j] = s[j];
        }
    }
    uint4 p01;
    uint2 p2;
    split3(v[0], v[1], p01.x, p01.z, p2.x);
    split3(v[2], v[3], p01.y, p01.w, p2.y);
    unsigned char *d = book + (size_t)k * a.kstr0 + quarter * 16;
    for (int c = 0; c < a.kstr0; c += 64) *reinterpret_cast<uint4 *>(d + c) = p01;
    d = book + (size_t)(a.K + 1) * a.kstr0 + (size_t)k * a.kstr1 + quarter * 8;
    for (int c = 0; c < a.kstr1; c += 32) *reinterpret_cast<uint2 *>(d + c) = p2;
}

__device__ __forceinline__ unsigned lds32(unsigned addr) {
    unsigned v;
    asm volatile("ld.shared.b32 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds128(unsigned addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}
__device__ __forceinline__ uint2 lds64(unsigned addr) {
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}

template <int REGS>
__device__ __forceinline__ void regs_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(REGS));
}
template <int REGS>
__device__ __forceinline__ void regs_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(REGS));
}

// A staged row: where its input vector is.
struct RowInfo {
    int base, iy, ix;  // offset of channel 0, coordinates at phase 0
};
__device__ __forceinline__ RowInfo row_info(const Args &a, int q) {
    const int n = q / a.img, rem = q - n * a.img;
    const int Y = rem / a.pitch, X = rem - Y * a.pitch;
    RowInfo r;
    r.iy = (Y + a.dymin) * a.stride;
    r.ix = (X + a.dxmin) * a.stride;
    r.base = n < a.N ? n * a.Cs * a.H * a.W + r.iy * a.W + r.ix : 0;
    if (n >= a.N) r.iy = INT_MIN / 2;  // past the last image: zeros
    return r;
}
// Terms 8 h .. + 7 of a block at a row.
template <int CSP>
__device__ __forceinline__ void load8(const Args &a, const Blk &k, int h, const RowInfo &r,
                                      float (&v)[8]) {
    constexpr int QV = quarters_of(CSP);
    const int HW = a.H * a.W;
    if (!a.mixed) {
        const int iy = r.iy + a.ay[k.ph], ix = r.ix + a.ax[k.ph];
        const bool in = iy >= 0 && iy < a.H && ix >= 0 && ix < a.W;
        const float *src = a.x + (r.base + a.ay[k.ph] * a.W + a.ax[k.ph]);
        if ((CSP == 4 || CSP == 8) && a.xvec) {
            const int c = k.t0 * CSP + h * 8;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 f0 = in && c < a.Cs ? *reinterpret_cast<const float4 *>(src + c) : z;
            const float4 f1 = in && c + 4 < a.Cs ? *reinterpret_cast<const float4 *>(src + c + 4) : z;
            v[0] = f0.x, v[1] = f0.y, v[2] = f0.z, v[3] = f0.w;
            v[4] = f1.x, v[5] = f1.y, v[6] = f1.z, v[7] = f1.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int m = k.t0 + (QV == 1 ? 2 * h + i / 4 : h), j = QV == 1 ? i % 4 : i;
                v[i] = in && j < CSP && m < a.M ? src[(m * CSP + j) * HW] : 0.f;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int t = k.t0 + (QV == 1 ? 2 * h + i / 4 : h), j = QV == 1 ? i % 4 : i;
            const int m = t / a.nph, ph = t - m * a.nph;
            const int iy = r.iy + a.ay[ph], ix = r.ix + a.ax[ph];
            const bool in = j < CSP && m < a.M && iy >= 0 && iy < a.H && ix >= 0 && ix < a.W;
            v[i] = in ? a.x[r.base + (m * CSP + j) * HW + a.ay[ph] * a.W + a.ax[ph]] : 0.f;
        }
    }
}
__device__ __forceinline__ void split8(const float (&v)[8], uint4 &o0, uint4 &o1, uint4 &o2) {
    split3(v[0], v[1], o0.x, o1.x, o2.x);
    split3(v[2], v[3], o0.y, o1.y, o2.y);
    split3(v[4], v[5], o0.z, o1.z, o2.z);
    split3(v[6], v[7], o0.w, o1.w, o2.w);
}

// The inputs' pieces, once per call: xpre[block][piece][half][row][8 bf16], or
// (one tap) xpre[tile][block][piece][half][row of the tile][8 bf16]; and (the
// last blocks) the codebooks'.
template <int CSP>
__global__ void __launch_bounds__(256) presplit_kernel(const __grid_constant__ Args a,
                                                       uint4 *__restrict__ out,
                                                       unsigned char *__restrict__ books) {
    grid_dep_sync();
    const int qb = (int)((a.qr + 255) / 256), xb = qb * 2 * a.nb;  // blocks on inputs
    if ((int)blockIdx.x >= xb) {
        const int per = (a.K + 1) * 4, e = (blockIdx.x - xb) * 256 + threadIdx.x;
        const int b = e / per;
        if (b < (a.mixed ? a.nb : a.cbp))
            book_item<CSP>(a, b * block_vectors(CSP), e - b * per, books + (size_t)b * a.book);
        return;
    }
    const int g = blockIdx.x / qb;  // block and half
    const long long q = (long long)(blockIdx.x - g * qb) * 256 + threadIdx.x;
    if (q >= a.qr) return;
    const RowInfo r = row_info(a, (int)q);
    const Blk k = block_of(a, g >> 1);
    float v[8];
    load8<CSP>(a, k, g & 1, r, v);
    uint4 o0, o1, o2;
    split8(v, o0, o1, o2);
    long long plane = a.qr;
    uint4 *d = out + ((size_t)(g >> 1) * 6 + (g & 1)) * a.qr + q;
    if (a.noff == 1) {  // tiles do not overlap: each one's stages in one piece
        const int nt = (int)q / a.NT;
        plane = a.rpad;
        d = out + (((size_t)nt * a.nb + (g >> 1)) * 6 + (g & 1)) * a.rpad + ((int)q - nt * a.NT);
    }
    d[0] = o0;
    d[2 * plane] = o1;
    d[4 * plane] = o2;
}

// ONE: blocks of a single step (FC layers and 1x1 kernels), two to a stage,
// which is then one accumulation group: every role advances by whole stages.
// (With the general loops these took 1,300 clocks a step whatever was copied:
// the gather warps' path from block to block was the longest of all.)
template <int CSP, bool ONE>
__global__ void __launch_bounds__(kThreads, 1) contract_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (known to be uniform)
    unsigned char *const xs = smem;
    unsigned char *const ds = xs + (size_t)a.S * a.xstage;
    unsigned char *const cs = ds + (size_t)a.S * a.dstage;
    int *const taps = reinterpret_cast<int *>(cs + (size_t)a.S * a.cstage);  // [nph][noff]
    float *const stage_out = reinterpret_cast<float *>(taps + a.nph * a.noff);

    if (tid == 0) {
        for (int i = 0; i < a.S; ++i) {
            // the staging threads' cp.async copies and their other stores; ONE: one
            // warp's, and the thread of the bulk copies
            mbar_init(&sh.x_full[i], ONE ? 65 : 2 * kStageThreads);
            // the MMAs' commits (ONE: of the one warp that uses it) and 8 gather warps
            mbar_init(&sh.x_empty[i], (ONE ? 1 : 2) + 8);
        }
        const int drains = 4 * ((a.NT + kWgCols - 1) / kWgCols);
        for (int i = 0; i < kGB; ++i) {
            mbar_init(&sh.ready[i], 8 + drains);
            mbar_init(&sh.a_empty[i], 1);
            mbar_init(&sh.d_full[i], 1);
            mbar_init(&sh.done[i], 1);
        }
        sh.give_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_async_smem();
    }
    if (warp == 11) tmem_alloc(&sh.tmem, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const unsigned tmem = sh.tmem;
    const unsigned a_col0 = tmem + 2 * kNTMax;
    // (the staging warps wait for the previous kernel after the constants)
    if (!(a.early && (warp == 8 || warp == 9))) grid_dep_sync();

    if (warp < 12) regs_dec<kRegsRoles>();
    else regs_inc<kRegsDrain>();
    if (warp < 8) {
        // ------------------------------------------------ codeword gather
        // This thread has four channels (its warp's 4 (lane / 4) .. + 3, which
        // sit in TMEM lanes lane / 4 + 0, 8, 16, 24) and a quarter of the terms.
        constexpr int QV = quarters_of(CSP), NV = block_vectors(CSP);
        const int quarter = lane & 3, ch = (warp & 3) * 32 + (lane & ~3);
        const bool mine = warp >= 4;  // the step of every group that is this warp's
        const unsigned kmax = (unsigned)(a.K - 1);
        const int noff = a.noff, crow = a.crow, row_skip = a.ndx * crow;
        // the four channels' codes in the code rows of this quarter's
        // sub-vector: a word, or (packed, or rows off the 16-byte alignment)
        // two words and a shift
        const bool two_words = ONE && (a.cbits || a.cmis);
        const int cbits = a.cbits, cshift = (ch * cbits) & 31;
        const unsigned bits = cbits ? (unsigned)cbits : 8u, cmask = (1u << bits) - 1u;
        const unsigned ccol = (unsigned)((quarter / QV) * noff * crow) +
                              (cbits ? (unsigned)(ch * cbits >> 5) * 4 : (unsigned)ch);
        // this lane's place in a sub-codeword, and its copy
        const unsigned kstr0 = (unsigned)a.kstr0, kstr1 = (unsigned)a.kstr1;
        const unsigned off0 = quarter * 16 + ((lane >> 2) * 64 & (kstr0 - 1));
        const unsigned off1 = (unsigned)(a.K + 1) * kstr0 + quarter * 8 + ((lane >> 2) * 32 & (kstr1 - 1));
        const unsigned a_dst = a_col0 + ((unsigned)((warp & 3) * 32) << 16) + (mine ? kACols : 0);
        const unsigned cs_addr = smem_addr(cs), ds_addr = smem_addr(ds);
        // one step: codes at cp (and shift), the block's codebook at book, into A
        // buffer buf
        auto step = [&](unsigned cp, [[maybe_unused]] unsigned shift, unsigned book, bool in,
                        [[maybe_unused]] int ct_left, unsigned buf, unsigned par) -> bool {
            unsigned w = lds32(cp);
            if (two_words) w = __funnelshift_r(w, lds32(cp + 4), shift);
#ifdef QCNN_DEBUG_CHECKS
            for (int j = 0; j < 4; ++j)
                QCNN_CHECK(!in || j >= ct_left || ((w >> (j * bits)) & cmask) <= kmax,
                           QCNN_CHECK_CODE);
#endif
            const unsigned k0 = in ? kstr0 : 0u, k1 = in ? kstr1 : 0u;
            const unsigned r0 = book + off0 + (in ? 0u : (unsigned)a.K * kstr0);
            const unsigned r1 = book + off1 + (in ? 0u : (unsigned)a.K * kstr1);
            uint4 p01[4];
            uint2 p2[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned c = min((w >> (j * bits)) & cmask, kmax);
                p01[j] = lds128(r0 + c * k0);
                p2[j] = lds64(r1 + c * k1);
            }
            if (!wait_warp(sh, &sh.a_empty[buf], par ^ 1)) return false;
            tc_fence_after_sync();
            const unsigned col = a_dst + buf * (kG * kACols);
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // lanes 0-15, 16-31
                const unsigned to = col + ((unsigned)(16 * h) << 16);
                const uint4 &u0 = p01[2 * h], &u1 = p01[2 * h + 1];
                tmem_st_16x256(to, u0.x, u0.y, u1.x, u1.y, u0.z, u0.w, u1.z, u1.w);
                tmem_st_16x256(to + 16, p2[2 * h].x, p2[2 * h].y, p2[2 * h + 1].x,
                               p2[2 * h + 1].y);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive(&sh.ready[buf]);
            return true;
        };
        int slot = 0;
        unsigned spar = 0;  // its use parity
        unsigned g = 0;     // groups so far
        bool ok = true;
        for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
            const Unit un = unit_of(a, u);
            [[maybe_unused]] const int ct_left = a.Ct - (un.mt * kMT + ch);
            if constexpr (ONE) {
                const int bend = min(a.nb, un.st1 * 2);
                const unsigned c1 = ccol + (mine ? (unsigned)(NV * crow) : 0u);
                const unsigned k1 = mine ? (unsigned)a.book : 0u;
                for (int b = un.st0 * 2 + mine; b - mine < bend; b += 2, ++g) {
                    if (!(ok = wait_warp(sh, &sh.x_full[slot], spar))) break;
                    const unsigned buf = g & 1, par = (g >> 1) & 1;
                    if (b < bend) {
                        const int t = b * NV + quarter / QV;
                        const unsigned mis = (unsigned)(t * a.cmis) & 15u;
                        ok = step(cs_addr + (unsigned)(slot * a.cstage) + c1 + (mis & 12u),
                                  cshift + (mis & 3u) * 8, ds_addr + (unsigned)(slot * a.dstage) + k1,
                                  t < a.M, ct_left, buf, par);
                    } else if ((ok = wait_warp(sh, &sh.a_empty[buf], par ^ 1)) && lane == 0) {
                        arrive(&sh.ready[buf]);  // (a last group of one step)
                    }
                    if (!ok) break;
                    __syncwarp();
                    if (lane == 0) arrive(&sh.x_empty[slot]);
                    if (++slot == a.S) {
                        slot = 0;
                        spar ^= 1;
                    }
                }
                continue;
            }
            int left = unit_steps(a, un);
            bool second = false;
            for (int st = un.st0; st < un.st1 && ok; ++st) {
                if (!(ok = wait_warp(sh, &sh.x_full[slot], spar))) break;
                const unsigned cst = cs_addr + (unsigned)(slot * a.cstage);
                const unsigned book = ds_addr + (unsigned)(slot * a.dstage);
                {
                    const Blk k = block_of(a, st);
                    // (a sub-vector past the last: the zero row of the codebook)
                    bool in = a.mixed || k.t0 + quarter / QV < a.M;
                    unsigned cy = cst + ccol + (unsigned)((k.y0 * a.ndx + k.x0) * crow);
                    unsigned vy = cst + (unsigned)(a.taboff + (k.y0 * a.ndx + k.x0) * 4);
                    for (int dy = k.y0; dy <= k.y1 && ok; ++dy, cy += row_skip, vy += a.ndx * 4) {
                        unsigned cp = cy, vp = vy;
                        for (int dx = k.x0; dx <= k.x1; ++dx, cp += crow, vp += 4) {
                            const bool now = second == mine;
                            const unsigned buf = g & 1, par = (g >> 1) & 1;
                            --left;
                            if (second || left == 0) {
                                if (!second && mine) {
                                    // a last group of one step: the other
                                    // warpgroup adds nothing to it (but must not
                                    // arrive in the phase before)
                                    if (!(ok = wait_warp(sh, &sh.a_empty[buf], par ^ 1))) break;
                                    if (lane == 0) arrive(&sh.ready[buf]);
                                }
                                ++g;
                                second = false;
                            } else {
                                second = true;
                            }
                            if (!now) continue;
                            if (a.mixed) in = lds32(vp) >> quarter & 1;
                            if (!(ok = step(cp, 0u, book, in, ct_left, buf, par))) break;
                        }
                    }
                }
                __syncwarp();
                if (ok && lane == 0) arrive(&sh.x_empty[slot]);
                if (++slot == a.S) {
                    slot = 0;
                    spar ^= 1;
                }
            }
        }
    } else if (warp < 10) {
        // ------------------------------------------------------- staging
        constexpr int QV = quarters_of(CSP), NV = block_vectors(CSP);
        const int ptid = tid - 256;
        const int noff = a.noff;
        bool synced = !a.early, ok = true;
        int slot = 0, staged = 0;
        unsigned spar = 0;
        // code copies: per_row pieces of 16 bytes; this thread's piece and first row
        // (ONE: of a warp's 32 threads; a row that may begin inside a piece has
        // one more)
        const int per_row = ONE && a.cbits ? a.cbits : 8 + (ONE && a.cmis ? 1 : 0);
        const int sthread = ONE ? lane : ptid;
        const int r_first = sthread / per_row, q_first = sthread - r_first * per_row;
        const int r_step = (ONE ? 32 : kStageThreads) / per_row;
        // where tap (dy, dx) of each phase is in a sub-space's codes (-1: nowhere)
        for (int e = ptid; e < a.nph * noff; e += kStageThreads) {
            const int ph = e / noff, off = e - ph * noff;
            const int dy = off / a.ndx, dx = off - dy * a.ndx;
            const int pk = ((dy + a.dymin) * a.stride + a.ay[ph] + a.pad) * a.kw +
                           (dx + a.dxmin) * a.stride + a.ax[ph] + a.pad;
            taps[e] = dy >= a.dy0[ph] && dy <= a.dy1[ph] && dx >= a.dx0[ph] && dx <= a.dx1[ph]
                          ? pk * a.code_pk
                          : -1;
        }
        asm volatile("bar.sync 1, 64;\n" ::: "memory");
        for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
            const Unit un = unit_of(a, u);
            // first byte of this channel tile in a code row, and those after its last
            const int width = ONE && a.cbits ? 16 * a.cbits : kMT;
            const int row = a.code_pk ? a.code_pk : a.code_m;
            const int col0 = un.mt * width, col1 = min(col0 + width, row);
            for (int st = un.st0; st < un.st1; ++st) {
                if (!(ok = wait_warp(sh, &sh.x_empty[slot], spar ^ 1))) break;
                if constexpr (ONE) {
                    const int b0 = st * 2, nblk = min(2, a.nb - b0), t0 = b0 * NV;
                    uint64_t *const full = &sh.x_full[slot];
                    if (warp == 8) {  // (the other warp copies the codes meanwhile)
                        if (!synced) {
                            grid_dep_sync();
                            synced = true;
                        }
                        if (elect_one()) {
                            const unsigned bb = (unsigned)(a.book * nblk);
                            const unsigned xb = (unsigned)(nblk * 6 * a.rpad * 16);
                            mbar_expect_tx(full, bb + xb);
                            unsigned char *const book = ds + (size_t)slot * a.dstage;
                            unsigned char *const xd = xs + (size_t)slot * a.xstage;
                            const unsigned char *bs = a.bpre + (size_t)b0 * a.book;
                            const unsigned char *x = reinterpret_cast<const unsigned char *>(
                                a.xpre + ((size_t)un.nt * a.nb + b0) * 6 * a.rpad);
                            bulk_load(xd, x, xb, full);
                            bulk_load(book, bs, bb, full);
                            arrive(full);
                        }
                        __syncwarp();
                        ++staged;
                        if (++slot == a.S) {
                            slot = 0;
                            spar ^= 1;
                        }
                        continue;
                    }
                    // codes: rows of 128 channels, one per sub-vector, in the 16-byte
                    // pieces that have some of them (the last piece of all may be
                    // cut off).  A row of FC byte codes begins anywhere; copied byte by
                    // byte where Ct is no multiple of 16, a stage took 16,000 clocks
                    // (3048 -> 1625, K 128, on 40 images 77.3 us, in pieces 17.4).
                    const int rows = min(t0 + nblk * NV, a.M) - t0;
                    const size_t all = (size_t)a.M * row;
                    unsigned char *const cst = cs + (size_t)slot * a.cstage;
                    if (r_first < r_step)
                        for (int r = r_first; r < rows; r += r_step) {
                            const size_t begin = (size_t)(t0 + r) * row;
                            const size_t at = ((begin + col0) & ~(size_t)15) + q_first * 16;
                            if (at >= begin + col1) continue;
                            const unsigned n = all - at < 16 ? (unsigned)(all - at) : 16u;
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                                             smem_addr(cst + r * a.crow + q_first * 16)),
                                         "l"(a.codes + at), "r"(n)
                                         : "memory");
                        }
                    cp_async_arrive(full);
                    if (!synced) {
                        grid_dep_sync();
                        synced = true;
                    }
                    arrive(full);
                    ++staged;
                    if (++slot == a.S) {
                        slot = 0;
                        spar ^= 1;
                    }
                    continue;
                }
                const Blk k0 = block_of(a, st);
                const int t0 = k0.t0, m0 = a.mixed ? t0 / a.nph : t0;
                const int t1 = min(t0 + NV, a.mixed ? a.M * a.nph : a.M);
                unsigned char *cst = cs + (size_t)slot * a.cstage;
                unsigned char *const book = ds + (size_t)slot * a.dstage;
                uint64_t *const full = &sh.x_full[slot];
                // bulk copies, by one thread and as few as can be (each takes
                // it 50 clocks): codebooks and inputs
                if (warp == 8) {
                    if (elect_one()) {
                        if (!synced) grid_dep_sync();
                        mbar_expect_tx(full, (unsigned)a.book);
                        bulk_load(book, a.bpre + (size_t)(a.mixed ? st : st - k0.ph * a.cbp) * a.book,
                                  (unsigned)a.book, full);
                        unsigned char *d = xs + (size_t)slot * a.xstage;
                        if (noff == 1) {  // the block's image of the tile, in one piece
                            const unsigned bytes = (unsigned)(6 * a.rpad * 16);
                            mbar_expect_tx(full, bytes);
                            bulk_load(d, a.xpre + ((size_t)un.nt * a.nb + st) * 6 * a.rpad, bytes, full);
                        } else {  // its pieces' rows
                            const unsigned bytes = (unsigned)a.rows * 16;
                            const uint4 *s = a.xpre + (size_t)st * 6 * a.qr + un.q0;
                            mbar_expect_tx(full, bytes * 6);
                            for (int i = 0; i < 6; ++i, d += a.rpad * 16, s += a.qr)
                                bulk_load(d, s, bytes, full);
                        }
                    }
                    __syncwarp();
                }
                // codes: one row of 128 channels per (sub-vector, tap)
                const int rows = (t1 - t0) * noff, col = col0 + q_first * 16;
                if (col >= col1) {
                    // (a piece past the last channel)
                } else if (a.nph == 1) {  // rows follow one another
                    const uint8_t *s = a.codes + (size_t)(t0 * noff + r_first) * row + col;
                    unsigned char *d = cst + r_first * a.crow + q_first * 16;
                    const size_t s_step = (size_t)r_step * row;
                    const int d_step = r_step * a.crow;
#pragma unroll 4
                    for (int r = r_first; r < rows; r += r_step, s += s_step, d += d_step)
                        cp_async16(d, s);
                } else {
                    int off = r_first;
                    int m = a.mixed ? m0 : t0, ph = a.mixed ? t0 - m0 * a.nph : k0.ph;
                    unsigned char *d = cst + r_first * a.crow + q_first * 16;
                    for (int r = r_first; r < rows; r += r_step, off += r_step, d += r_step * a.crow) {
                        while (off >= noff) {
                            off -= noff;
                            if (!a.mixed) ++m;
                            else if (++ph == a.nph) {
                                ph = 0;
                                ++m;
                            }
                        }
                        const int tap = taps[ph * noff + off];
                        if (tap >= 0) cp_async16(d, a.codes + (size_t)m * a.code_m + (tap + col));
                    }
                }
                cp_async_arrive(full);
                if (a.mixed) {  // per tap the quarters that have it
                    int *valid = reinterpret_cast<int *>(cst + a.taboff);
                    for (int off = ptid; off < noff; off += kStageThreads) {
                        const int dy = off / a.ndx, dx = off - dy * a.ndx;
                        unsigned w = 0;
                        for (int i = 0; i < 4; ++i) {
                            const int t = t0 + i / QV, m = t / a.nph, ph = t - m * a.nph;
                            if (m < a.M && dy >= a.dy0[ph] && dy <= a.dy1[ph] && dx >= a.dx0[ph] &&
                                dx <= a.dx1[ph])
                                w |= 1u << i;
                        }
                        valid[off] = (int)w;
                    }
                }
                if (!synced) {
                    grid_dep_sync();
                    synced = true;
                }
                arrive(full);
                ++staged;
                if (++slot == a.S) {
                    slot = 0;
                    spar ^= 1;
                }
            }
        }
        if (!synced) grid_dep_sync();
        // The CTA leaves with no copy of its own under way: the last stages' copies
        // are waited for.  (A warp that gave up may be up to S stages short of the
        // other one, whose barriers still need its arrivals to complete.)
        if (lane == 0) sh.staged[warp - 8] = staged;
        asm volatile("bar.sync 1, 64;\n" ::: "memory");
        const int all = max(sh.staged[0], sh.staged[1]);
        for (int i = staged; i < all; ++i) {
            uint64_t *const full = &sh.x_full[i % a.S];
            if (!ONE || warp == 9) {
                arrive(full);
                arrive(full);
            } else if (lane == 0) {
                arrive(full);
            }
        }
        for (int i = max(0, all - a.S); i < all; ++i)
            mbar_wait_bounded(&sh.x_full[i % a.S], (unsigned)(i / a.S) & 1, kPolls);
    } else if (warp >= 12) {
        // -------------------------------------------- group sums, epilogue
        const int wg = (warp - 12) >> 2, quarter = warp & 3;
        const int col0 = wg * kWgCols, cols = min(kWgCols, a.NT - col0);
        if (cols > 0) {
            // (the gather puts channel 4 i + j of a warp's 32 in lane i + 8 j)
            const int chan = 4 * (lane & 7) + (lane >> 3), row = quarter * 32 + chan;
            const unsigned tl = tmem + ((unsigned)(quarter * 32) << 16) + col0;
            // This warp's outputs on their way to memory: [32 channels][pitch].
            // ONE: half of its columns at a time, which leaves room for a third
            // stage buffer (fc6 of 256 images, when clusters shared its copies: 120
            // us with all columns, 108; the others, whose stages last longer, lost
            // 1 to 4% at batch 1 and won as little at the largest).
            const int opitch = ONE ? kOutPitch : cols + 1;
            float *const outb = stage_out + (ONE ? (wg * 4 + quarter) * 32 * kOutPitch
                                                 : kMT * (col0 + wg) + quarter * 32 * opitch);
            const int HoWo = a.Ho * a.Wo;
            // outputs waiting in outb: next channel, channels, and per lane
            // where its columns go (-1: nowhere)
            int prow = 0, prows = 0, po0 = -1;
            [[maybe_unused]] int po1 = -1;
            float *py = a.y;
            // FC: outb goes column by column (image by image), lanes across
            // channels, which are consecutive in memory
            const bool fc = ONE && a.img == 1;
            auto pump = [&](int n) {  // up to n more channels (columns) to memory
                n = min(prows, prow + n);
                if (fc) {
                    for (; prow < n; ++prow)
                        if (po0 >= 0) py[(size_t)prow * a.Ct] = outb[lane * opitch + prow];
                    return;
                }
                for (; prow < n; ++prow) {
                    float *yr = py + (size_t)prow * HoWo;
                    if (po0 >= 0) yr[po0] = outb[prow * opitch + lane];
                    if (!ONE && po1 >= 0) yr[po1] = outb[prow * opitch + 32 + lane];
                }
            };
            // the output offset of column c of a unit's (-1: a gap or past the end)
            auto place = [&](const Unit &un, int c) {
                const int q = un.q0 + col0 + c;
                const int n = q / a.img, rem = q - n * a.img;
                const int Y = rem / a.pitch, X = rem - Y * a.pitch;
                return c < cols && n < a.N && Y < a.Ho && X < a.Wo
                           ? n * a.Ct * HoWo + Y * a.Wo + X
                           : -1;
            };
            unsigned g = 0;  // groups so far
            bool ok = true, redo = false;
            if (lane < kGB) arrive(&sh.ready[lane]);  // empty to begin with
            for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
                const Unit un = unit_of(a, u);
                const int groups = (unit_steps(a, un) + kG - 1) / kG;
                // (the outputs before leave during all but the last groups)
                const int per_group = (32 + max(1, groups - 2) - 1) / max(1, groups - 2);
                float acc[kWgCols];
#pragma unroll
                for (int i = 0; i < kWgCols; ++i) acc[i] = 0.f;
                const int ct = un.mt * kMT + row;
                const bool last = a.splits == 1;
                const float bv = last && a.bias && ct < a.Ct ? a.bias[ct] : 0.f;
                const bool relu = a.relu && last;
                for (int i = 0; i < groups; ++i, ++g) {
                    const unsigned buf = g & 1;
                    if (i + 1 == groups) {
                        pump(32);  // all of the unit before
                        if constexpr (!ONE) {  // (off the path that ends this unit)
                            const int c0 = un.mt * kMT + quarter * 32;
                            prows = min(32, a.Ct - c0);
                            po0 = place(un, lane);
                            po1 = place(un, lane + 32);
                            py = a.y + (size_t)un.split * a.N * a.Ct * HoWo + (size_t)c0 * HoWo;
                            prow = max(0, prows);  // (not there yet)
                        }
                    }
                    if (!(ok = wait_warp(sh, &sh.d_full[buf], (g >> 1) & 1))) break;
                    tc_fence_after_sync();
#pragma unroll
                    for (int c = 0; c < kWgCols; c += 16) {
                        if (c < cols) {
                            float t[16];
                            tmem_ld16(tl + buf * kNTMax + c, t);
#pragma unroll
                            for (int e = 0; e < 16; e += 2)
                                add2(acc[c + e], acc[c + e + 1], t[e], t[e + 1]);
                        }
                    }
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) arrive(&sh.ready[buf]);
                    if (i + 1 < groups) pump(per_group);
                }
                if (!ok) break;
                float *const orow = outb + chan * opitch;
                float2 chk = make_float2(0.f, 0.f);  // NaN if any sum is not finite
#pragma unroll
                for (int e = 0; e < kWgCols; e += 2)
                    chk = __ffma2_rn(make_float2(acc[e], acc[e + 1]), make_float2(0.f, 0.f), chk);
                unsigned bad0 = 0, bad1 = 0;  // columns whose sum is not
                if (!(chk.x + chk.y == 0.f)) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        if (!(fabsf(acc[e]) <= 3.402823466e38f)) bad0 |= 1u << e;
                        if (!(fabsf(acc[e + 32]) <= 3.402823466e38f)) bad1 |= 1u << e;
                    }
                }
                // columns C0 .. C1 - 1 to outb
                auto put = [&](auto C0, auto C1) {
#pragma unroll
                    for (int c = C0; c < C1; c += 16) {
                        if (c < cols) {
#pragma unroll
                            for (int e = c; e < c + 16; e += 2) {
                                const float2 v = __ffma2_rn(make_float2(acc[e], acc[e + 1]),
                                                            make_float2(kSumScale, kSumScale),
                                                            make_float2(bv, bv));
                                orow[e - C0] = relu ? fmaxf(v.x, 0.f) : v.x;
                                orow[e + 1 - C0] = relu ? fmaxf(v.y, 0.f) : v.y;
                            }
                        }
                    }
                    prow = 0;
                    if constexpr (ONE) {
                        const int ch0 = un.mt * kMT + quarter * 32;
                        if (fc) {
                            prows = min(min(cols, a.N - (un.q0 + col0)) - C0, 32);
                            po0 = ch0 + lane < a.Ct ? 0 : -1;
                            py = a.y + ((size_t)un.split * a.N + un.q0 + col0 + C0) * a.Ct + ch0 + lane;
                        } else {
                            prows = min(32, a.Ct - ch0);
                            po0 = place(un, C0 + lane);
                            py = a.y + (size_t)un.split * a.N * a.Ct * HoWo + (size_t)ch0 * HoWo;
                        }
                    }
                };
                if constexpr (ONE) {
                    __syncwarp();  // (the unit before has left outb)
                    put(std::integral_constant<int, 0>(), std::integral_constant<int, 32>());
                    if (cols > 32) {
                        __syncwarp();
                        pump(32);
                        __syncwarp();
                        put(std::integral_constant<int, 32>(), std::integral_constant<int, 64>());
                    }
                } else {
                    put(std::integral_constant<int, 0>(), std::integral_constant<int, 64>());
                }
                redo |= __any_sync(0xffffffffu, (bad0 | bad1) != 0 && ct < a.Ct);
                while ((bad0 | bad1) && ct < a.Ct) {  // (NaN: see plain_outputs)
                    const int c = bad0 ? __ffs((int)bad0) - 1 : __ffs((int)bad1) + 31;
                    if (bad0) bad0 &= bad0 - 1;
                    else bad1 &= bad1 - 1;
                    const float nan = __int_as_float(0x7fffffff);
                    const int o = place(un, c);
                    if (ONE && c < 32 && cols > 32) {  // (has left outb)
                        if (o >= 0) a.y[((size_t)un.split * a.N * a.Ct + ct) * HoWo + o] = nan;
                    } else {
                        orow[ONE ? c & 31 : c] = nan;
                    }
                }
                __syncwarp();
            }
            __syncwarp();
            pump(32);
            // Sums that are not finite, after all else of this CTA: no other warp
            // waits for these, however many they are.
            if (redo && ok) {
                __syncwarp();
                for (int u = blockIdx.x; u < a.units; u += gridDim.x) {
                    const Unit un = unit_of(a, u);
                    plain_outputs<CSP>(a, un, un.mt * kMT + quarter * 32, col0, cols);
                }
            }
        }
    } else {
        // ------------------------------------------------------ MMA issue
        // One thread of each of two warps, which take the accumulation groups
        // in turn: a wait's answer comes back behind the MMAs that the same
        // warp has issued, so a single one left the tensor core idle between
        // groups (1,275 clocks a group of 960).  One barrier covers a group:
        // A written (whose writers have seen the inputs staged) and the
        // accumulator drained.
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16(a.NT);
            const unsigned lbo = (unsigned)a.rpad * 16;
            const uint64_t piece = (uint64_t)(2 * lbo >> 4);  // descriptor units between pieces
            const uint64_t xdesc = smem_desc_kmajor(xs, lbo, 128);
            const unsigned pitch = (unsigned)a.pitch, xunits = (unsigned)a.xstage >> 4;
            const int nb = a.nb, S = a.S;
            int slot = 0;
            unsigned spar = 0;  // its use parity
            unsigned g = 0;     // groups issued
            bool ok = true;
            const unsigned buf = (unsigned)(warp & 1);  // this warp's buffers
            const unsigned dcol = tmem + buf * kNTMax, ac = a_col0 + buf * (kG * kACols);
            static_assert(kGB == 2 && kG == 2, "two warps; two steps");
            auto issue_group = [&](uint64_t d0, uint64_t d1, bool two) {
                tc_fence_after_sync();
                // the small products first, then the large ones
                issue_small(dcol, ac, d0, piece, idesc, false);
                if (two) issue_small(dcol, ac + kACols, d1, piece, idesc, true);
                mma_bf16_ts(dcol, ac, d0, idesc, true);
                if (two) mma_bf16_ts(dcol, ac + kACols, d1, idesc, true);
                mma_commit(&sh.a_empty[buf]);
                mma_commit(&sh.d_full[buf]);
            };
            for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
                const Unit un = unit_of(a, u);
                if constexpr (ONE) {
                    const int bend = min(nb, un.st1 * 2);
                    for (int b = un.st0 * 2; b < bend; b += 2, ++g) {
                        // (only a stage's own warp releases it: an arrival before
                        // the stage is there would count for the use before)
                        if ((g & 1) == buf) {
                            const uint64_t d0 = xdesc + slot * xunits, d1 = d0 + 3 * piece;
                            if (!(ok = wait_one(sh, &sh.ready[buf], (g >> 1) & 1))) break;
                            issue_group(d0, d1, b + 1 < bend);
                            mma_commit(&sh.x_empty[slot]);
                        }
                        if (++slot == S) {
                            slot = 0;
                            spar ^= 1;
                        }
                    }
                    continue;
                }
                int left = unit_steps(a, un);
                // the next step: block (and stage) b, d its B operand (in
                // descriptor units), cx and cy taps left in its row and column
                int b = un.st0;
                Blk k = block_of(a, b);
                unsigned d = slot * xunits + (unsigned)k.y0 * pitch + (unsigned)k.x0;
                int nx = k.x1 - k.x0 + 1, cx = nx, cy = k.y1 - k.y0 + 1;
                unsigned skip = pitch - (unsigned)(nx - 1);
                // stage buffers whose last step has been taken, and their use
                // parities
                unsigned release = 0, parity = 0;
                auto take = [&]() -> uint64_t {
                    const uint64_t r = xdesc + d;
                    if (--cx > 0) {
                        ++d;
                    } else if (--cy > 0) {
                        cx = nx;
                        d += skip;
                    } else {
                        release |= 1u << slot;
                        parity = (parity & ~(1u << slot)) | spar << slot;
                        if (++slot == S) {
                            slot = 0;
                            spar ^= 1;
                        }
                        if (++b < nb) {
                            k = block_of(a, b);
                            nx = k.x1 - k.x0 + 1;
                            cx = nx;
                            cy = k.y1 - k.y0 + 1;
                            skip = pitch - (unsigned)(nx - 1);
                            d = slot * xunits + (unsigned)k.y0 * pitch + (unsigned)k.x0;
                        }
                    }
                    return r;
                };
                for (; left > 0 && ok; left -= kG, ++g) {
                    // a group: two steps, or a last one alone
                    const uint64_t d0 = take();
                    const bool two = left > 1;
                    uint64_t d1 = d0;
                    if (two) d1 = take();
                    const bool mine = (g & 1) == buf;
                    if (mine) {
                        if (!(ok = wait_one(sh, &sh.ready[buf], (g >> 1) & 1))) break;
                        issue_group(d0, d1, two);
                    }
                    while (release) {  // (this warp's MMAs on them have all been issued)
                        const int i = __ffs((int)release) - 1;
                        // (no step of it in this warp's group: see above)
                        if (!mine && !(ok = wait_one(sh, &sh.x_full[i], parity >> i & 1))) break;
                        mma_commit(&sh.x_empty[i]);
                        release &= release - 1;
                    }
                }
            }
            // nothing in flight when the tensor memory is freed
            mma_commit(&sh.done[buf]);
            mbar_wait_bounded(&sh.done[buf], 0, kPolls);
        }
        __syncwarp();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 11) tmem_dealloc(tmem, 512);
}

int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// The s stride phases of one axis: offset t = ky - pad = d * s + p.
struct Axis {
    int n = 0, dmin = 0, nd = 1;
    int p[16], d0[16], d1[16];  // per phase: first and last tap (relative to dmin)
};
bool axis_phases(int k, int s, int pad, Axis *x) {
    bool have[16] = {};
    int lo[16], hi[16];
    if (s > 16) return false;
    int dmin = INT_MAX, dmax = INT_MIN;
    for (int t = 0; t < k; ++t) {
        const int d = floor_div(t - pad, s), p = t - pad - d * s;
        if (!have[p]) lo[p] = hi[p] = d;
        have[p] = true;
        lo[p] = std::min(lo[p], d);
        hi[p] = std::max(hi[p], d);
        dmin = std::min(dmin, d);
        dmax = std::max(dmax, d);
    }
    x->dmin = dmin;
    x->nd = dmax - dmin + 1;
    for (int p = 0; p < s; ++p)
        if (have[p]) {
            x->p[x->n] = p;
            x->d0[x->n] = lo[p] - dmin;
            x->d1[x->n++] = hi[p] - dmin;
        }
    return true;
}
// Cells from one row (image) of the padded grid to the next: all that the
// taps reach, or fewer where what they reach past the end is zero and so are
// the first cells of the next row.
int axis_pitch(int in, int out, int s, const Axis &x) {
    const int zeros = -x.dmin;                    // leading zero cells
    const int reach = out + x.nd - 1;             // cells read
    const int shared = std::max({out, cdiv(in, s) + zeros, reach - zeros});
    return std::min(reach, shared);
}

}  // namespace

struct ContractFns {
    void (*main)(Args);
    void (*pre)(Args, uint4 *, unsigned char *);
};
template <bool ONE>
static ContractFns contract_fns_of(int csp) {
    switch (csp) {
        case 1: return {contract_kernel<1, ONE>, presplit_kernel<1>};
        case 2: return {contract_kernel<2, ONE>, presplit_kernel<2>};
        case 3: return {contract_kernel<3, ONE>, presplit_kernel<3>};
        case 4: return {contract_kernel<4, ONE>, presplit_kernel<4>};
        case 5: return {contract_kernel<5, ONE>, presplit_kernel<5>};
        case 6: return {contract_kernel<6, ONE>, presplit_kernel<6>};
        case 7: return {contract_kernel<7, ONE>, presplit_kernel<7>};
        default: return {contract_kernel<8, ONE>, presplit_kernel<8>};
    }
}
static ContractFns contract_fns(int csp, bool one) {
    return one ? contract_fns_of<true>(csp) : contract_fns_of<false>(csp);
}

ContractPlan plan_contract(const ConvShape &s, int min_splits) {
    ContractPlan best;
    if (s.bf16) return best;
    Axis ya, xa;
    if (!axis_phases(s.kh, s.stride, s.pad, &ya) || !axis_phases(s.kw, s.stride, s.pad, &xa))
        return best;
    const int nph = ya.n * xa.n;
    if (nph > 16) return best;
    const long long pitch = axis_pitch(s.W, s.Wo, s.stride, xa);
    const long long rows_img = axis_pitch(s.H, s.Ho, s.stride, ya);
    const long long img = pitch * rows_img;
    const long long Q = (s.N - 1) * img + (s.Ho - 1) * pitch + s.Wo;
    const long long reach = (ya.nd - 1) * pitch + xa.nd - 1;
    if (Q >= (1ll << 30) || reach > 4096) return best;
    const int noff = ya.nd * xa.nd;
    // channel order of strided layers: one phase per block of 16 channels
    // (taps that a phase lacks are skipped), or sub-vector by sub-vector with
    // the phases innermost (no padding of few channels to 16)
    long long pure = 0;
    const int NV = block_vectors(s.Csp), cbp = cdiv(s.M, NV);
    for (int y = 0; y < ya.n; ++y)
        for (int x = 0; x < xa.n; ++x)
            pure += (long long)cbp * (ya.d1[y] - ya.d0[y] + 1) * (xa.d1[x] - xa.d0[x] + 1);
    // (mixed: a block has the taps that any of its phases has)
    const int nbm = cdiv(s.M * nph, NV);
    long long mix = 0;
    for (int b = 0; b < nbm; ++b) {
        int y0 = INT_MAX, y1 = 0, x0 = INT_MAX, x1 = 0;
        for (int i = 0; i < NV; ++i) {
            const int ph = (b * NV + i) % nph, yi = ph / xa.n, xi = ph % xa.n;
            y0 = std::min(y0, ya.d0[yi]);
            y1 = std::max(y1, ya.d1[yi]);
            x0 = std::min(x0, xa.d0[xi]);
            x1 = std::max(x1, xa.d1[xi]);
        }
        mix += (y1 - y0 + 1) * (x1 - x0 + 1);
        if (mix >= pure) break;
    }
    const int mixed = nph > 1 && mix < pure;
    const long long steps = mixed ? mix : pure;
    const int nb = mixed ? nbm : cbp * nph;
    // (144: rows of successive sub-vectors start in different banks; room for
    // packed rows of 8 bits, so that both kinds of codes make the same plan)
    const int crow = 144;
    const int m_tiles = cdiv(s.Ct, kMT);
    const int sms = num_sms();
    // several blocks per stage where a block is a single step
    const int kbs = noff == 1 && nph == 1 ? 2 : 1;
    const int n_stages = cdiv(nb, kbs);
    const size_t taboff = align_up((size_t)kbs * NV * noff * crow, 16);
    const size_t cstage = align_up(taboff + (mixed ? (size_t)noff * 4 : 0), 16);
    const int nt_hi = (int)std::min<long long>(kNTMax, (Q + 15) / 16 * 16);
    for (int NT = 16; NT <= nt_hi; NT += 16) {
        const int rows = NT + (int)reach;
        int rpad = rows;
        while (rpad % 8 != 1) ++rpad;  // staged FC rows then store without conflicts
        const size_t xstage = (size_t)kbs * 6 * rpad * 16;
        const size_t outs = kbs > 1 ? (size_t)cdiv(NT, kWgCols) * kOutPitch : NT + 3;
        const size_t fixed = (size_t)nph * noff * 4 + outs * kMT * 4;
        // as many copies in the codebooks as let two stage buffers fit
        static const int copies[3][2] = {{2, 4}, {2, 2}, {1, 1}};
        size_t kstr0 = 0, kstr1 = 0, stage = 0;
        for (const auto &c : copies) {
            kstr0 = 64 * c[0];
            kstr1 = 32 * c[1];
            stage = xstage + kbs * (s.K + 1) * (kstr0 + kstr1) + cstage;
            if (fixed + 2 * stage <= kSmemMax) break;
        }
        int S = kStagesMax;
        while (S > 2 && fixed + S * stage > kSmemMax) --S;
        if (fixed + S * stage > kSmemMax || (rpad * 16) >> 4 > 0x3FFF) continue;
        const int n_tiles = cdiv((int)Q, NT);
        const long long tiles = (long long)n_tiles * m_tiles;
        if (tiles > (1 << 24)) continue;
        // (a stage's bytes at 20 per clock and SM, the L2's rate when all SMs read)
        const double bytes = (double)xstage + kbs * (s.K + 1) * (kstr0 + kstr1) + cstage;
        const double per_step = std::max({3.0 * NT + 60.0, 450.0, bytes / 20.0 / (kbs > 1 ? kbs : noff)});
        for (int sp = min_splits; sp <= std::min(n_stages, 64); ++sp) {
            const int sps = cdiv(n_stages, sp);
            if (cdiv(n_stages, sps) != sp) continue;
            const long long units = tiles * sp;
            const double waves = (double)((units + sms - 1) / sms);
            const double part = sp > 1 ? 2.0 * sp * s.N * s.Ct * s.Ho * s.Wo * 4.0 / 3000.0 + 5000.0 : 0.0;
            const double score = waves * ((double)steps * sps / n_stages * per_step + 2500.0) + part;
            if (best.ok && score >= best.score) continue;
            // (inputs past a scratch of 2 GB, or a grid past 2^30: the tables)
            const long long qr = (long long)n_tiles * NT + reach;
            const long long pre = (long long)nb * 96 * (noff == 1 ? (long long)n_tiles * rpad : qr);
            if (pre > (2ll << 30) || (qr + 255) / 256 * 2 * nb > (1ll << 30)) continue;
            best.ok = true;
            best.score = score;
            best.NT = NT;
            best.splits = sp;
            best.stages_per_split = sps;
            best.S = S;
            best.rows = rows;
            best.rpad = rpad;
            best.xstage = (int)xstage;
            best.kstr0 = (int)kstr0;
            best.kstr1 = (int)kstr1;
            best.smem = fixed + S * stage;
            best.n_tiles = n_tiles;
            best.units = (int)units;
            best.ctas = (int)std::min<long long>(units, sms);
            best.qr = qr;
            best.pre_bytes = align_up((size_t)pre, kWsAlign);
            best.book_bytes = (size_t)(mixed ? nb : cbp) * (s.K + 1) * (kstr0 + kstr1);
            best.partial_bytes = sp > 1 ? (size_t)sp * s.N * s.Ct * s.Ho * s.Wo * sizeof(float) : 0;
        }
    }
    best.taboff = (int)taboff;
    best.scratch = align_up(best.pre_bytes + best.book_bytes, kWsAlign) +
                   align_up(best.partial_bytes, kWsAlign);
    best.steps = (int)steps;
    best.mixed = mixed;
    best.kbs = kbs;
    best.nb = nb;
    best.n_stages = n_stages;
    best.m_tiles = m_tiles;
    best.cstage = (int)cstage;
    best.crow = crow;
    return best;
}

qcnn_status launch_contract(const ConvShape &s, const ContractPlan &p, const float *x,
                            const float *D, const uint8_t *codes, FcCodes fc, const float *bias,
                            float *y, int relu, void *ws, cudaStream_t st, bool early,
                            bool leave_partials) {
    float *partial_ws = reinterpret_cast<float *>(ws);
    uint4 *pre_ws = reinterpret_cast<uint4 *>(static_cast<uint8_t *>(ws) +
                                              align_up(p.partial_bytes, kWsAlign));
    Axis ya, xa;
    if (!axis_phases(s.kh, s.stride, s.pad, &ya) || !axis_phases(s.kw, s.stride, s.pad, &xa))
        return QCNN_ERR_UNSUPPORTED;
    Args a = {};
    a.x = x;
    a.D = D;
    a.codes = codes;
    a.bias = p.splits > 1 ? nullptr : bias;
    a.y = p.splits > 1 ? partial_ws : y;
    a.N = s.N;
    a.Cs = s.Cs;
    a.H = s.H;
    a.W = s.W;
    a.Ct = s.Ct;
    a.kw = s.kw;
    a.stride = s.stride;
    a.pad = s.pad;
    a.Csp = s.Csp;
    a.K = s.K;
    a.M = s.M;
    a.Ho = s.Ho;
    a.Wo = s.Wo;
    a.relu = relu;
    a.pitch = axis_pitch(s.W, s.Wo, s.stride, xa);
    a.img = a.pitch * axis_pitch(s.H, s.Ho, s.stride, ya);
    a.ndx = xa.nd;
    a.noff = ya.nd * xa.nd;
    a.dymin = ya.dmin;
    a.dxmin = xa.dmin;
    a.nph = 0;
    for (int yi = 0; yi < ya.n; ++yi)
        for (int xi = 0; xi < xa.n; ++xi) {
            const int i = a.nph++;
            a.ay[i] = ya.p[yi];
            a.ax[i] = xa.p[xi];
            a.dy0[i] = ya.d0[yi];
            a.dy1[i] = ya.d1[yi];
            a.dx0[i] = xa.d0[xi];
            a.dx1[i] = xa.d1[xi];
        }
    a.mixed = p.mixed;
    a.steps = p.steps;
    const int NV = block_vectors(s.Csp);
    // (blocks NV sub-vectors apart repeat their phases after nph blocks at most)
    a.kinds = a.nph;
    for (int k = 0; k < a.nph; ++k) {
        a.ry0[k] = a.rx0[k] = INT_MAX;
        a.ry1[k] = a.rx1[k] = 0;
        for (int i = 0; i < (p.mixed ? NV : 1); ++i) {
            const int ph = p.mixed ? (k * NV + i) % a.nph : k;
            a.ry0[k] = std::min(a.ry0[k], a.dy0[ph]);
            a.ry1[k] = std::max(a.ry1[k], a.dy1[ph]);
            a.rx0[k] = std::min(a.rx0[k], a.dx0[ph]);
            a.rx1[k] = std::max(a.rx1[k], a.dx1[ph]);
        }
    }
    a.cbp = cdiv(s.M, block_vectors(s.Csp));
    a.nb = p.nb;
    a.kbs = p.kbs;
    a.n_stages = p.n_stages;
    a.stages_per_split = p.stages_per_split;
    a.splits = p.splits;
    a.S = p.S;
    a.NT = p.NT;
    a.n_tiles = p.n_tiles;
    a.m_tiles = p.m_tiles;
    a.units = p.units;
    a.rows = p.rows;
    a.rpad = p.rpad;
    a.xstage = p.xstage;
    a.kstr0 = p.kstr0;
    a.kstr1 = p.kstr1;
    a.book = (s.K + 1) * (p.kstr0 + p.kstr1);
    a.dstage = p.kbs * a.book;
    a.cstage = p.cstage;
    a.taboff = p.taboff;
    a.qr = p.qr;
    unsigned char *book_ws = reinterpret_cast<unsigned char *>(pre_ws) + p.pre_bytes;
    a.xpre = pre_ws;
    a.bpre = book_ws;
    a.cbits = fc.bits;
    a.crow = p.crow;
    if (fc.bits) {
        a.code_m = (int)fc_packed_pitch(s.Ct, s.K);
    } else if (fc.yes) {
        a.code_m = s.Ct;
        a.cmis = s.Ct & 15;
    } else {
        a.code_pk = packed_ct(s.Ct);
        a.code_m = s.kh * s.kw * a.code_pk;
    }
    a.dvec = reinterpret_cast<uintptr_t>(D) % 16 == 0;
    a.xvec = s.H * s.W == 1 && s.Cs % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
    a.early = early ? 1 : 0;
    const ContractFns fn = contract_fns(s.Csp, p.kbs > 1);
    qcnn_status rc = allow_smem(reinterpret_cast<const void *>(fn.main));
    if (rc != QCNN_OK) return rc;
    const long long xb = (p.qr + 255) / 256 * 2 * p.nb;
    const long long books = (long long)(p.mixed ? p.nb : a.cbp) * (s.K + 1) * 4;
    rc = launch_pdl(fn.pre, dim3((unsigned)(xb + (books + 255) / 256)), dim3(256), 0, st, a, pre_ws,
                    book_ws);
    if (rc != QCNN_OK) return rc;
    rc = launch_pdl(fn.main, dim3(p.ctas), dim3(kThreads), p.smem, st, a);
    if (rc != QCNN_OK || p.splits == 1 || leave_partials) return rc;
    return launch_split_reduce(partial_ws, p.splits, (size_t)s.N * s.Ct * s.Ho * s.Wo, s.Ct,
                               s.Ho * s.Wo, bias, relu, y, st, true);
}

}  // namespace qcnn
