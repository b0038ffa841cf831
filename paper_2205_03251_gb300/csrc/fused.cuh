// Fused interpreter: a run of prefix-ordered nodes is first decoded, 128
// nodes at a time by the whole warp, into a short list of instructions, and
// the list is then executed with lanes as test cases.
//
// A scan of prefix order from right to left needs a stack only for operands
// that are values of whole subtrees.  Four forms of instruction cover it (f
// a function, L a leaf, acc the running value, i.e. that of the subtree to
// the right):
//   f L L    push acc; acc = f(L, L)
//   f L .    acc = f(L, acc)       the left operand is a leaf, the right one was just evaluated
//   f f ..   acc = f(acc, pop)     the left operand was just evaluated
//   f g L L  acc = f(g(L, L), acc) Boolean sets: the left operand has two leaves; neither a push nor a pop
//   L        push acc; acc = L     a leaf that no function to its left takes at once
// A node's form depends on its own opcode and its two neighbours' on either
// side, so 32 lanes decode 128 nodes with a few byte-parallel operations
// each, and leaves -- half of all nodes -- mostly cost no instruction of
// their own.  Every opcode is still applied to every test case, to the same
// operands in the same order: the values are the same bits.
//
// Stack depth: B(q), the number of complete subtrees in [q, end), bounds the
// number of entries between two instructions (one of them the initial
// running value).  The decoder knows it, so the executor has no checks: the
// window of W entries in shared memory slides over the stack from chunk to
// chunk (entries below it in a global overflow area), and a chunk of 128
// nodes whose depths span more than the window runs on the global area alone.
// A malformed run has B below 1 after one of its nodes, or not 1 at its
// start.  The first is found as the chunk with that node is decoded: chunks to
// its right have run by then, that one does not, so nothing leaves the stack.
#pragma once
#include "interp.cuh"

#define FX_CHUNK 128                       // nodes decoded at a time: one 32-bit word per lane
#define FX_CODE_WORDS (FX_CHUNK + 2)       // instructions of a chunk, the end mark, and one read ahead
#define FX_CODE_BYTES (FX_CODE_WORDS * 8)
#define FX_EXIT 30u
#define FX_BROWS 16u                       // rows of the Boolean leaf table (opcodes 4..14 are inputs)

// Instruction index: the function in the order + - * /, the leaf kinds x and
// constant (binary32 and integer sets), or any input (Boolean sets, whose
// leaves all come from one table).  FX_EXIT ends a list.
//   0..15  f L L: 4 f + 2 (left is a constant) + (right is a constant)
//   16..23 f L .: 16 + 2 f + (left is a constant)
//   24..27 f f ..: 24 + f
//   28, 29 L: 28 + (it is a constant)
//   32..95 f g L L (Boolean): 32 + 16 f + 4 g + 3
// Boolean: the constant bits are all set.
//
// f g L L saves the Boolean sets, whose leaves are all of one kind, a dispatch
// and a round trip through the stack for 16 more pieces of code (full
// evaluation of 29.6 M nodes of the 11-multiplexer set 1.71 -> 1.58 ms).  The
// other sets would need 48 more, whose instruction fetches cost more than the
// dispatches they save: 0.5 GB of binary32 trees 9.0 -> 14.5 ms, 29 M nodes
// of integer trees 1.77 -> 1.97 ms.  (And a paired product followed by a paired sum
// in one piece of code is joined into one rounding by the assembler, also
// with .rn on both: 22 % of random triples differ.)

__device__ __forceinline__ uint32_t fx_signs(uint32_t v) {      // each byte all ones or zeros by its top bit
    uint32_t r;
    asm("prmt.b32 %0, %1, %1, 0xBA98;" : "=r"(r) : "r"(v));
    return r;
}
// 0xFF in every byte of t that is zero
__device__ __forceinline__ uint32_t fx_zero_bytes(uint32_t t) {
    return fx_signs(~(((t & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | t));
}
// 0xFF in every byte of w that is a function (opcode below 4)
__device__ __forceinline__ uint32_t fx_funcs(uint32_t w) { return fx_zero_bytes(w & 0xFCFCFCFCu); }

__device__ __forceinline__ void fx_sts(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v)); }
// instruction `idx` at the list address `at` and its operand one word on, if `on` is not zero (predicated: no branch)
__device__ __forceinline__ void fx_put(uint32_t on, uint32_t at, uint32_t idx, uint32_t y) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u32 [%1], %2;\n\t@p st.shared.u32 [%1+12], %3;\n\t}"
                 ::"r"(on), "r"(at), "r"(idx), "r"(y));
}

// The lane's word of a chunk: bytes [q, q + 4) of the run [s, e), positions
// outside the run replaced by 0xFF (a leaf).  `ld(q)` reads the word at q, a
// multiple of 4; it is not called for a word without a node of the run.
template <typename LD>
__device__ __forceinline__ uint32_t fx_word(LD ld, int32_t q, uint32_t s, uint32_t e) {
    if (q >= (int32_t)e || q + 4 <= (int32_t)s) return 0xFFFFFFFFu;
    uint32_t w = ld((uint32_t)q);
    if (q < (int32_t)s) w |= 0xFFFFFFFFu >> (32 - 8 * (s - (uint32_t)q));
    if (q + 4 > (int32_t)e) w |= 0xFFFFFFFFu << (8 * (e - (uint32_t)q));
    return w;
}

// What the decoder carries from one chunk to the next (right to left).
struct FxCarry {
    uint32_t w, f;       // this chunk's word and its function mask
    uint32_t rw, rf;     // lane 0's word and mask of the chunk to the right
    int32_t B;           // subtrees complete to the right of this chunk
};

struct FxChunk {
    uint32_t n;          // instructions, including the captures' end marks
    int32_t in, mx, mn;  // B before the chunk (uniform); largest and smallest B after this lane's nodes
    bool bad;            // malformed
};

// Decode the chunk at `base` (c.w, c.f; fl: the mask of the chunk to the
// left) into the list at shared address `code`.  word j holds the index of
// instruction j and the operand of instruction j - 1, so that the executor
// has the index of the next instruction one instruction early.  lt: shared
// address of the leaf table, LS bytes per opcode.  caps: 0x01 in the bytes of nodes after which the list is
// interrupted by an end mark (CAP).
template <int V, bool CAP, int LS>
__device__ __forceinline__ FxChunk fx_decode(FxCarry& c, uint32_t fl_word, int32_t base, uint32_t s, uint32_t e,
                                             uint32_t code, uint32_t lt, uint32_t caps) {
    const int lane = lane_id();
    const int32_t q = base + 4 * lane;
    const uint32_t w = c.w, f = c.f;
    // neighbours' words and masks
    uint32_t wr = __shfl_down_sync(FULL, w, 1), fr = __shfl_down_sync(FULL, f, 1), fl = __shfl_up_sync(FULL, f, 1);
    const uint32_t fl31 = __shfl_sync(FULL, fl_word, 31);
    if (lane == 31) { wr = c.rw; fr = c.rf; }
    if (lane == 0) fl = fl31;
    c.rw = __shfl_sync(FULL, w, 0);
    c.rf = __shfl_sync(FULL, f, 0);
    // positions inside the run
    uint32_t valid = 0xFFFFFFFFu;
    if (q < (int32_t)s || q + 4 > (int32_t)e) {
        if (q >= (int32_t)e || q + 4 <= (int32_t)s) valid = 0u;
        else {
            if (q < (int32_t)s) valid &= 0xFFFFFFFFu << (8 * (s - (uint32_t)q));
            if (q + 4 > (int32_t)e) valid &= 0xFFFFFFFFu >> (32 - 8 * (e - (uint32_t)q));
        }
    }
    const uint32_t n1 = __funnelshift_r(w, wr, 8), n2 = __funnelshift_r(w, wr, 16);      // the next two opcodes
    const uint32_t f1 = __funnelshift_r(f, fr, 8), f2 = __funnelshift_r(f, fr, 16);      // are they functions
    const uint32_t p1 = __funnelshift_l(fl, f, 8), p2 = __funnelshift_l(fl, f, 16);      // the two before
    // f L L; and f g L L, where g's instruction becomes part of f's (not while values are captured: g may be asked for)
    const uint32_t isll = f & ~f1 & ~f2;
    uint32_t pair = 0u, taken = 0u;
    if (V == VB && !CAP) {
        pair = f & f1 & ~f2 & ~__funnelshift_r(f, fr, 24);
        taken = isll & p1;
    }
    // a function makes an instruction, a leaf when neither node before it takes it
    const uint32_t head = valid & ((f & ~taken) | ~(f | p1 | p2));
    // depths: +1 per leaf, -1 per function, summed from the right
    const uint32_t step = (valid & 0x01010101u) | (valid & f);
    const int d3 = __dp4a((int)step, 0x01000000, 0), d2 = __dp4a((int)step, 0x01010000, 0);
    const int d1 = __dp4a((int)step, 0x01010100, 0), d0 = __dp4a((int)step, 0x01010101, 0);
    uint32_t own = (uint32_t)__popc(head & 0x01010101u);
    if (CAP) own += (uint32_t)__popc(caps);
    own += (uint32_t)d0 << 16;
    uint32_t sum = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(FULL, sum, o);
        if (lane + o < 32) sum += v;
    }
    const uint32_t all = __shfl_sync(FULL, sum, 0);
    const uint32_t right = sum - own;
    const int b0 = c.B + ((int32_t)right >> 16);
    FxChunk r;
    r.n = all & 0xFFFFu;
    r.in = c.B;
    r.mx = b0 + max(max(d3, d2), max(d1, d0));
    r.mn = b0 + min(min(d3, d2), min(d1, d0));
    c.B += (int32_t)all >> 16;
    // Well formed: one subtree or more complete after every node, so that each function finds two operands.  Words past
    // the run's end have none yet, nor need the word that holds the end (at most three nodes of it; its top byte is not
    // valid): there the next test says it all.
    // a function among the last two nodes of the run has no operands
    const int32_t last2 = (int32_t)e - 2 - q;
    const bool tail = (valid & f) != 0 && last2 < 4 && (valid & f & (last2 <= 0 ? 0xFFFFFFFFu : 0xFFFFFFFFu << (8 * last2))) != 0;
    r.bad = __any_sync(FULL, r.mn < (int32_t)(valid >> 31) || tail);
    // instruction indexes of the four bytes at once
    uint32_t idx, A;                     // index; the byte of the first operand
    uint32_t both, second = n2;          // f L L and f g L L with two table operands; the byte of the second
    if (V == VB) {
        const uint32_t ll = ((w << 2) & 0x0C0C0C0Cu) | 0x03030303u, lf = ((w << 1) & 0x06060606u) | 0x11111111u;
        const uint32_t fp = (w & 0x03030303u) | 0x18181818u;
        const uint32_t fg = (((w & 0x03030303u) << 4) + 0x23232323u) | ((n1 << 2) & 0x0C0C0C0Cu);
        idx = (isll & ll) | (f & ~f1 & f2 & lf) | (f & f1 & ~pair & fp) | (~f & 0x1D1D1D1Du) | (pair & fg);
        A = (pair & n2) | (f & ~pair & n1) | (~f & w);
        both = isll | pair;
        second = (pair & __funnelshift_r(w, wr, 24)) | (~pair & n2);
    } else {
        const uint32_t x = fx_zero_bytes(w ^ 0x04040404u);
        const uint32_t xr = fx_zero_bytes(wr ^ 0x04040404u);
        const uint32_t x1 = __funnelshift_r(x, xr, 8), x2 = __funnelshift_r(x, xr, 16);
        const uint32_t k1 = ~x1 & 0x02020202u, k2 = ~x2 & 0x01010101u;
        const uint32_t ll = ((w << 2) & 0x0C0C0C0Cu) | k1 | k2;
        const uint32_t lf = ((w << 1) & 0x06060606u) | 0x10101010u | (~x1 & 0x01010101u);
        const uint32_t fp = (w & 0x03030303u) | 0x18181818u;
        const uint32_t lp = 0x1C1C1C1Cu | (~x & 0x01010101u);
        idx = (isll & ll) | (f & ~f1 & f2 & lf) | (f & f1 & fp) | (~f & lp);
        A = (~f & w) | (f & ((isll & x1 & n2) | (~(isll & x1) & n1)));   // the constant: the right leaf when the left one is x
        both = isll & ~x1 & ~x2;
    }
    // the lane's instructions in execution order: from its last byte down
    uint32_t at = code + ((right & 0xFFFFu) << 3);
    const uint32_t size = (uint32_t)LS, most = (V == VB) ? FX_BROWS - 1u : 0xFFu;
#pragma unroll
    for (int j = 3; j >= 0; --j) {
        const uint32_t on = head & (1u << (8 * j));
        const uint32_t y2 = (lt << 16) + ((second >> (8 * j)) & most) * (size << 16);
        const uint32_t y = lt + ((A >> (8 * j)) & most) * size + ((both & (1u << (8 * j))) ? y2 : 0u);
        fx_put(on, at, (idx >> (8 * j)) & 0xFFu, y);
        at += on ? 8u : 0u;
        if (CAP) {
            const uint32_t cap = caps & (1u << (8 * j));
            if (cap) fx_sts(at, FX_EXIT);
            at += cap ? 8u : 0u;
        }
    }
    if (lane == 0) fx_sts(code + (r.n << 3), FX_EXIT);
    __syncwarp();
    return r;
}

// ---- executor
//
// One block of PTX: every instruction ends with an indirect branch to the
// next (declared uniform: all lanes read the same list).  Registers: a.. the
// running value, x.. the inputs, sa the next free stack entry, ip the list;
// nx is the index of the next instruction, loaded one instruction early.
//
// A value of K cases is K 32-bit registers (form S1, S2), or for the
// binary32 set at K = 2 and 4 one or two pairs (P2, P4) on which one
// instruction computes two cases; there the table holds each constant twice.
//
// Operations over a whole value (d, a, b: register prefixes; c: one register
// or pair for all cases):
//   FXO_f(ins, d, a, b)   FXR_f(ins, d, a, c)   FXL_f(ins, d, c, b)   FXM_f(d, a)   FXB_f(d, c)
#define FXO_S1(ins, d, a, b) ins " " d "0, " a "0, " b "0;\n\t"
#define FXR_S1(ins, d, a, c) ins " " d "0, " a "0, " c ";\n\t"
#define FXL_S1(ins, d, c, b) ins " " d "0, " c ", " b "0;\n\t"
#define FXM_S1(d, a) "mov.b32 " d "0, " a "0;\n\t"
#define FXB_S1(d, c) "mov.b32 " d "0, " c ";\n\t"
#define FXO_S2(ins, d, a, b) FXO_S1(ins, d, a, b) ins " " d "1, " a "1, " b "1;\n\t"
#define FXR_S2(ins, d, a, c) FXR_S1(ins, d, a, c) ins " " d "1, " a "1, " c ";\n\t"
#define FXL_S2(ins, d, c, b) FXL_S1(ins, d, c, b) ins " " d "1, " c ", " b "1;\n\t"
#define FXM_S2(d, a) FXM_S1(d, a) "mov.b32 " d "1, " a "1;\n\t"
#define FXB_S2(d, c) FXB_S1(d, c) "mov.b32 " d "1, " c ";\n\t"
#define FXO_P2(ins, d, a, b) FXO_S1(ins, d, a, b)
#define FXR_P2(ins, d, a, c) FXR_S1(ins, d, a, c)
#define FXL_P2(ins, d, c, b) FXL_S1(ins, d, c, b)
#define FXM_P2(d, a) "mov.b64 " d "0, " a "0;\n\t"
#define FXB_P2(d, c) "mov.b64 " d "0, " c ";\n\t"
#define FXO_P4(ins, d, a, b) FXO_S2(ins, d, a, b)
#define FXR_P4(ins, d, a, c) FXR_S2(ins, d, a, c)
#define FXL_P4(ins, d, c, b) FXL_S2(ins, d, c, b)
#define FXM_P4(d, a) FXM_P2(d, a) "mov.b64 " d "1, " a "1;\n\t"
#define FXB_P4(d, c) FXB_P2(d, c) "mov.b64 " d "1, " c ";\n\t"
// one value from or to shared memory, and its stride on the stack
#define FXLD_S1(r, at) "ld.shared.b32 " r "0, [" at "];\n\t"
#define FXST_S1(at, r) "st.shared.b32 [" at "], " r "0;\n\t"
#define FXLD_S2(r, at) "ld.shared.v2.b32 {" r "0, " r "1}, [" at "];\n\t"
#define FXST_S2(at, r) "st.shared.v2.b32 [" at "], {" r "0, " r "1};\n\t"
#define FXLD_P2(r, at) "ld.shared.b64 " r "0, [" at "];\n\t"
#define FXST_P2(at, r) "st.shared.b64 [" at "], " r "0;\n\t"
#define FXLD_P4(r, at) "ld.shared.v2.b64 {" r "0, " r "1}, [" at "];\n\t"
#define FXST_P4(at, r) "st.shared.v2.b64 [" at "], {" r "0, " r "1};\n\t"
#define FXBY_S1 "128"
#define FXBY_S2 "256"
#define FXBY_P2 "256"
#define FXBY_P4 "512"
// one constant
#define FXC_S1(r, at) "ld.shared.b32 " r ", [" at "];\n\t"
#define FXC_S2(r, at) FXC_S1(r, at)
#define FXC_P2(r, at) "ld.shared.b64 " r ", [" at "];\n\t"
#define FXC_P4(r, at) FXC_P2(r, at)

#define FX_NEXT "mov.b32 nx, ix;\n\tld.shared.v2.b32 {ix, oy}, [ip];\n\tadd.u32 ip, ip, 8;\n\t"
#define FX_GO "brx.idx.uni nx, FXT;\n"
#define FX_PUSH(F) FXST_##F("sa", "a") "add.u32 sa, sa, " FXBY_##F ";\n\t"
#define FX_POP(F) "sub.u32 sa, sa, " FXBY_##F ";\n\t" FXLD_##F("r", "sa")
#define FX_CST(F) FXC_##F("c0", "oy")
#define FX_TWO(F) "and.b32 t, oy, 0xFFFF;\n\tshr.u32 u, oy, 16;\n\t" FXC_##F("c0", "t") FXC_##F("c1", "u")

// The seven instructions of a function that is one machine instruction (o:
// its number): labels FXA for f L L by leaf kinds, FXM for f L ., FXP for f f ..
#define FX_FUNC(F, o, ins)                                                                                          \
    "FXA" o "0:\n\t" FX_NEXT FX_PUSH(F) FXO_##F(ins, "a", "x", "x") FX_GO                                            \
    "FXA" o "1:\n\t" FX_CST(F) FX_NEXT FX_PUSH(F) FXR_##F(ins, "a", "x", "c0") FX_GO                                 \
    "FXA" o "2:\n\t" FX_CST(F) FX_NEXT FX_PUSH(F) FXL_##F(ins, "a", "c0", "x") FX_GO                                 \
    "FXA" o "3:\n\t" FX_TWO(F) FX_NEXT FX_PUSH(F) ins " c0, c0, c1;\n\t" FXB_##F("a", "c0") FX_GO                    \
    "FXM" o "0:\n\t" FX_NEXT FXO_##F(ins, "a", "x", "a") FX_GO                                                       \
    "FXM" o "1:\n\t" FX_CST(F) FX_NEXT FXL_##F(ins, "a", "c0", "a") FX_GO                                            \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(F) FXO_##F(ins, "a", "a", "r") FX_GO
// Division: operands to n.. and r.., then the shared body at FXDV.
#define FX_LONG(F, o)                                                                                               \
    "FXA" o "0:\n\t" FX_NEXT FX_PUSH(F) FXM_##F("n", "x") FXM_##F("r", "x") "bra.uni FXDV;\n"                        \
    "FXA" o "1:\n\t" FX_CST(F) FX_NEXT FX_PUSH(F) FXM_##F("n", "x") FXB_##F("r", "c0") "bra.uni FXDV;\n"             \
    "FXA" o "2:\n\t" FX_CST(F) FX_NEXT FX_PUSH(F) FXB_##F("n", "c0") FXM_##F("r", "x") "bra.uni FXDV;\n"             \
    "FXA" o "3:\n\t" FX_TWO(F) FX_NEXT FX_PUSH(F) FXB_##F("n", "c0") FXB_##F("r", "c1") "bra.uni FXDV;\n"            \
    "FXM" o "0:\n\t" FX_NEXT FXM_##F("r", "a") FXM_##F("n", "x") "bra.uni FXDV;\n"                                   \
    "FXM" o "1:\n\t" FX_CST(F) FX_NEXT FXM_##F("r", "a") FXB_##F("n", "c0") "bra.uni FXDV;\n"                        \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(F) FXM_##F("n", "a") "bra.uni FXDV;\n"

// Protected binary32 division.  When every operand of the warp lies within
// [2^-60, 2^60] no step below can overflow or lose bits, and the quotient is
// Markstein's (IBM J. Res. Dev. 34, 1990): y an approximate reciprocal, one
// Newton step y += y (1 - b y), q = a y, q += y (a - b q).  For this
// machine's rcp.approx it is the correctly rounded quotient for all 2^46
// pairs of significands (every pair was compared with its remainder); the
// scale of the operands does not change a bit of it.  Without the Newton step
// 79,381 pairs would be one unit off.  Any other operand -- zero, tiny, huge,
// not finite -- sends the warp to FXDR: 1 for a zero divisor (as 1 / 1), else
// the machine's division.
#define FXD_IN(v, w, z) "max.NaN.f32 h, " v ", " w ", " z ";\n\tmin.f32 l, " v ", " w ", " z ";\n\t"
#define FXD_MORE2(v, w) "max.NaN.f32 h, h, " v ", " w ";\n\tmin.f32 l, l, " v ", " w ";\n\t"
#define FXD_ONE(k) "setp.eq.f32 p, d" #k ", 0f00000000;\n\tselp.b32 m" #k ", 0x3F800000, m" #k ", p;\n\t"           \
                   "selp.b32 d" #k ", 0x3F800000, d" #k ", p;\n\tdiv.rn.f32 m" #k ", m" #k ", d" #k ";\n\t"
#define FXD_TEST "setp.le.f32 p, h, 0f5D800000;\n\tsetp.ge.and.f32 p, l, 0f21800000, p;\n\t"                        \
                 "vote.sync.all.pred p, p, 0xFFFFFFFF;\n\t@!p bra.uni FXDR;\n\t"
#define FXD_ABS(k) "abs.f32 e" #k ", m" #k ";\n\tabs.f32 g" #k ", d" #k ";\n\t"
#define FXD_PAIR(i, ka, kb) /* pair i holds cases ka and kb; m: numerators, d: divisors */                          \
    "rcp.approx.ftz.f32 e" #ka ", d" #ka ";\n\trcp.approx.ftz.f32 e" #kb ", d" #kb ";\n\tmov.b64 y, {e" #ka ", e" #kb "};\n\t" \
    "xor.b64 v, r" #i ", 0x8000000080000000;\n\tfma.rn.f32x2 z, v, y, one;\n\tfma.rn.f32x2 y, y, z, y;\n\t"          \
    "mul.rn.f32x2 q, n" #i ", y;\n\tfma.rn.f32x2 z, v, q, n" #i ";\n\tfma.rn.f32x2 a" #i ", z, y, q;\n\t"
#define FXDIV_S1                                                                                                    \
    "mov.b32 m0, n0;\n\tmov.b32 d0, r0;\n\t" FXD_ABS(0)                                                              \
    "max.NaN.f32 h, e0, g0;\n\tmin.f32 l, e0, g0;\n\t" FXD_TEST                                                      \
    "rcp.approx.ftz.f32 e0, d0;\n\tneg.f32 g0, d0;\n\tfma.rn.f32 h, g0, e0, 0f3F800000;\n\tfma.rn.f32 e0, e0, h, e0;\n\t" \
    "mul.rn.f32 h, m0, e0;\n\tfma.rn.f32 l, g0, h, m0;\n\tfma.rn.f32 a0, l, e0, h;\n\t" FX_GO                        \
    "FXDR:\n\t" FXD_ONE(0) "mov.b32 a0, m0;\n\t" FX_GO
#define FXDIV_P2                                                                                                    \
    "mov.b64 {m0, m1}, n0;\n\tmov.b64 {d0, d1}, r0;\n\t" FXD_ABS(0) FXD_ABS(1)                                       \
    FXD_IN("e0", "e1", "g0") "max.NaN.f32 h, h, g1;\n\tmin.f32 l, l, g1;\n\t" FXD_TEST FXD_PAIR(0, 0, 1) FX_GO       \
    "FXDR:\n\t" FXD_ONE(0) FXD_ONE(1) "mov.b64 a0, {m0, m1};\n\t" FX_GO
#define FXDIV_P4                                                                                                    \
    "mov.b64 {m0, m1}, n0;\n\tmov.b64 {d0, d1}, r0;\n\tmov.b64 {m2, m3}, n1;\n\tmov.b64 {d2, d3}, r1;\n\t"           \
    FXD_ABS(0) FXD_ABS(1) FXD_ABS(2) FXD_ABS(3) FXD_IN("e0", "e1", "g0") FXD_MORE2("g1", "e2") FXD_MORE2("e3", "g2") \
    "max.NaN.f32 h, h, g3;\n\tmin.f32 l, l, g3;\n\t" FXD_TEST FXD_PAIR(0, 0, 1) FXD_PAIR(1, 2, 3) FX_GO              \
    "FXDR:\n\t" FXD_ONE(0) FXD_ONE(1) FXD_ONE(2) FXD_ONE(3) "mov.b64 a0, {m0, m1};\n\tmov.b64 a1, {m2, m3};\n\t" FX_GO
// integers: 1 for a zero divisor (1 / 1); INT32_MIN / -1 = INT32_MIN (divided by 1 instead)
#define FX_IDIV1(k) "setp.eq.s32 p, r" #k ", 0;\n\tselp.b32 n" #k ", 1, n" #k ", p;\n\tselp.b32 r" #k ", 1, r" #k ", p;\n\t" \
                    "setp.eq.s32 p, r" #k ", -1;\n\tsetp.eq.and.s32 p, n" #k ", 0x80000000, p;\n\t"                    \
                    "selp.b32 r" #k ", 1, r" #k ", p;\n\tdiv.s32 a" #k ", n" #k ", r" #k ";\n\t"
#define FX_IDIV_S1 FX_IDIV1(0) FX_GO
#define FX_IDIV_S2 FX_IDIV1(0) FX_IDIV1(1) FX_GO
// Boolean: every leaf is a row of the table, at the lane's place
#define FX_BFUNC(F, o, ins, post)                                                                                   \
    "FXA" o "3:\n\tand.b32 t, oy, 0xFFFF;\n\tshr.u32 u, oy, 16;\n\tadd.u32 t, t, lo;\n\tadd.u32 u, u, lo;\n\t"       \
    FXLD_##F("n", "t") FXLD_##F("r", "u") FX_NEXT FX_PUSH(F) FXO_##F(ins, "a", "n", "r") post FX_GO                  \
    "FXM" o "1:\n\tadd.u32 t, oy, lo;\n\t" FXLD_##F("n", "t") FX_NEXT FXO_##F(ins, "a", "n", "a") post FX_GO         \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(F) FXO_##F(ins, "a", "a", "r") post FX_GO
// f g L L
#define FX_BPAIR(F, fo, go, fi, fpost, gi, gpost)                                                                   \
    "FXC" fo go ":\n\tand.b32 t, oy, 0xFFFF;\n\tshr.u32 u, oy, 16;\n\tadd.u32 t, t, lo;\n\tadd.u32 u, u, lo;\n\t"     \
    FXLD_##F("n", "t") FXLD_##F("r", "u") FX_NEXT FXO_##F(gi, "r", "n", "r") gpost FXO_##F(fi, "a", "r", "a") fpost FX_GO
#define FX_BPAIRS(F, fo, fi, fpost)                                                                                 \
    FX_BPAIR(F, fo, "0", fi, fpost, "and.b32", "") FX_BPAIR(F, fo, "1", fi, fpost, "or.b32", "")                      \
    FX_BPAIR(F, fo, "2", fi, fpost, "and.b32", FXNR_##F) FX_BPAIR(F, fo, "3", fi, fpost, "or.b32", FXNR_##F)
#define FXN_S1 "not.b32 a0, a0;\n\t"
#define FXN_S2 FXN_S1 "not.b32 a1, a1;\n\t"
#define FXNR_S1 "not.b32 r0, r0;\n\t"
#define FXNR_S2 FXNR_S1 "not.b32 r1, r1;\n\t"

#define FX_REGS_S ".reg .b32 a0, a1, x0, x1, r0, r1, n0, n1, c0, c1;\n\t"
#define FX_REGS_P ".reg .b64 a0, a1, x0, x1, r0, r1, n0, n1, c0, c1, y, z, v, q, one;\n\tmov.b64 one, 0x3F8000003F800000;\n\t"
#define FX_REGS                                                                                                     \
    ".reg .pred p;\n\t.reg .b32 ix, oy, nx, t, u, ip, sa, lo, h, l, m0, m1, m2, m3, d0, d1, d2, d3;\n\t"             \
    ".reg .b32 e0, e1, e2, e3, g0, g1, g2, g3;\n\t"
#define FX_TABLE                                                                                                    \
    "FXT: .branchtargets FXA00, FXA01, FXA02, FXA03, FXA10, FXA11, FXA12, FXA13, FXA20, FXA21, FXA22, FXA23, "       \
    "FXA30, FXA31, FXA32, FXA33, FXM00, FXM01, FXM10, FXM11, FXM20, FXM21, FXM30, FXM31, FXP00, FXP10, FXP20, "      \
    "FXP30, FXL0, FXL1, FXEND;\n\t"
#define FX_BROW4(l) l ", " l ", " l ", " l
#define FX_BROW(f) FX_BROW4("FXC" f "0") ", " FX_BROW4("FXC" f "1") ", " FX_BROW4("FXC" f "2") ", " FX_BROW4("FXC" f "3")
#define FX_BTABLE                                                                                                   \
    "FXT: .branchtargets FXA03, FXA03, FXA03, FXA03, FXA13, FXA13, FXA13, FXA13, FXA23, FXA23, FXA23, FXA23, "       \
    "FXA33, FXA33, FXA33, FXA33, FXM01, FXM01, FXM11, FXM11, FXM21, FXM21, FXM31, FXM31, FXP00, FXP10, FXP20, "      \
    "FXP30, FXL1, FXL1, FXEND, FXEND, " FX_BROW("0") ", " FX_BROW("1") ", " FX_BROW("2") ", " FX_BROW("3") ";\n\t"
#define FX_START "ld.shared.v2.b32 {ix, oy}, [ip];\n\tadd.u32 ip, ip, 8;\n\t" FX_NEXT FX_GO
#define FX_STOP "FXEND:\n\tsub.u32 ip, ip, 8;\n\t"
#define FX_LEAVES(F)                                                                                                \
    "FXL0:\n\t" FX_NEXT FX_PUSH(F) FXM_##F("a", "x") FX_GO                                                           \
    "FXL1:\n\t" FX_CST(F) FX_NEXT FX_PUSH(F) FXB_##F("a", "c0") FX_GO
#define FX_BODY_F(F, w)                                                                                             \
    FX_FUNC(F, "0", "add.rn.f32" w) FX_FUNC(F, "1", "sub.rn.f32" w) FX_FUNC(F, "2", "mul.rn.f32" w) FX_LONG(F, "3")  \
    "FXDV:\n\t" FXDIV_##F FX_LEAVES(F) FX_STOP
#define FX_BODY_I(F)                                                                                                \
    FX_FUNC(F, "0", "add.u32") FX_FUNC(F, "1", "sub.u32") FX_FUNC(F, "2", "mul.lo.u32") FX_LONG(F, "3")              \
    "FXDV:\n\t" FX_IDIV_##F FX_LEAVES(F) FX_STOP
#define FX_BODY_B(F)                                                                                                \
    FX_BFUNC(F, "0", "and.b32", "") FX_BFUNC(F, "1", "or.b32", "") FX_BFUNC(F, "2", "and.b32", FXN_##F)              \
    FX_BFUNC(F, "3", "or.b32", FXN_##F)                                                                              \
    FX_BPAIRS(F, "0", "and.b32", "") FX_BPAIRS(F, "1", "or.b32", "") FX_BPAIRS(F, "2", "and.b32", FXN_##F)           \
    FX_BPAIRS(F, "3", "or.b32", FXN_##F)                                                                             \
    "FXL1:\n\tadd.u32 t, oy, lo;\n\t" FX_NEXT FX_PUSH(F) FXLD_##F("a", "t") FX_GO FX_STOP

// Run the list at shared address `ip` up to an end mark; afterwards ip is
// where to go on from.  lo: the lane's offset in a row of the Boolean table.
template <int K, int V>
__device__ __forceinline__ void fx_exec(uint32_t& ip, float (&a)[K], uint32_t& sa, const float (&x)[K], uint32_t lo) {
    if constexpr (K == 1) {
#define FX_ASM(TAB, BODY)                                                                                           \
    asm volatile("{\n\t" FX_REGS FX_REGS_S TAB "mov.b32 a0, %0;\n\tmov.b32 sa, %1;\n\tmov.b32 ip, %2;\n\t"           \
                 "mov.b32 x0, %3;\n\tmov.b32 lo, %4;\n\t" FX_START BODY                                             \
                 "mov.b32 %0, a0;\n\tmov.b32 %1, sa;\n\tmov.b32 %2, ip;\n\t}"                                        \
                 : "+f"(a[0]), "+r"(sa), "+r"(ip) : "f"(x[0]), "r"(lo) : "memory")
        if constexpr (V == VF) FX_ASM(FX_TABLE, FX_BODY_F(S1, ""));
        else if constexpr (V == VI) FX_ASM(FX_TABLE, FX_BODY_I(S1));
        else FX_ASM(FX_BTABLE, FX_BODY_B(S1));
#undef FX_ASM
    } else if constexpr (K == 2 && V != VF) {
#define FX_ASM(TAB, BODY)                                                                                           \
    asm volatile("{\n\t" FX_REGS FX_REGS_S TAB "mov.b32 a0, %0;\n\tmov.b32 a1, %1;\n\tmov.b32 sa, %2;\n\t"           \
                 "mov.b32 ip, %3;\n\tmov.b32 x0, %4;\n\tmov.b32 x1, %5;\n\tmov.b32 lo, %6;\n\t" FX_START BODY         \
                 "mov.b32 %0, a0;\n\tmov.b32 %1, a1;\n\tmov.b32 %2, sa;\n\tmov.b32 %3, ip;\n\t}"                     \
                 : "+f"(a[0]), "+f"(a[1]), "+r"(sa), "+r"(ip) : "f"(x[0]), "f"(x[1]), "r"(lo) : "memory")
        if constexpr (V == VI) FX_ASM(FX_TABLE, FX_BODY_I(S2));
        else FX_ASM(FX_BTABLE, FX_BODY_B(S2));
#undef FX_ASM
    } else if constexpr (K == 2) {
        asm volatile("{\n\t" FX_REGS FX_REGS_P FX_TABLE "mov.b64 a0, {%0, %1};\n\tmov.b32 sa, %2;\n\tmov.b32 ip, %3;\n\t"
                     "mov.b64 x0, {%4, %5};\n\t" FX_START FX_BODY_F(P2, "x2")
                     "mov.b64 {%0, %1}, a0;\n\tmov.b32 %2, sa;\n\tmov.b32 %3, ip;\n\t}"
                     : "+f"(a[0]), "+f"(a[1]), "+r"(sa), "+r"(ip) : "f"(x[0]), "f"(x[1]) : "memory");
    } else {
        static_assert(K == 4 && V == VF, "four cases per lane: binary32 only");
        asm volatile("{\n\t" FX_REGS FX_REGS_P FX_TABLE "mov.b64 a0, {%0, %1};\n\tmov.b64 a1, {%2, %3};\n\t"
                     "mov.b32 sa, %4;\n\tmov.b32 ip, %5;\n\tmov.b64 x0, {%6, %7};\n\tmov.b64 x1, {%8, %9};\n\t"
                     FX_START FX_BODY_F(P4, "x2")
                     "mov.b64 {%0, %1}, a0;\n\tmov.b64 {%2, %3}, a1;\n\tmov.b32 %4, sa;\n\tmov.b32 %5, ip;\n\t}"
                     : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+r"(sa), "+r"(ip)
                     : "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]) : "memory");
    }
}

// Per-warp context of a fused run.
template <int K>
struct FxCtx {
    uint32_t stack;      // this lane's first stack entry (shared address; entries 128 K bytes apart)
    uint32_t code;       // the warp's instruction list (shared address)
    uint32_t lt;         // leaf table (shared address below 64 KB: operands hold two 16-bit addresses)
    uint32_t lo;         // this lane's offset in a row of the Boolean leaf table
    uint32_t W, maxd;    // entries in shared memory, entries in all
    float* g;            // global overflow: maxd entries x 32 lanes x K
    float x[K];          // the lane's inputs (binary32, integer)
};

// Leaf table of a CTA.  Binary32 and integer sets: the constants by opcode.
// Boolean sets: 16 rows by opcode (4.. the inputs) of the words of each case
// block, lane by lane, K words per lane; a row is 128 K bytes.
template <int K, int V>
struct FxTable {
    // bytes of an entry: a Boolean row, a constant (twice at K = 2 and 4: operands of paired instructions)
    static constexpr int row = V == VB ? 32 * K * 4 : (V == VF && K > 1) ? 8 : 4;
    __host__ __device__ static uint32_t bytes(uint32_t ncb) { return V == VB ? FX_BROWS * row * ncb : 256u * row; }
    // address of case block cb's table
    __device__ static uint32_t at(uint32_t base, uint32_t cb) { return V == VB ? base + cb * FX_BROWS * row : base; }
    __device__ static void fill(float* tab, const float* consts, uint32_t ncb) {
        if (V == VB) {
            for (uint32_t i = threadIdx.x; i < FX_BROWS * 32 * K * ncb; i += blockDim.x) {
                const uint32_t k = i % K, lane = (i / K) % 32, op = (i / (32 * K)) % FX_BROWS, cb = i / (32 * K * FX_BROWS);
                const uint32_t b = op - 4u, w = cb * 32 * K + k * 32 + lane;
                tab[i] = op < 4u ? 0.0f : __uint_as_float(mux_word(b, mux_pattern(b < 5u ? b : 0u), w));
            }
        } else {
            constexpr uint32_t n = row / 4;
            for (uint32_t i = threadIdx.x; i < 256 * n; i += blockDim.x) tab[i] = (i / n >= 5) ? consts[i / n - 5] : 0.0f;
        }
    }
};

// Slide the window: entries [0, lo) of the stack are in global memory, the
// others at stack + (i - lo) entries.  Every lane moves its own column.
template <int K>
__device__ __forceinline__ void fx_slide(const FxCtx<K>& c, uint32_t& lo, uint32_t& sa, uint32_t to) {
    constexpr uint32_t stride = 32 * K * 4;
    float* g = c.g + lane_id() * K;
    const uint32_t have = (sa - c.stack) / stride;          // entries in the window
    float v[K];
    if (to > lo) {
        const uint32_t n = to - lo;
        for (uint32_t j = 0; j < n; ++j) { lds_vec<K>(c.stack + j * stride, v); vstore<K>(g + (size_t)(lo + j) * 32 * K, v); }
        for (uint32_t j = n; j < have; ++j) { lds_vec<K>(c.stack + j * stride, v); sts_vec<K>(c.stack + (j - n) * stride, v); }
        sa -= n * stride;
    } else {
        const uint32_t n = lo - to;
        for (uint32_t j = have; j-- > 0;) { lds_vec<K>(c.stack + j * stride, v); sts_vec<K>(c.stack + (j + n) * stride, v); }
        for (uint32_t j = 0; j < n; ++j) { vload<K>(g + (size_t)(to + j) * 32 * K, v); sts_vec<K>(c.stack + j * stride, v); }
        sa += n * stride;
    }
    lo = to;
}

// The list at ip with the whole stack, `dep` entries, in the global area.
template <int K, int V>
__device__ __forceinline__ void fx_exec_global(uint32_t& ip, float (&a)[K], uint32_t& dep, const FxCtx<K>& c) {
    float* g = c.g + lane_id() * K;
    auto push = [&]() { vstore<K>(g + (size_t)dep * 32 * K, a); ++dep; };
    auto leaf = [&](uint32_t y, bool cst, float (&v)[K]) {
        if constexpr (V == VB) { lds_vec<K>(y + c.lo, v); (void)cst; }
        else {
            const float cv = cst ? lds_f32(y) : 0.0f;
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = cst ? cv : c.x[k];
        }
    };
    for (;; ip += 8) {
        const uint32_t idx = lds_u32(ip), y = lds_u32(ip + 12);
        if (idx == FX_EXIT) break;
        float l[K], r[K];
        // What a chunk of great depths mostly holds comes first: leaves that wait, functions that take two values.  (A lone
        // warp pays for each branch: 3,000 left combs of 1,023 nodes x 100 cases 15.4 -> 13.9 ms.)
        if (idx >= 28u) {
            if (V == VB && idx >= 32u) {
                leaf(y & 0xFFFFu, true, l);
                leaf(y >> 16, true, r);
                apply_vec<K, V>((idx >> 2) & 3u, l, r);
                apply_vec<K, V>((idx - 32u) >> 4, l, a);
            } else {
                push();
                leaf(y, idx & 1u, l);
            }
#pragma unroll
            for (int k = 0; k < K; ++k) a[k] = l[k];
        } else if (idx >= 24u) {
            --dep;
            vload<K>(g + (size_t)dep * 32 * K, r);
            apply_vec<K, V>(idx - 24u, a, r);
        } else {
            if (idx < 16u) {
                const bool ca = idx & 2u, cb = idx & 1u;
                push();
                leaf(ca && cb ? y & 0xFFFFu : y, ca, l);
                leaf(ca && cb ? y >> 16 : y, cb, r);
                apply_vec<K, V>(idx >> 2, l, r);
            } else {
                leaf(y, idx & 1u, l);
                apply_vec<K, V>((idx - 16u) >> 1, l, a);
            }
#pragma unroll
            for (int k = 0; k < K; ++k) a[k] = l[k];
        }
    }
    ip += 8;                       // past the end mark
}

// Make the window fit the chunk about to run; false when its depths span
// more than the window (the stack is then all in the global area).  `lo`
// entries are below the window; an instruction whose leaves lie in the chunk
// to the right leaves the stack up to two entries short of B.
// need(): called before the global area is first used; false when there is none.
struct FxHave {
    __device__ bool operator()() const { return true; }
};
template <int K, typename NEED>
__device__ __forceinline__ bool fx_fit(const FxChunk& ch, const FxCtx<K>& c, uint32_t& lo, uint32_t& sa, bool& ok,
                                       NEED& need) {
    const int32_t top = (int32_t)(lo + c.W);
    const bool low = lo > 0 && (ch.in < (int32_t)lo + 2 || ch.mn < (int32_t)lo);
    if (!__any_sync(FULL, ch.in > top || ch.mx > top || low)) return true;
    const int32_t mx = max(ch.in, __reduce_max_sync(FULL, ch.mx));
    const int32_t mn = max(0, min(ch.in - 2, __reduce_min_sync(FULL, ch.mn)));
    if (mx > (int32_t)c.maxd || !need()) { ok = false; return true; }
    const int32_t span = mx - mn;
    if (span <= (int32_t)c.W) {
        fx_slide<K>(c, lo, sa, (uint32_t)max(0, mn - ((int32_t)c.W - span) / 2));
        return true;
    }
    fx_slide<K>(c, lo, sa, lo + (sa - c.stack) / (32 * K * 4));
    return false;
}

// Evaluate the nodes [s, e): afterwards a holds the value of the subtree at
// s.  `ld(q)` reads the 32-bit word at position q (a multiple of 4); w0, w1
// are this lane's words of the last chunk and of the one to its left, read
// by the caller (fx_first), who can have them in flight early.  `stop`: a
// shared word that, once nonzero, ends the run early with *aborted set.
template <int K, int V, typename LD, typename NEED = FxHave>
__device__ __forceinline__ bool fx_run(LD ld, uint32_t s, uint32_t e, uint32_t w0, uint32_t w1, const FxCtx<K>& c,
                                       float (&a)[K], NEED need = NEED(), const volatile uint32_t* stop = nullptr,
                                       bool* aborted = nullptr) {
    const int lane = lane_id();
    int32_t base = (int32_t)((e - 1) & ~(uint32_t)(FX_CHUNK - 1));
    FxCarry cy;
    cy.w = w0;
    cy.f = fx_funcs(w0);
    cy.rw = 0xFFFFFFFFu;
    cy.rf = 0u;
    cy.B = 0;
    uint32_t sa = c.stack, lo = 0, wl = w1;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = 0.f;
    for (;;) {
        // (one decision for the warp: what follows needs all of its lanes)
        if (stop && __any_sync(FULL, *stop != 0u)) { *aborted = true; return true; }
        const uint32_t fl = fx_funcs(wl);
        const uint32_t wn = fx_word(ld, base - 2 * FX_CHUNK + 4 * lane, s, e);     // in flight during this chunk
        const FxChunk ch = fx_decode<V, false, FxTable<K, V>::row>(cy, fl, base, s, e, c.code, c.lt, 0u);
        if (ch.bad) { ok = false; break; }
        uint32_t ip = c.code;
        const bool fits = fx_fit<K>(ch, c, lo, sa, ok, need);
        if (!ok) break;
        if (fits) fx_exec<K, V>(ip, a, sa, c.x, c.lo);
        else fx_exec_global<K, V>(ip, a, lo, c);
        __syncwarp();
        if (base <= (int32_t)s) break;
        base -= FX_CHUNK;
        cy.w = wl;
        cy.f = fl;
        wl = wn;
    }
    return ok && cy.B == 1;
}

// fx_run over a whole tree [0, e) that also hands out the values of chosen
// nodes: cap(k) is called by the whole warp when a holds the value of the
// subtree at pos(k); the positions pos(0) > pos(1) > ... (ncap of them) are
// functions, or the root.  The instruction list is interrupted after each
// (its buffer holds FX_CAP_BYTES).
#define FX_CAP_BYTES ((2 * FX_CHUNK + 2) * 8)
template <int K, int V, typename LD, typename PosF, typename CapF>
__device__ __forceinline__ bool fx_run_capture(LD ld, uint32_t e, const FxCtx<K>& c, float (&a)[K], uint32_t ncap, PosF pos,
                                               CapF cap) {
    const int lane = lane_id();
    int32_t base = (int32_t)((e - 1) & ~(uint32_t)(FX_CHUNK - 1));
    FxCarry cy;
    cy.w = fx_word(ld, base + 4 * lane, 0u, e);
    uint32_t wl = fx_word(ld, base - FX_CHUNK + 4 * lane, 0u, e);
    cy.f = fx_funcs(cy.w);
    cy.rw = 0xFFFFFFFFu;
    cy.rf = 0u;
    cy.B = 0;
    uint32_t sa = c.stack, lo = 0, k = 0;
    int32_t nextp = ncap ? (int32_t)pos(0) : -1;
    bool ok = true;
    FxHave have;
#pragma unroll
    for (int j = 0; j < K; ++j) a[j] = 0.f;
    for (;;) {
        const uint32_t fl = fx_funcs(wl);
        const uint32_t wn = fx_word(ld, base - 2 * FX_CHUNK + 4 * lane, 0u, e);     // in flight during this chunk
        uint32_t caps = 0, n = 0;
        while (nextp >= base) {
            if ((nextp - base) >> 2 == lane) caps |= 1u << (8 * (nextp & 3));
            ++n;
            nextp = (k + n < ncap) ? (int32_t)pos(k + n) : -1;
        }
        const FxChunk ch = fx_decode<V, true, FxTable<K, V>::row>(cy, fl, base, 0u, e, c.code, c.lt, caps);
        if (ch.bad) { ok = false; break; }
        const bool fits = fx_fit<K>(ch, c, lo, sa, ok, have);
        if (!ok) break;
        uint32_t ip = c.code;
        for (uint32_t j = 0;; ++j) {
            if (fits) fx_exec<K, V>(ip, a, sa, c.x, c.lo);
            else fx_exec_global<K, V>(ip, a, lo, c);
            if (j == n) break;
            cap(k + j);
        }
        k += n;
        __syncwarp();
        if (base <= 0) break;
        base -= FX_CHUNK;
        cy.w = wl;
        cy.f = fl;
        wl = wn;
    }
    return ok && cy.B == 1;
}

// this lane's words of the run's last chunk and of the one before it
template <typename LD>
__device__ __forceinline__ void fx_first(LD ld, uint32_t s, uint32_t e, uint32_t& w0, uint32_t& w1) {
    const int32_t base = (int32_t)((e - 1) & ~(uint32_t)(FX_CHUNK - 1)) + 4 * lane_id();
    w0 = fx_word(ld, base, s, e);
    w1 = fx_word(ld, base - FX_CHUNK, s, e);
}
