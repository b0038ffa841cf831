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
//   L        push acc; acc = L     a leaf that no function to its left takes at once
// A node's form depends on its own opcode and its two neighbours' on either
// side, so 32 lanes decode 128 nodes with a few byte-parallel operations
// each, and leaves -- half of all nodes -- mostly cost no instruction of
// their own.  Every opcode is still applied to every test case, to the same
// operands in the same order: the values are the same bits.
//
// Stack depth: B(q), the number of complete subtrees in [q, end), is the
// number of entries between two instructions (one of them the initial
// running value).  The decoder knows it, so the executor has no checks: a
// chunk of 128 nodes whose depths stay within the shared window runs on it
// alone, any other chunk on a checked path with the global overflow area,
// and a malformed run (B negative somewhere, or not 1 at its start) is
// refused before anything is executed that could leave the stack.
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
// Boolean: the constant bits are all set.

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
    bool over, bad;      // deeper than the window; malformed
};

// Decode the chunk at `base` (c.w, c.f; fl: the mask of the chunk to the
// left) into the list at shared address `code`.  word j holds the index of
// instruction j and the operand of instruction j - 1, so that the executor
// has the index of the next instruction one instruction early.  lt: shared
// address of the leaf table (constants: 4 bytes per opcode; Boolean: LS bytes
// per input).  caps: 0x01 in the bytes of nodes after which the list is
// interrupted by an end mark (CAP).
template <int V, bool CAP, int LS>
__device__ __forceinline__ FxChunk fx_decode(FxCarry& c, uint32_t fl_word, int32_t base, uint32_t s, uint32_t e,
                                             uint32_t W, uint32_t code, uint32_t lt, uint32_t caps) {
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
    // a function always makes an instruction, a leaf when neither node before it takes it
    const uint32_t head = valid & (f | ~(p1 | p2));
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
    const int mx = b0 + max(max(d3, d2), max(d1, d0)), mn = b0 + min(min(d3, d2), min(d1, d0));
    FxChunk r;
    r.n = all & 0xFFFFu;
    r.over = c.B > (int)W || __any_sync(FULL, mx > (int)W);      // before the chunk's first node, or after any of them
    c.B += (int32_t)all >> 16;
    // a function among the last two nodes of the run has no operands
    const int32_t last2 = (int32_t)e - 2 - q;
    const bool tail = (valid & f) != 0 && last2 < 4 && (valid & f & (last2 <= 0 ? 0xFFFFFFFFu : 0xFFFFFFFFu << (8 * last2))) != 0;
    r.bad = __any_sync(FULL, mn < 0 || tail);
    // instruction indexes of the four bytes at once
    uint32_t idx, A;                     // index; the byte of the first operand
    uint32_t both = 0;                   // f L L with two table operands
    if (V == VB) {
        const uint32_t ll = ((w << 2) & 0x0C0C0C0Cu) | 0x03030303u, lf = ((w << 1) & 0x06060606u) | 0x11111111u;
        const uint32_t fp = (w & 0x03030303u) | 0x18181818u;
        idx = (f & ~f1 & ~f2 & ll) | (f & ~f1 & f2 & lf) | (f & f1 & fp) | (~f & 0x1D1D1D1Du);
        A = (f & n1) | (~f & w);
        both = f & ~f1 & ~f2;
    } else {
        const uint32_t x = fx_zero_bytes(w ^ 0x04040404u);
        const uint32_t xr = fx_zero_bytes(wr ^ 0x04040404u);
        const uint32_t x1 = __funnelshift_r(x, xr, 8), x2 = __funnelshift_r(x, xr, 16);
        const uint32_t k1 = ~x1 & 0x02020202u, k2 = ~x2 & 0x01010101u;
        const uint32_t ll = ((w << 2) & 0x0C0C0C0Cu) | k1 | k2;
        const uint32_t lf = ((w << 1) & 0x06060606u) | 0x10101010u | (~x1 & 0x01010101u);
        const uint32_t fp = (w & 0x03030303u) | 0x18181818u;
        const uint32_t lp = 0x1C1C1C1Cu | (~x & 0x01010101u);
        const uint32_t isll = f & ~f1 & ~f2;
        idx = (isll & ll) | (f & ~f1 & f2 & lf) | (f & f1 & fp) | (~f & lp);
        A = (~f & w) | (f & ((isll & x1 & n2) | (~(isll & x1) & n1)));   // the constant: the right leaf when the left one is x
        both = isll & ~x1 & ~x2;
    }
    // the lane's instructions in execution order: from its last byte down
    uint32_t at = code + ((right & 0xFFFFu) << 3);
    const uint32_t size = (V == VB) ? (uint32_t)LS : 4u, most = (V == VB) ? FX_BROWS - 1u : 0xFFu;
#pragma unroll
    for (int j = 3; j >= 0; --j) {
        if (head & (1u << (8 * j))) {
            uint32_t y = lt + ((A >> (8 * j)) & most) * size;
            if (both & (1u << (8 * j))) y |= (lt + ((n2 >> (8 * j)) & most) * size) << 16;
            fx_sts(at, (idx >> (8 * j)) & 0xFFu);
            fx_sts(at + 12, y);
            at += 8;
            if (CAP && (caps & (1u << (8 * j)))) {
                fx_sts(at, FX_EXIT);
                at += 8;
            }
        }
    }
    if (lane == 0) fx_sts(code + (r.n << 3), FX_EXIT);
    __syncwarp();
    return r;
}

// ---- executor
//
// One block of PTX: every instruction ends with an indirect branch to the
// next (declared uniform: all lanes read the same list).  Registers: a0.. the
// running value, x0.. the inputs, sa the next free stack entry, ip the list;
// nx is the index of the next instruction, loaded one instruction early.
#define FX1(ins, d, a, b) ins " " d "0, " a "0, " b "0;\n\t"
#define FX2(ins, d, a, b) FX1(ins, d, a, b) ins " " d "1, " a "1, " b "1;\n\t"
#define FX4(ins, d, a, b) FX2(ins, d, a, b) ins " " d "2, " a "2, " b "2;\n\t" ins " " d "3, " a "3, " b "3;\n\t"
// second or first operand the same register for all cases
#define FXR1(ins, d, a, b) ins " " d "0, " a "0, " b ";\n\t"
#define FXR2(ins, d, a, b) FXR1(ins, d, a, b) ins " " d "1, " a "1, " b ";\n\t"
#define FXR4(ins, d, a, b) FXR2(ins, d, a, b) ins " " d "2, " a "2, " b ";\n\t" ins " " d "3, " a "3, " b ";\n\t"
#define FXL1(ins, d, a, b) ins " " d "0, " a ", " b "0;\n\t"
#define FXL2(ins, d, a, b) FXL1(ins, d, a, b) ins " " d "1, " a ", " b "1;\n\t"
#define FXL4(ins, d, a, b) FXL2(ins, d, a, b) ins " " d "2, " a ", " b "2;\n\t" ins " " d "3, " a ", " b "3;\n\t"
#define FXM1(d, a) "mov.b32 " d "0, " a "0;\n\t"
#define FXM2(d, a) FXM1(d, a) "mov.b32 " d "1, " a "1;\n\t"
#define FXM4(d, a) FXM2(d, a) "mov.b32 " d "2, " a "2;\n\tmov.b32 " d "3, " a "3;\n\t"
#define FXB1(d, a) "mov.b32 " d "0, " a ";\n\t"
#define FXB2(d, a) FXB1(d, a) "mov.b32 " d "1, " a ";\n\t"
#define FXB4(d, a) FXB2(d, a) "mov.b32 " d "2, " a ";\n\tmov.b32 " d "3, " a ";\n\t"
#define FXV1(r) "{" r "0}"
#define FXV2(r) "{" r "0, " r "1}"
#define FXV4(r) "{" r "0, " r "1, " r "2, " r "3}"
#define FXLD1 "ld.shared.b32 "
#define FXLD2 "ld.shared.v2.b32 "
#define FXLD4 "ld.shared.v4.b32 "
#define FXST1 "st.shared.b32 "
#define FXST2 "st.shared.v2.b32 "
#define FXST4 "st.shared.v4.b32 "
#define FXSV1(r) r "0"
#define FXSV2(r) FXV2(r)
#define FXSV4(r) FXV4(r)
#define FXBY1 "128"
#define FXBY2 "256"
#define FXBY4 "512"

#define FX_NEXT "mov.b32 nx, ix;\n\tld.shared.v2.b32 {ix, oy}, [ip];\n\tadd.u32 ip, ip, 8;\n\t"
#define FX_GO "brx.idx.uni nx, FXT;\n"
#define FX_PUSH(K) FXST##K "[sa], " FXSV##K("a") ";\n\tadd.u32 sa, sa, " FXBY##K ";\n\t"
#define FX_POP(K) "sub.u32 sa, sa, " FXBY##K ";\n\t" FXLD##K FXSV##K("r") ", [sa];\n\t"
#define FX_CST "ld.shared.b32 c0, [oy];\n\t"
#define FX_TWO "and.b32 t, oy, 0xFFFF;\n\tshr.u32 u, oy, 16;\n\tld.shared.b32 c0, [t];\n\tld.shared.b32 c1, [u];\n\t"

// the twelve instructions of a function that is one machine instruction `ins`: labels L<b>.. for f L L, M<b>.. for
// f L ., P<b> for f f ..
#define FX_FUNC(K, o, ins)                                                                                          \
    "FXA" o "0:\n\t" FX_NEXT FX_PUSH(K) FX##K(ins, "a", "x", "x") FX_GO                                              \
    "FXA" o "1:\n\t" FX_CST FX_NEXT FX_PUSH(K) FXR##K(ins, "a", "x", "c0") FX_GO                                     \
    "FXA" o "2:\n\t" FX_CST FX_NEXT FX_PUSH(K) FXL##K(ins, "a", "c0", "x") FX_GO                                     \
    "FXA" o "3:\n\t" FX_TWO FX_NEXT FX_PUSH(K) ins " c0, c0, c1;\n\t" FXB##K("a", "c0") FX_GO                        \
    "FXM" o "0:\n\t" FX_NEXT FX##K(ins, "a", "x", "a") FX_GO                                                         \
    "FXM" o "1:\n\t" FX_CST FX_NEXT FXL##K(ins, "a", "c0", "a") FX_GO                                                \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(K) FX##K(ins, "a", "a", "r") FX_GO
// a function of several machine instructions: operands to n.. and r.., then the shared body at FXDV
#define FX_LONG(K, o)                                                                                               \
    "FXA" o "0:\n\t" FX_NEXT FX_PUSH(K) FXM##K("n", "x") FXM##K("r", "x") "bra.uni FXDV;\n"                          \
    "FXA" o "1:\n\t" FX_CST FX_NEXT FX_PUSH(K) FXM##K("n", "x") FXB##K("r", "c0") "bra.uni FXDV;\n"                  \
    "FXA" o "2:\n\t" FX_CST FX_NEXT FX_PUSH(K) FXB##K("n", "c0") FXM##K("r", "x") "bra.uni FXDV;\n"                  \
    "FXA" o "3:\n\t" FX_TWO FX_NEXT FX_PUSH(K) FXB##K("n", "c0") FXB##K("r", "c1") "bra.uni FXDV;\n"                 \
    "FXM" o "0:\n\t" FX_NEXT FXM##K("r", "a") FXM##K("n", "x") "bra.uni FXDV;\n"                                     \
    "FXM" o "1:\n\t" FX_CST FX_NEXT FXM##K("r", "a") FXB##K("n", "c0") "bra.uni FXDV;\n"                             \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(K) FXM##K("n", "a") "bra.uni FXDV;\n"
// protected division: 1 for a zero divisor, without dividing by it (1 / 1)
#define FX_FDIV1(k) "setp.eq.f32 p, r" #k ", 0f00000000;\n\tselp.b32 n" #k ", 0x3F800000, n" #k ", p;\n\t"          \
                    "selp.b32 r" #k ", 0x3F800000, r" #k ", p;\n\tdiv.rn.f32 a" #k ", n" #k ", r" #k ";\n\t"
#define FX_FDIVS1 FX_FDIV1(0)
#define FX_FDIVS2 FX_FDIV1(0) FX_FDIV1(1)
#define FX_FDIVS4 FX_FDIV1(0) FX_FDIV1(1) FX_FDIV1(2) FX_FDIV1(3)
// integers: 1 for a zero divisor (1 / 1); INT32_MIN / -1 = INT32_MIN (divided by 1 instead)
#define FX_IDIV1(k) "setp.eq.s32 p, r" #k ", 0;\n\tselp.b32 n" #k ", 1, n" #k ", p;\n\tselp.b32 r" #k ", 1, r" #k ", p;\n\t" \
                    "setp.eq.s32 p, r" #k ", -1;\n\tsetp.eq.and.s32 p, n" #k ", 0x80000000, p;\n\t"                    \
                    "selp.b32 r" #k ", 1, r" #k ", p;\n\tdiv.s32 a" #k ", n" #k ", r" #k ";\n\t"
#define FX_IDIVS1 FX_IDIV1(0)
#define FX_IDIVS2 FX_IDIV1(0) FX_IDIV1(1)
// Boolean leaves: this lane's words of an input, at the lane's place of the table row
#define FX_BLD(K, r, a) FXLD##K FXSV##K(r) ", [" a "];\n\t"
#define FX_BFUNC(K, o, ins, post)                                                                                   \
    "FXA" o "3:\n\tand.b32 t, oy, 0xFFFF;\n\tshr.u32 u, oy, 16;\n\tadd.u32 t, t, lo;\n\tadd.u32 u, u, lo;\n\t"       \
    FX_BLD(K, "n", "t") FX_BLD(K, "r", "u") FX_NEXT FX_PUSH(K) FX##K(ins, "a", "n", "r") post FX_GO                  \
    "FXM" o "1:\n\tadd.u32 t, oy, lo;\n\t" FX_BLD(K, "n", "t") FX_NEXT FX##K(ins, "a", "n", "a") post FX_GO          \
    "FXP" o "0:\n\t" FX_NEXT FX_POP(K) FX##K(ins, "a", "a", "r") post FX_GO
#define FXN1 "not.b32 a0, a0;\n\t"
#define FXN2 FXN1 "not.b32 a1, a1;\n\t"

#define FX_REGS                                                                                                     \
    ".reg .pred p;\n\t.reg .b32 a0, a1, a2, a3, x0, x1, x2, x3, r0, r1, r2, r3, n0, n1, n2, n3;\n\t"                 \
    ".reg .b32 c0, c1, ix, oy, nx, t, u, ip, sa, lo;\n\t"
#define FX_TABLE                                                                                                    \
    "FXT: .branchtargets FXA00, FXA01, FXA02, FXA03, FXA10, FXA11, FXA12, FXA13, FXA20, FXA21, FXA22, FXA23, "       \
    "FXA30, FXA31, FXA32, FXA33, FXM00, FXM01, FXM10, FXM11, FXM20, FXM21, FXM30, FXM31, FXP00, FXP10, FXP20, "      \
    "FXP30, FXL0, FXL1, FXEND;\n\t"
#define FX_BTABLE                                                                                                   \
    "FXT: .branchtargets FXA03, FXA03, FXA03, FXA03, FXA13, FXA13, FXA13, FXA13, FXA23, FXA23, FXA23, FXA23, "       \
    "FXA33, FXA33, FXA33, FXA33, FXM01, FXM01, FXM11, FXM11, FXM21, FXM21, FXM31, FXM31, FXP00, FXP10, FXP20, "      \
    "FXP30, FXL1, FXL1, FXEND;\n\t"
#define FX_START "ld.shared.v2.b32 {ix, oy}, [ip];\n\tadd.u32 ip, ip, 8;\n\t" FX_NEXT FX_GO
#define FX_LEAVES(K)                                                                                                \
    "FXL0:\n\t" FX_NEXT FX_PUSH(K) FXM##K("a", "x") FX_GO                                                            \
    "FXL1:\n\t" FX_CST FX_NEXT FX_PUSH(K) FXB##K("a", "c0") FX_GO
#define FX_BODY_F(K)                                                                                                \
    FX_FUNC(K, "0", "add.rn.f32") FX_FUNC(K, "1", "sub.rn.f32") FX_FUNC(K, "2", "mul.rn.f32") FX_LONG(K, "3")        \
    "FXDV:\n\t" FX_FDIVS##K FX_GO FX_LEAVES(K) "FXEND:\n\tsub.u32 ip, ip, 8;\n\t"
#define FX_BODY_I(K)                                                                                                \
    FX_FUNC(K, "0", "add.u32") FX_FUNC(K, "1", "sub.u32") FX_FUNC(K, "2", "mul.lo.u32") FX_LONG(K, "3")              \
    "FXDV:\n\t" FX_IDIVS##K FX_GO FX_LEAVES(K) "FXEND:\n\tsub.u32 ip, ip, 8;\n\t"
#define FX_BODY_B(K)                                                                                                \
    FX_BFUNC(K, "0", "and.b32", "") FX_BFUNC(K, "1", "or.b32", "") FX_BFUNC(K, "2", "and.b32", FXN##K)               \
    FX_BFUNC(K, "3", "or.b32", FXN##K)                                                                               \
    "FXL1:\n\tadd.u32 t, oy, lo;\n\t" FX_NEXT FX_PUSH(K) FX_BLD(K, "a", "t") FX_GO                                   \
    "FXEND:\n\tsub.u32 ip, ip, 8;\n\t"

// Run the list at shared address `ip` up to an end mark; afterwards ip is
// where to go on from.  lo: the lane's offset in a row of the Boolean table.
template <int K, int V>
__device__ __forceinline__ void fx_exec(uint32_t& ip, float (&a)[K], uint32_t& sa, const float (&x)[K], uint32_t lo) {
    if constexpr (K == 1) {
#define FX_ASM1(TAB, BODY)                                                                                          \
    asm volatile("{\n\t" FX_REGS TAB "mov.b32 a0, %0;\n\tmov.b32 sa, %1;\n\tmov.b32 ip, %2;\n\t"                     \
                 "mov.b32 x0, %3;\n\tmov.b32 lo, %4;\n\t" FX_START BODY                                             \
                 "mov.b32 %0, a0;\n\tmov.b32 %1, sa;\n\tmov.b32 %2, ip;\n\t}"                                        \
                 : "+f"(a[0]), "+r"(sa), "+r"(ip) : "f"(x[0]), "r"(lo) : "memory")
        if constexpr (V == VF) FX_ASM1(FX_TABLE, FX_BODY_F(1));
        else if constexpr (V == VI) FX_ASM1(FX_TABLE, FX_BODY_I(1));
        else FX_ASM1(FX_BTABLE, FX_BODY_B(1));
    } else if constexpr (K == 2) {
#define FX_ASM2(TAB, BODY)                                                                                          \
    asm volatile("{\n\t" FX_REGS TAB "mov.b32 a0, %0;\n\tmov.b32 a1, %1;\n\tmov.b32 sa, %2;\n\tmov.b32 ip, %3;\n\t"  \
                 "mov.b32 x0, %4;\n\tmov.b32 x1, %5;\n\tmov.b32 lo, %6;\n\t" FX_START BODY                          \
                 "mov.b32 %0, a0;\n\tmov.b32 %1, a1;\n\tmov.b32 %2, sa;\n\tmov.b32 %3, ip;\n\t}"                     \
                 : "+f"(a[0]), "+f"(a[1]), "+r"(sa), "+r"(ip) : "f"(x[0]), "f"(x[1]), "r"(lo) : "memory")
        if constexpr (V == VF) FX_ASM2(FX_TABLE, FX_BODY_F(2));
        else if constexpr (V == VI) FX_ASM2(FX_TABLE, FX_BODY_I(2));
        else FX_ASM2(FX_BTABLE, FX_BODY_B(2));
    } else {
        static_assert(K == 4 && V == VF, "four cases per lane: binary32 only");
        asm volatile("{\n\t" FX_REGS FX_TABLE
                     "mov.b32 a0, %0;\n\tmov.b32 a1, %1;\n\tmov.b32 a2, %2;\n\tmov.b32 a3, %3;\n\tmov.b32 sa, %4;\n\t"
                     "mov.b32 ip, %5;\n\tmov.b32 x0, %6;\n\tmov.b32 x1, %7;\n\tmov.b32 x2, %8;\n\tmov.b32 x3, %9;\n\t"
                     "mov.b32 lo, %10;\n\t" FX_START FX_BODY_F(4)
                     "mov.b32 %0, a0;\n\tmov.b32 %1, a1;\n\tmov.b32 %2, a2;\n\tmov.b32 %3, a3;\n\tmov.b32 %4, sa;\n\t"
                     "mov.b32 %5, ip;\n\t}"
                     : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+r"(sa), "+r"(ip)
                     : "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "r"(lo) : "memory");
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
    float* g;            // global overflow: (maxd - W) entries x 32 lanes x K
    float x[K];          // the lane's inputs (binary32, integer)
};

// Leaf table of a CTA.  Binary32 and integer sets: the constants by opcode.
// Boolean sets: 16 rows by opcode (4.. the inputs) of the words of each case
// block, lane by lane, K words per lane; a row is 128 K bytes.
template <int K, int V>
struct FxTable {
    static constexpr int row = 32 * K * 4;                     // bytes of a Boolean row
    __host__ __device__ static uint32_t bytes(uint32_t ncb) { return V == VB ? FX_BROWS * row * ncb : 1024u; }
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
            for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) tab[i] = (i >= 5) ? consts[i - 5] : 0.0f;
        }
    }
};

// The list at ip on the checked path: entries from W on live in the global
// overflow area.  sa counts as on the fast path (it is only read through the
// window).  False when the stack is deeper than maxd.
template <int K, int V>
__device__ __forceinline__ bool fx_exec_checked(uint32_t& ip, float (&a)[K], uint32_t& sa, const FxCtx<K>& c) {
    constexpr uint32_t stride = 32 * K * 4;
    const int lane = lane_id();
    uint32_t dep = (sa - c.stack) / stride;
    bool ok = true;
    auto push = [&]() {
        if (dep < c.W) sts_vec<K>(c.stack + dep * stride, a);
        else if (dep < c.maxd) vstore<K>(c.g + ((size_t)(dep - c.W) * 32 + lane) * K, a);
        else ok = false;
        if (dep < c.maxd) ++dep;
    };
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
        if (idx >= FX_EXIT) break;
        float l[K], r[K];
        if (idx < 16u) {
            const bool ca = idx & 2u, cb = idx & 1u;
            push();
            leaf(ca && cb ? y & 0xFFFFu : y, ca, l);
            leaf(ca && cb ? y >> 16 : y, cb, r);
            apply_vec<K, V>(idx >> 2, l, r);
#pragma unroll
            for (int k = 0; k < K; ++k) a[k] = l[k];
        } else if (idx < 24u) {
            leaf(y, idx & 1u, l);
            apply_vec<K, V>((idx - 16u) >> 1, l, a);
#pragma unroll
            for (int k = 0; k < K; ++k) a[k] = l[k];
        } else if (idx < 28u) {
            if (dep) --dep;
            if (dep < c.W) lds_vec<K>(c.stack + dep * stride, r);
            else vload<K>(c.g + ((size_t)(dep - c.W) * 32 + lane) * K, r);
            apply_vec<K, V>(idx - 24u, a, r);
        } else {
            leaf(y, idx & 1u, l);
            push();
#pragma unroll
            for (int k = 0; k < K; ++k) a[k] = l[k];
        }
    }
    ip += 8;                       // past the end mark
    sa = c.stack + dep * stride;
    return ok;
}

// Evaluate the nodes [s, e): afterwards a holds the value of the subtree at
// s.  `ld(q)` reads the 32-bit word at position q (a multiple of 4); w0, w1
// are this lane's words of the last chunk and of the one to its left, read
// by the caller (fx_first), who can have them in flight early.  `stop`: a
// shared word that, once nonzero, ends the run early with *aborted set.
template <int K, int V, typename LD>
__device__ __forceinline__ bool fx_run(LD ld, uint32_t s, uint32_t e, uint32_t w0, uint32_t w1, const FxCtx<K>& c,
                                       float (&a)[K], const volatile uint32_t* stop = nullptr, bool* aborted = nullptr) {
    const int lane = lane_id();
    int32_t base = (int32_t)((e - 1) & ~(uint32_t)(FX_CHUNK - 1));
    FxCarry cy;
    cy.w = w0;
    cy.f = fx_funcs(w0);
    cy.rw = 0xFFFFFFFFu;
    cy.rf = 0u;
    cy.B = 0;
    uint32_t sa = c.stack, wl = w1;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = 0.f;
    for (;;) {
        if (stop && *stop) { *aborted = true; return true; }
        const uint32_t fl = fx_funcs(wl);
        const uint32_t wn = fx_word(ld, base - 2 * FX_CHUNK + 4 * lane, s, e);     // in flight during this chunk
        const FxChunk ch = fx_decode<V, false, FxTable<K, V>::row>(cy, fl, base, s, e, c.W, c.code, c.lt, 0u);
        if (ch.bad) { ok = false; break; }
        uint32_t ip = c.code;
        if (!ch.over) fx_exec<K, V>(ip, a, sa, c.x, c.lo);
        else ok &= fx_exec_checked<K, V>(ip, a, sa, c);
        __syncwarp();
        if (base <= (int32_t)s) break;
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
