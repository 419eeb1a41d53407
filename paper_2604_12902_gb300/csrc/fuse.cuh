// fuse.cuh -- fused instructions: runs of word-RASP instructions decoded once,
// when programs are loaded, and executed as one step of a lane's loop.
//
// What bounds the one-instruction loop (fast_loop_ptx): every VM-step fetches
// its own 16-byte pair and evaluates every guard of the Sec. 2.1 case equation
// (about 79 thread instructions and 1.5 L1 accesses per VM-step), and in long
// runs a step waits for its fetch, its operand and the guards in a row. As
// long as a VM has not written into its program words (Sec. 1.1's stored
// program; `Regs::clean`), none of that depends on its state: the opcode, the
// operand's range, the jump target and whether a jump on a constant is taken
// are known when the program is loaded.
//
// So a program is held as 16-byte entries. An entry is the longest run of
// instructions from one instruction on that fits the form
//
//   a <- imm1 | a <- a op M[j1], op = ADD or MUL (SUB), or y :: M[j1] (PRI) |
//   M[k] <- a (STO) or the next tape word (RD) | a <- imm2 | a <- a + M[j2] |
//   BNZ t, or, in the loop on 4-byte words, M[k2] <- a (STO)
//
// (every part optional, in this order) with jumps on constants followed. Only
// the entries that runs from instruction 0 can reach are kept, in instruction
// order (about half an entry per instruction, so that a loop of about ten
// VM-steps is two or three neighbouring entries); a bit mask per 64
// instructions maps between instructions and entries. The loads of M[j1] and
// M[j2] go out together. Every guard was resolved by the decoder:
// an instruction that could leave the common case -- invalid opcode, operand
// or target outside [0, n), odd target, a write into program words, BNZ to
// itself, i (+) 2 past the program, an immediate or address that does not fit
// -- ends the run before it, and an entry that would start with one is a stall
// (count 0). Two guards stay dynamic: the step countdown (an entry runs only
// if all of its VM-steps fit) and RD at the end of the tape. A lane that
// stalls applies nothing and keeps its place, so the loop needs no vote; the
// caller takes the general step (step_general) for such lanes together.
#pragma once

#include "engine.cuh"

namespace rasp {

// Entry: x = j1 | k << 16, y = j2 | flags << 16, z = imm1 | imm2 << 16
// (signed 16-bit), w = t | f << 16 (entries taken, next; while a program is
// decoded, instructions). A stall (count 0) holds its instruction in x.
enum : uint32_t {
  FO_COUNT = 0x001Fu << 16,   // VM-steps of the entry (0: stall)
  FO_L1 = 0x0020u << 16,      // a <- imm1
  FO_ADD = 0x0040u << 16,     // a <- a + M[j1]
  FO_MUL = 0x0080u << 16,     // a <- a * M[j1] (classic set: a - M[j1])
  FO_PRI = 0x0100u << 16,     // y :: M[j1]
  FO_STO = 0x0200u << 16,     // M[k] <- a
  FO_RD = 0x0400u << 16,      // M[k] <- next tape word
  FO_L2 = 0x0800u << 16,      // a <- imm2
  FO_LD2 = 0x1000u << 16,     // a <- a + M[j2]
  FO_FWD = 0x2000u << 16,     // a <- a + the value STO wrote (j2 = k)
  FO_BNZ = 0x4000u << 16,     // jump to t if the condition holds, else f
  FO_ST2 = 0x8000u << 16,     // M[t] <- a (no jump: t holds k2)
  FO_HALT = 0x8000u << 16,    // (stall) a fixed point: an invalid opcode
  FO_MEM = 0x4000u << 16,     // (stall, entry 0) the program mostly writes into itself: run it from memory
};
constexpr uint32_t kFuseMaxCount = 24;       // VM-steps per entry (a stop inside an entry is taken one step at a time)
constexpr uint32_t kFuseMaxInstr = 0xFFFFu;  // instructions of a program whose entries can be indexed

// Program words as the decoder reads them.
__device__ __forceinline__ ulonglong2 fuse_pair(const uint64_t* src, uint32_t k, uint64_t wmask) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(src + k);
  return make_ulonglong2(q.x & wmask, q.y & wmask);
}
__device__ __forceinline__ ulonglong2 fuse_pair(const int32_t* src, uint32_t k, uint64_t wmask) {
  const int2 q = *reinterpret_cast<const int2*>(src + k);
  return make_ulonglong2((uint64_t)(int64_t)q.x & wmask, (uint64_t)(int64_t)q.y & wmask);
}

// The scan of one run: instructions are taken as long as they fit. Its state is
// the next free part of the form (stage 0 imm1, 1 op, 2 store, 3 imm2, 4 add,
// 5 second store or jump) and a constant in a that is not yet placed.
// plen: words of the program; n: the smallest memory that runs it; mok:
// instructions whose pair and i (+) 2 need no reduction; own: M holds the
// program words (they may be read as data); two: entries may hold the second
// store. It takes the slowest loops of the halting workload from 3.1 to 4.0
// VM-steps per entry (run of 2^18 programs 121 -> 92 ms), and costs 6 of about
// 65 instructions on 8-byte words, where the template and uneven batches gain
// little from it (1.96 -> 2.05 ms).
struct FuseScan {
  uint32_t e, p, stage, cnt, flags, j1, k, j2, i1, i2, t, cv;
  bool pend, jump;      // a holds the constant cv (16 bits); a jump on it is taken

  __device__ __forceinline__ void start(uint32_t at) {
    e = p = at;
    stage = cnt = flags = j1 = k = j2 = i1 = i2 = cv = 0u;
    t = at;
    pend = jump = false;
  }

  // Take instruction (o, j) at p; false when the run has ended (at p).
  __device__ __forceinline__ bool step(uint64_t o, uint64_t j, uint32_t plen, uint32_t n, uint32_t mok,
                                       uint64_t wmask, bool classic, bool own, bool two) {
    const uint32_t op = o - 1ull < 7ull ? (uint32_t)o : 0u;
    const uint32_t jm = (uint32_t)j;
    const bool room = p + 1u < mok;
    bool ok = room, go = true;
    uint32_t np = p + 1u;
    if (op == 5u) {
      const bool target = !(jm & 1u) && (j >> 1) < (uint64_t)mok && jm != 2u * p;
      if (pend) {                                        // a is a constant: the jump is decided
        ok = jump ? target : room;
        np = jump ? jm >> 1 : np;
      } else {
        ok = target && room && !(flags & FO_ST2);
        if (ok) {
          flags |= FO_BNZ;
          t = jm >> 1;
        }
        go = false;
      }
    } else if (op == 1u) {
      const bool small = ((uint64_t)(int64_t)(int16_t)(uint16_t)j & wmask) == j;
      ok = room && stage <= 3u && (small || (own && 2u * p + 1u <= 0xFFFFu));
      if (ok) {
        pend = small;
        cv = jm & 0xFFFFu;
        jump = classic ? j - 1ull < (wmask >> 1) : j != 0ull;
        if (!small) {                                    // a wide constant: 0 + the program word itself
          const bool first = stage == 0u;
          flags |= first ? FO_L1 | FO_ADD : FO_L2 | FO_LD2;
          j1 = first ? 2u * p + 1u : j1;
          j2 = first ? j2 : 2u * p + 1u;
          stage = first ? 2u : 5u;
        }
      }
    } else {
      // parts that take an address, by opcode 2 ADD, 3 MUL, 4 STO, 6 RD, 7 PRI:
      // the last stage that may take it, the stage behind it, its flag; RD and
      // PRI do not use a, so a constant may wait past them
      const uint32_t at = 4u * op;
      const uint32_t last = (0x12021100u >> at) & 15u, behind = (0x23032200u >> at) & 15u;
      const uint32_t flag = op == 2u ? FO_ADD : op == 3u ? FO_MUL : op == 4u ? FO_STO : op == 6u ? FO_RD : FO_PRI;
      const bool code = jm < plen, store = op == 4u || op == 6u;
      const bool one = stage <= last && (!pend || stage == 0u || op >= 6u);
      const bool late = !one && stage <= (pend ? 3u : op == 2u ? 4u : 5u) &&
                        (op == 2u ? !((flags & FO_RD) && jm == k) : op == 4u && two);
      ok = room && op != 0u && j < (uint64_t)n && j <= 0xFFFFull && !(code && (store || !own)) && (one || late);
      if (ok) {
        if (pend && (one ? stage == 0u : true)) {        // the constant's place: imm1 while the form is empty
          flags |= one ? FO_L1 : FO_L2;
          i1 = one ? cv : i1;
          i2 = one ? i2 : cv;
          pend = false;
        }
        const uint32_t second = op == 4u ? FO_ST2 : ((flags & FO_STO) && jm == k ? FO_FWD : FO_LD2);
        flags |= one ? flag : second;
        j1 = one && !store ? jm : j1;
        k = one && store ? jm : k;
        j2 = !one && op == 2u ? jm : j2;
        t = !one && op == 4u ? jm : t;
        stage = one ? behind : (op == 2u ? 5u : 6u);
      }
    }
    if (ok) {
      p = np;
      cnt += 1u;
    }
    return ok && go && cnt < kFuseMaxCount;
  }

  // The entry, once the run has ended at an instruction of opcode o.
  __device__ __forceinline__ uint4 entry(uint64_t o) {
    if (!cnt) return make_uint4(e, o - 1ull >= 7ull ? FO_HALT : 0u, 0u, e | (e << 16));
    if (pend) {                                          // the constant that a holds after the run
      flags |= stage == 0u ? FO_L1 : FO_L2;
      i1 = stage == 0u ? cv : i1;
      i2 = stage == 0u ? i2 : cv;
    }
    return make_uint4(j1 | (k << 16), j2 | flags | (cnt << 16), i1 | (i2 << 16), t | (p << 16));
  }
};

// ------------------------------------------------------------------ the lane's side
// A VM's data view while it takes general steps beside the fused loop: a
// write into its program words is noticed (Regs::clean).
template <class Mem>
struct CodeView {
  Mem M;
  uint32_t plen;
};
template <class Mem>
__device__ __forceinline__ ulonglong2 mem_pair(const CodeView<Mem>& V, bool clean, uint32_t k) {
  return mem_pair(V.M, clean, k);
}
template <class Mem>
__device__ __forceinline__ uint64_t mem_rd(const CodeView<Mem>& V, bool clean, uint32_t k) {
  return mem_rd(V.M, clean, k);
}
template <class Mem>
__device__ __forceinline__ void mem_wr(CodeView<Mem>& V, bool& clean, uint32_t k, uint64_t v) {
  if (k < V.plen) clean = false;
  bool dummy = false;
  mem_wr(V.M, dummy, k, v);
}

// The records of program p (one per 64 instructions: x, y = the mask of the
// instructions with an entry, z = entries before them) start at record
// prog_off[p] / 128 + p, its entries at entry prog_off[p] / 2.
struct FuseProg {
  const uint4* tab;
  const uint4* rec;
  uint32_t plen, mok;   // program words; instructions that may have an entry
};
__host__ __device__ inline uint64_t fuse_records(uint64_t prog_words, uint64_t programs) {
  return prog_words / 128u + programs + 1u;
}
__device__ __forceinline__ uint64_t fuse_mask(uint4 r) { return ((uint64_t)r.y << 32) | r.x; }
__device__ __forceinline__ uint32_t fuse_rank(uint4 r, uint32_t e) {
  return r.z + (uint32_t)__popcll(fuse_mask(r) & ((1ull << (e & 63u)) - 1ull));
}

__device__ __forceinline__ FuseProg fuse_prog(const RunState& S, uint32_t v, uint32_t ilim) {
  const uint32_t p = S.prog_of_vm ? S.prog_of_vm[v] : v;
  const uint64_t po = S.prog_off[p];
  FuseProg G;
  G.plen = (uint32_t)(S.prog_off[p + 1] - po);
  G.mok = min(G.plen, ilim) >> 1;
  G.tab = S.fops + (po >> 1);
  G.rec = S.frec + (po >> 7) + p;
  return G;
}

// The entry of instruction e, or ~0.
__device__ __forceinline__ uint32_t fuse_find(const FuseProg& G, uint32_t e) {
  if (e >= G.mok) return ~0u;
  const uint4 r = G.rec[e >> 6];
  return (fuse_mask(r) >> (e & 63u)) & 1ull ? fuse_rank(r, e) : ~0u;
}

// The instruction of entry q (q below the number of entries).
__device__ __forceinline__ uint32_t fuse_instr(const FuseProg& G, uint32_t q) {
  uint32_t lo = 0, hi = (G.plen + 127u) / 128u;          // records with z <= q
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (G.rec[mid].z <= q) lo = mid;
    else hi = mid;
  }
  const uint4 r = G.rec[lo];
  uint64_t mask = fuse_mask(r);
  for (uint32_t k = q - r.z; k; --k) mask &= mask - 1ull;
  return 64u * lo + (uint32_t)__ffsll((long long)mask) - 1u;
}

// A lane's place in its program's entries.
struct Fused {
  const uint4* tab;     // the program's entries
  uint4 op;             // the entry at cur (when on)
  uint32_t cur;
  bool on;              // the VM runs from its entries (its i is the entry's instruction)
  uint32_t mark;        // Regs::left after its last general step
  uint32_t debt;        // VM-steps that its stalls have cost beyond those its entries ran (kFuseGone: it has left)
};
constexpr uint32_t kFuseGone = ~0u;

// The VM's next step needs the general path (or its run may stop here).
__device__ __forceinline__ bool fuse_stalled(const Fused& F, const Regs& r, const Params& P) {
  const uint32_t c = (F.op.y >> 16) & 31u;
  return c - 1u >= r.left || ((F.op.y & FO_RD) && r.u0 >= P.ell);
}

// A VM is taken: no stalls yet.
__device__ __forceinline__ void fuse_begin(Fused& F, const Regs& r) {
  F.mark = r.left;
  F.debt = 0u;
}

// Enter the entries at i if an entry starts there.
__device__ __forceinline__ void fuse_enter(const FuseProg& G, Fused& F, const Regs& r) {
  F.on = false;
  if (!r.clean || r.ibase != 0ull || (r.ip & 1u)) return;
  const uint32_t q = r.ip ? fuse_find(G, r.ip >> 1) : (G.mok ? 0u : ~0u);   // instruction 0 has entry 0
  if (q == ~0u) return;
  F.on = true;
  F.cur = q;
  F.tab = G.tab;
  F.op = G.tab[q];
}

// What fuse_attach reads of VM v before its registers are armed, so that a
// kernel can issue these loads beside the registers'.
struct FuseRow {
  uint64_t po, pe;      // the program's words
  uint32_t p;
  uint32_t dirty;
};
__device__ __forceinline__ FuseRow fuse_row(const RunState& S, uint32_t v) {
  FuseRow w;
  w.dirty = S.codedirty[v];
  w.p = S.prog_of_vm ? S.prog_of_vm[v] : v;
  w.po = S.prog_off[w.p];
  w.pe = S.prog_off[w.p + 1];
  return w;
}

// VM v's entries (after arm_regs); without them it runs one instruction at a time.
__device__ __forceinline__ void fuse_attach(const RunState& S, const FuseRow& w, Regs& r, Fused& F) {
  r.clean = w.dirty == 0u;
  FuseProg G;
  G.plen = (uint32_t)(w.pe - w.po);
  G.mok = min(G.plen, r.ilim) >> 1;
  G.tab = S.fops + (w.po >> 1);
  G.rec = S.frec + (w.po >> 7) + w.p;
  fuse_begin(F, r);
  fuse_enter(G, F, r);
  if (F.on && !(F.op.y & FO_COUNT) && (F.op.y & FO_MEM)) F.on = r.clean = false;
}

// `iters` (even) entries of every lane of `mask` (all of them call it together).
// Word sizes: 8-byte words of M and a 64-bit accumulator, or (narrow, w <= 32)
// 4-byte words and 32-bit arithmetic. Per entry: the dynamic guards (px, a
// lane that stalls clears its flags and so applies nothing), both loads, the
// parts of the form in order under their flags, then the next entry. RD and
// PRI (a few per program) are a side block that a warp vote skips.
//
// STO waits for both loads: its value is combined with (v1 | v2) & zero, a
// zero that the compiler cannot see. A store to a 128-byte line whose fill is
// still in flight makes the fill useless: the next load of that line misses
// again, and if the same store comes again before that fill has landed, the
// line never settles. Measured on one VM whose loop (4 entries, all words in
// one line) ran into this: 5,019 of 20,013 loads missed L1, 555 instead of
// 266 cycles per entry.
#define RASP_F_GUARD \
      "bfe.u32 c, %2, 16, 5;\n\t" \
      "add.u32 t0, c, -1;\n\t" \
      "setp.ge.u32 px, t0, %6;\n\t" \
      "and.b32 t0, %2, 0x04000000;\n\t" \
      "setp.ne.u32 pr, t0, 0;\n\t" \
      "setp.ge.and.u32 pr, %7, %14, pr;\n\t" \
      "or.pred px, px, pr;\n\t" \
      "selp.b32 ye, 0, %2, px;\n\t"
#define RASP_F_ADDR(B) \
      "and.b32 j, %1, 0xFFFF;\n\t" \
      "mad.wide.u32 ad1, j, " B ", %10;\n\t" \
      "and.b32 j, %2, 0xFFFF;\n\t" \
      "mad.wide.u32 ad2, j, " B ", %10;\n\t" \
      "shr.u32 j, %1, 16;\n\t" \
      "mad.wide.u32 ads, j, " B ", %10;\n\t" \
      "and.b32 t0, ye, 0x01C00000;\n\t" \
      "setp.ne.u32 p1, t0, 0;\n\t" \
      "and.b32 t0, ye, 0x10000000;\n\t" \
      "setp.ne.u32 p2, t0, 0;\n\t"
#define RASP_F_TEST(P, BIT) \
      "and.b32 t0, ye, " BIT ";\n\t" \
      "setp.ne.u32 " P ", t0, 0;\n\t"
// RD: M[k] <- u_(u_0 + 1), u_0 += 1; PRI: y :: M[j1] while y_0 < s
#define RASP_F_IO(LD, ST, V, TV) \
      RASP_F_TEST("pr", "0x05000000") \
      "vote.sync.any.pred pr, pr, %16;\n\t" \
      "@!pr bra.uni RASP_FNOIO;\n\t" \
      RASP_F_TEST("pr", "0x04000000") \
      "mad.wide.u32 ad1, %7, 8, %12;\n\t" \
      "@pr " LD " " TV ", [ad1];\n\t" \
      "@pr " ST " [ads], " TV ";\n\t" \
      "@pr add.u32 %7, %7, 1;\n\t" \
      RASP_F_TEST("pr", "0x01000000") \
      "setp.lt.and.u32 pr, %8, %15, pr;\n\t" \
      "mad.wide.u32 ad1, %8, 8, %13;\n\t" \
      "@pr " ST " [ad1], " V ";\n\t" \
      "@pr add.u32 %8, %8, 1;\n\t" \
      "RASP_FNOIO:\n\t"
// Entries are read by plain loads, not by ld.global.nc: the serving kernel
// stays resident while the entries of new requests are written where those of
// finished ones lay, and what it reads after claiming a VM has to be ordered by
// its fence.
// Both entries that may come next are loaded beside the operands (f into the
// entry's own registers, whose fields have been taken apart by then), so that
// an entry waits for one round of loads and not for two in a row.
#define RASP_F_AHEAD(FETCH) \
      "shr.s32 i2, %3, 16;\n\t" \
      "and.b32 jt, %4, 0xFFFF;\n\t" \
      "shr.u32 jf, %4, 16;\n\t" \
      RASP_F_TEST("pb", "0x40000000") \
      FETCH
#define RASP_F_FETCH_GL \
      "mad.wide.u32 ad1, jf, 16, %11;\n\t" \
      "mad.wide.u32 ad2, jt, 16, %11;\n\t" \
      "@!px ld.global.v4.u32 {%1, %2, %3, %4}, [ad1];\n\t" \
      "@pb ld.global.v4.u32 {tx, ty, tz, tw}, [ad2];\n\t"
// entries in shared memory (%11 = their 32-bit address)
#define RASP_F_FETCH_SH \
      "mad.lo.u32 t0, jf, 16, %11;\n\t" \
      "mad.lo.u32 j, jt, 16, %11;\n\t" \
      "@!px ld.shared.v4.u32 {%1, %2, %3, %4}, [t0];\n\t" \
      "@pb ld.shared.v4.u32 {tx, ty, tz, tw}, [j];\n\t"
// the next entry, and the VM-steps of this one
#define RASP_F_NEXT \
      "selp.b32 j, jt, jf, pt;\n\t" \
      "@!px mov.b32 %5, j;\n\t" \
      "@!px sub.u32 %6, %6, c;\n\t" \
      "@pt mov.b32 %1, tx;\n\t" \
      "@pt mov.b32 %2, ty;\n\t" \
      "@pt mov.b32 %3, tz;\n\t" \
      "@pt mov.b32 %4, tw;\n\t" \
      "}"
#define RASP_F_LOOP1(BODY) \
      BODY \
      "add.u32 it, it, -1;\n\t" \
      "setp.ne.u32 p1, it, 0;\n\t" \
      "@p1 bra.uni RASP_FLOOP;\n\t" \
      "}"
// two entries per turn (iters is even): 0.81 -> 0.79 ms for the entries in
// shared memory, slower for the others (2^20 templates 1.98 -> 2.18 ms)
#define RASP_F_LOOP2(BODY) \
      BODY BODY \
      "add.u32 it, it, -2;\n\t" \
      "setp.ne.u32 p1, it, 0;\n\t" \
      "@p1 bra.uni RASP_FLOOP;\n\t" \
      "}"
#define RASP_F_REGS \
      ".reg .pred px, pr, p1, p2, pt, pb;\n\t" \
      ".reg .b32 c, t0, ye, j, it, zz, jt, jf, i2, tx, ty, tz, tw;\n\t" \
      ".reg .b64 ad1, ad2, ads;\n\t"

// 8-byte words. %17 = 2^w - 1 (masked), %18 = its half (classic condition).
#define RASP_FW_HEAD "{\n\t" RASP_F_REGS ".reg .b64 v1, v2, im;\n\t" "mov.b32 it, %9;\n\tRASP_FLOOP:\n\t"
#define RASP_FW_A(FETCH) \
      "{\n\t" RASP_F_GUARD RASP_F_ADDR("8") \
      "@p1 ld.global.u64 v1, [ad1];\n\t" \
      "@p2 ld.global.u64 v2, [ad2];\n\t" \
      "cvt.s32.s16 t0, %3;\n\t" \
      "cvt.s64.s32 im, t0;\n\t" \
      RASP_F_AHEAD(FETCH) \
      RASP_F_TEST("p1", "0x00200000") \
      "@p1 mov.b64 %0, im;\n\t" \
      RASP_F_TEST("p1", "0x00400000") \
      "@p1 add.u64 %0, %0, v1;\n\t" \
      RASP_F_TEST("p1", "0x00800000")
#define RASP_FW_MUL "@p1 mul.lo.u64 %0, %0, v1;\n\t"
#define RASP_FW_SUB "@p1 sub.u64 %0, %0, v1;\n\t"
#define RASP_FW_MASK "and.b64 %0, %0, %17;\n\t"
#define RASP_FW_B \
      RASP_F_TEST("p1", "0x02000000") \
      "cvt.u32.u64 t0, v1;\n\t" \
      "cvt.u32.u64 j, v2;\n\t" \
      "lop3.b32 zz, t0, j, %19, 0xA8;\n\t" \
      "cvt.u64.u32 im, zz;\n\t" \
      "xor.b64 im, im, %0;\n\t" \
      "@p1 st.global.u64 [ads], im;\n\t" \
      RASP_F_IO("ld.global.u64", "st.global.u64", "v1", "im") \
      RASP_F_TEST("p1", "0x20000000") \
      "@p1 mov.b64 v2, %0;\n\t" \
      "cvt.s64.s32 im, i2;\n\t" \
      RASP_F_TEST("p1", "0x08000000") \
      "@p1 mov.b64 %0, im;\n\t" \
      RASP_F_TEST("p1", "0x30000000") \
      "@p1 add.u64 %0, %0, v2;\n\t"
#define RASP_FW_PT_WORD \
      "setp.ne.and.u64 pt, %0, 0, pb;\n\t"
#define RASP_FW_PT_CLASSIC \
      "add.u64 im, %0, -1;\n\t" \
      "setp.lt.and.u64 pt, im, %18, pb;\n\t"
#define RASP_FW_OPERANDS(TAB) \
  : "+l"(a), "+r"(F.op.x), "+r"(F.op.y), "+r"(F.op.z), "+r"(F.op.w), "+r"(F.cur), "+r"(left), "+r"(u0), "+r"(y0) \
  : "r"(iters), "l"(M), TAB, "l"(T), "l"(Y), "r"(ell), "r"(s), "r"(mask), "l"(wmask),                    \
    "l"(wmask >> 1), "r"(zero)                                                                                   \
  : "memory"

template <bool MASKED, bool CLASSIC>
__device__ __forceinline__ void fused_loop_ptx(uint64_t* M, const uint64_t* T, uint64_t* Y, uint32_t ell, uint32_t s,
                                               uint64_t wmask, uint32_t mask, uint32_t iters, uint32_t zero,
                                               uint64_t& a, Fused& F, uint32_t& left, uint32_t& u0, uint32_t& y0) {
  if constexpr (MASKED && CLASSIC) {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP1(
        RASP_FW_A(RASP_F_FETCH_GL) RASP_FW_SUB RASP_FW_MASK RASP_FW_B RASP_FW_MASK RASP_FW_PT_CLASSIC
        RASP_F_NEXT)
                 RASP_FW_OPERANDS("l"(F.tab)));
  } else if constexpr (MASKED) {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP1(
        RASP_FW_A(RASP_F_FETCH_GL) RASP_FW_MUL RASP_FW_MASK RASP_FW_B RASP_FW_MASK RASP_FW_PT_WORD
        RASP_F_NEXT)
                 RASP_FW_OPERANDS("l"(F.tab)));
  } else if constexpr (CLASSIC) {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP1(
        RASP_FW_A(RASP_F_FETCH_GL) RASP_FW_SUB RASP_FW_B RASP_FW_PT_CLASSIC RASP_F_NEXT)
                 RASP_FW_OPERANDS("l"(F.tab)));
  } else {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP1(RASP_FW_A(RASP_F_FETCH_GL) RASP_FW_MUL RASP_FW_B RASP_FW_PT_WORD RASP_F_NEXT)
                 RASP_FW_OPERANDS("l"(F.tab)));
  }
}

// The entries of a shared program in shared memory (word opcode set).
template <bool MASKED>
__device__ __forceinline__ void fused_loop_ptx_sh(uint64_t* M, uint32_t tab, const uint64_t* T, uint64_t* Y,
                                                  uint32_t ell, uint32_t s, uint64_t wmask, uint32_t mask,
                                                  uint32_t iters, uint32_t zero, uint64_t& a, Fused& F,
                                                  uint32_t& left, uint32_t& u0, uint32_t& y0) {
  if constexpr (MASKED) {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP2(
        RASP_FW_A(RASP_F_FETCH_SH) RASP_FW_MUL RASP_FW_MASK RASP_FW_B RASP_FW_MASK RASP_FW_PT_WORD
        RASP_F_NEXT)
                 RASP_FW_OPERANDS("r"(tab)));
  } else {
    asm volatile(RASP_FW_HEAD RASP_F_LOOP2(RASP_FW_A(RASP_F_FETCH_SH) RASP_FW_MUL RASP_FW_B RASP_FW_PT_WORD RASP_F_NEXT)
                 RASP_FW_OPERANDS("r"(tab)));
  }
}

// 4-byte words (w <= 32). Tape words and outputs are 8-byte words whose high
// halves are zero. %17 = 2^w - 1, %18 = its half.
#define RASP_FN_HEAD "{\n\t" RASP_F_REGS ".reg .b32 v1, v2, im;\n\t" "mov.b32 it, %9;\n\tRASP_FLOOP:\n\t"
#define RASP_FN_A(FETCH) \
      "{\n\t" RASP_F_GUARD RASP_F_ADDR("4") \
      "@p1 ld.global.u32 v1, [ad1];\n\t" \
      "@p2 ld.global.u32 v2, [ad2];\n\t" \
      "cvt.s32.s16 im, %3;\n\t" \
      RASP_F_AHEAD(FETCH) \
      RASP_F_TEST("p1", "0x00200000") \
      "@p1 mov.b32 %0, im;\n\t" \
      RASP_F_TEST("p1", "0x00400000") \
      "@p1 add.u32 %0, %0, v1;\n\t" \
      RASP_F_TEST("p1", "0x00800000")
#define RASP_FN_MUL "@p1 mul.lo.u32 %0, %0, v1;\n\t"
#define RASP_FN_SUB "@p1 sub.u32 %0, %0, v1;\n\t"
#define RASP_FN_MASK "and.b32 %0, %0, %17;\n\t"
#define RASP_FN_B \
      RASP_F_TEST("p1", "0x02000000") \
      "lop3.b32 zz, v1, v2, %19, 0xA8;\n\t" \
      "xor.b32 t0, zz, %0;\n\t" \
      "@p1 st.global.u32 [ads], t0;\n\t" \
      RASP_F_IO("ld.global.u32", "st.global.u32", "v1", "im") \
      RASP_F_TEST("p1", "0x20000000") \
      "@p1 mov.b32 v2, %0;\n\t" \
      RASP_F_TEST("p1", "0x08000000") \
      "@p1 mov.b32 %0, i2;\n\t" \
      RASP_F_TEST("p1", "0x30000000") \
      "@p1 add.u32 %0, %0, v2;\n\t"
#define RASP_FN_ST2 \
      "mad.wide.u32 ads, jt, 4, %10;\n\t" \
      "setp.lt.s32 p1, ye, 0;\n\t" \
      "xor.b32 t0, zz, %0;\n\t" \
      "@p1 st.global.u32 [ads], t0;\n\t"
#define RASP_FN_PT_WORD \
      "setp.ne.and.u32 pt, %0, 0, pb;\n\t"
#define RASP_FN_PT_CLASSIC \
      "add.u32 im, %0, -1;\n\t" \
      "setp.lt.and.u32 pt, im, %18, pb;\n\t"
#define RASP_FN_OPERANDS \
  : "+r"(a), "+r"(F.op.x), "+r"(F.op.y), "+r"(F.op.z), "+r"(F.op.w), "+r"(F.cur), "+r"(left), "+r"(u0), "+r"(y0) \
  : "r"(iters), "l"(M), "l"(F.tab), "l"(T), "l"(Y), "r"(ell), "r"(s), "r"(mask), "r"(wmask),                    \
    "r"(wmask >> 1), "r"(zero)                                                                                   \
  : "memory"

// MASK: w < 32.
template <bool MASK, bool CLASSIC>
__device__ __forceinline__ void fused_loop_ptx_narrow(uint32_t* M, const uint64_t* T, uint64_t* Y, uint32_t ell,
                                                      uint32_t s, uint32_t wmask, uint32_t mask, uint32_t iters,
                                                      uint32_t zero, uint32_t& a, Fused& F, uint32_t& left,
                                                      uint32_t& u0, uint32_t& y0) {
  if constexpr (MASK && CLASSIC) {
    asm volatile(RASP_FN_HEAD RASP_F_LOOP1(
        RASP_FN_A(RASP_F_FETCH_GL) RASP_FN_SUB RASP_FN_MASK RASP_FN_B RASP_FN_MASK RASP_FN_ST2 RASP_FN_PT_CLASSIC
        RASP_F_NEXT)
                 RASP_FN_OPERANDS);
  } else if constexpr (MASK) {
    asm volatile(RASP_FN_HEAD RASP_F_LOOP1(
        RASP_FN_A(RASP_F_FETCH_GL) RASP_FN_MUL RASP_FN_MASK RASP_FN_B RASP_FN_MASK RASP_FN_ST2 RASP_FN_PT_WORD
        RASP_F_NEXT)
                 RASP_FN_OPERANDS);
  } else if constexpr (CLASSIC) {
    asm volatile(RASP_FN_HEAD RASP_F_LOOP1(
        RASP_FN_A(RASP_F_FETCH_GL) RASP_FN_SUB RASP_FN_B RASP_FN_ST2 RASP_FN_PT_CLASSIC
        RASP_F_NEXT)
                 RASP_FN_OPERANDS);
  } else {
    asm volatile(RASP_FN_HEAD RASP_F_LOOP1(
        RASP_FN_A(RASP_F_FETCH_GL) RASP_FN_MUL RASP_FN_B RASP_FN_ST2 RASP_FN_PT_WORD
        RASP_F_NEXT)
                 RASP_FN_OPERANDS);
  }
}

}  // namespace rasp
