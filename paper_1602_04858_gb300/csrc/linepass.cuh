// linepass.cuh -- several colour passes of the multiplicative Schwarz smoother
// (Sec. 3.3) in one launch: the passes of one class of vertex lines.
//
// Colours are digits (v_x mod 3, v_y mod 3 [, v_z mod 3]).  Patches whose
// vertices differ by three or more cells in any direction neither share dofs
// nor couple, so for a fixed class of the cross digits the lines of vertices
// along x are independent of one another whatever the order of the x digits.
// A symmetric step visits the colours in an order that changes the x digit
// fastest, so its 2 3^d - 1 passes fall into runs of three to five passes of
// one class (0 1 2 | 3 4 5 | 6 7 8 7 6 | 5 4 3 | 2 1 0 1 2 | ...).  One launch
// runs a whole run: a thread-block cluster owns a line, each block a segment of
// its vertices, and the passes are ordered inside the launch instead of by
// dependent launches.
//
// A block keeps its strip of the line in shared memory for the whole launch:
// the window rows of x around the line, the patch rows of b and the cell
// coefficients, each row contiguous along x.  A patch's window is then the same
// set of strip offsets for every patch of the line, shifted by (K + 1) elements
// per vertex, so nothing is gathered per patch; only the inverses S_v stream
// through (cp.async.bulk, two or three buffers per team).  Updates within two
// vertices of a segment's end are also stored into the neighbour block's strip
// (distributed shared memory).
//
// A team of LW lanes owns a patch (several patches per warp where LW < 32):
//   1. local residual from the lane plan: two neighbouring lanes share a long
//      velocity row (one shuffle adds their parts), a lane any other row; plain
//      slots (coefficient x strip entry) and mass slots, which all belong to one
//      cell and are summed before the multiplication by its coefficient.  The
//      positions of a row's entries are the same for every patch of the line;
//      the patches at its ends only have other coefficients;
//   2. delta = S_v r: lane (row group g, part s) takes the columns s, s + SPL,
//      ...; FP32: the parts are reduced and scattered by shuffles so that lane l
//      ends with row l; elsewhere through shared memory, FP64 with groups of
//      rows that keep more lanes on its units.  Every warp of a team reads the
//      whole r, and on the shuffle path nothing orders the team's warps after
//      that: the residuals of a team of several warps take turns in two buffers,
//      so that the one a warp writes for the next patch is not the one a slower
//      warp still reads, and the barrier of that next patch orders the one after;
//   3. x|_v += delta in the strip.
//
// A warp beside the teams streams the inverses: it refills a buffer as soon as
// the team has released it, across pass boundaries.  The blocks of a line send
// their updates with st.async, which completes the bytes on a barrier of the
// receiver: a pass waits for exactly the neighbour updates it needs and no fence
// is executed (a cluster barrier or a release with copies in flight took 1,000 to
// 1,500 clocks per pass).  What bounds it: on the finest level the inverses' bytes
// (25 bytes per clock and SM), on coarse ones the chain of one patch update and
// of the launch.  Measured per colour pass (GB300, passes back to back, us), colour
// passes and line sweeps: 2-D RT_1 FP32 256^2 10.6 and 7.2, 128^2 3.6 and 2.7, 64^2 2.23
// and 1.74; FP64 256^2 58.6 and 49.3; BF16 192^2 6.5 and 4.8; RT_2 FP32 128^2 23.3 and
// 14.9; 3-D RT_0 FP32 64^3 7.9 and 4.5; RT_0 512^2 5.6 and 4.1.
#pragma once

#include "passplan.cuh"

namespace mgd {

// Lanes per patch (LW) and slots per lane: Z0 plain and ZM mass slots of the
// lane's first row, Z1 plain slots of a pressure row.  A velocity row of a node
// shared by two cells along the component's direction takes GS lanes, any other
// one lane, a pressure row GP (the second piece of one lane where GP = 0 or no
// lane is left).  One warp per patch (RT_2: three) leaves least work outside the
// slots; plans over 64 to 384 lanes, with a shorter chain of dependent work per
// patch, were slower on every level measured (2-D RT_1 64^2: 2.24 against 1.74 us
// per pass; RT_2 128^2: 22.9 against 14.9).
template <int D, int K> struct LinePlan;
template <> struct LinePlan<2, 0> {   // 4 shared rows of at most 11 + 4 entries, 4 pressure rows of 4
  static constexpr int LW = 8, Z0 = 6, ZM = 2, Z1 = 4, GS = 2, GP = 0;
};
template <> struct LinePlan<2, 1> {   // 8 shared rows of 34 + 6, 16 others of 20 + 3, 16 pressure rows of 6
  static constexpr int LW = 32, Z0 = 20, ZM = 3, Z1 = 6, GS = 2, GP = 0;
};
template <> struct LinePlan<2, 2> {   // 12 shared rows of 69 + 8, 48 others of 39 + 4, 36 pressure rows of 8
  static constexpr int LW = 96, Z0 = 39, ZM = 4, Z1 = 8, GS = 2, GP = 1;
};
template <> struct LinePlan<3, 0> {   // 12 shared rows of 17 + 4, 8 pressure rows of 6
  static constexpr int LW = 32, Z0 = 9, ZM = 2, Z1 = 0, GS = 2, GP = 1;
};

constexpr int LINE_MAX_SUB = 5;   // passes of a run

// Strip rows.  x rows in the order u_0, u_1, .., p, within a component the
// window's cross positions (y fastest); b rows likewise over the patch's cross
// positions; c rows the 2^(d-1) cell rows of the patch.
template <int D, int K>
struct LineRows {
  static constexpr int K1 = K + 1, WA = 2 * K1 + 1, WB = 4 * K1, WP = 2 * K1, UA = 2 * K + 1, UB = 2 * K + 2;
  // extent of the window (patch) of component c along the cross direction e
  static constexpr int wext(int c, int e) { return c == D ? WP : (c == e ? WA : WB); }
  static constexpr int uext(int c, int e) { return c < D && c == e ? UA : UB; }
  static constexpr int xrows(int c) { return D == 2 ? wext(c, 1) : wext(c, 1) * wext(c, D - 1); }
  static constexpr int brows(int c) { return D == 2 ? uext(c, 1) : uext(c, 1) * uext(c, D - 1); }
  static constexpr int xfirst(int c) { return c == 0 ? 0 : xfirst(c - 1) + xrows(c - 1); }
  static constexpr int bfirst(int c) { return c == 0 ? 0 : bfirst(c - 1) + brows(c - 1); }
  static constexpr int XROWS = xfirst(D) + xrows(D), BROWS = bfirst(D) + brows(D), CROWS = 1 << (D - 1);
};

// x row r of the line at cross vertex (v[1], .., v[D-1]): component and flat
// index of its node at x node 0; false if the row lies outside the domain.
template <int D, int K, typename T>
__host__ __device__ __forceinline__ bool line_xrow(const Lvl<D, K, T>& L, const int (&v)[D], int r, int& comp,
                                                   int64_t& base) {
  using R = LineRows<D, K>;
  constexpr int K1 = K + 1;
  comp = D;
#pragma unroll
  for (int c = D - 1; c >= 0; --c)
    if (r < R::xfirst(c + 1)) comp = c;
  int q = r;
#pragma unroll
  for (int c = 0; c <= D; ++c)
    if (comp == c) q = r - R::xfirst(c);
  bool ok = true;
  int64_t st = (comp == 0) ? L.N + 1 : L.N;
  base = L.off[0];
#pragma unroll
  for (int c = 1; c <= D; ++c)
    if (comp == c) base = L.off[c];
#pragma unroll
  for (int e = 1; e < D; ++e) {
    const int ext = comp == D ? R::WP : (comp == e ? R::WA : R::WB);
    const int le = (e == D - 1) ? q : q % ext;
    q /= ext;
    const int t = ((comp < D && comp != e) ? v[e] - 2 : v[e] - 1) * K1 + le;
    const int hi = comp == e ? L.N : L.N - 1;
    ok = ok && t >= 0 && t <= hi;
    base += (int64_t)t * st;
    st *= (comp == e) ? L.N + 1 : L.N;
  }
  return ok;
}

// b row r: its component, the x row that holds the same nodes, and the flat
// index at x node 0 (always inside the domain).
template <int D, int K, typename T>
__host__ __device__ __forceinline__ void line_brow(const Lvl<D, K, T>& L, const int (&v)[D], int r, int& comp,
                                                   int& xrow, int64_t& base) {
  using R = LineRows<D, K>;
  constexpr int K1 = K + 1;
  comp = D;
#pragma unroll
  for (int c = D - 1; c >= 0; --c)
    if (r < R::bfirst(c + 1)) comp = c;
  int q = r, xr = 0;
  int64_t bs = L.off[0];
#pragma unroll
  for (int c = 0; c <= D; ++c)
    if (comp == c) {
      q = r - R::bfirst(c);
      xr = R::xfirst(c);
      bs = L.off[c];
    }
  int64_t st = (comp == 0) ? L.N + 1 : L.N;
  int ws = 1;
#pragma unroll
  for (int e = 1; e < D; ++e) {
    const bool own = comp == e;
    const int ue = own ? R::UA : R::UB, we = comp == D ? R::WP : (own ? R::WA : R::WB);
    const int le = (e == D - 1) ? q : q % ue;
    q /= ue;
    const int t = (v[e] - 1) * K1 + le + (own ? 1 : 0);
    const int w0 = ((comp < D && !own) ? v[e] - 2 : v[e] - 1) * K1;
    xr += (t - w0) * ws;
    ws *= we;
    bs += (int64_t)t * st;
    st *= own ? L.N + 1 : L.N;
  }
  xrow = xr;
  base = bs;
}

// Strip position of a window column: row << 16 | column relative to the patch
// (the strip's first node is that of cell a - 2 for a segment starting at
// vertex a; a patch at vertex v adds (v - a)(K + 1)).
template <int D, int K>
inline int line_pos(int w) {
  using R = LineRows<D, K>;
  constexpr int K1 = K + 1;
  constexpr int WU = (D == 2) ? R::WA * R::WB : R::WA * R::WB * R::WB;
  const int c = std::min(w / WU, D), l = w - c * WU;
  const int e0 = c == D ? R::WP : (c == 0 ? R::WA : R::WB);
  return ((R::xfirst(c) + l / e0) << 16) | (l % e0 + ((c == 0 || c == D) ? K1 : 0));
}

// Strip rows have a pitch of this remainder modulo 32 entries: the bank of an
// entry then does not depend on the segment's length, and the tables order the
// entries for it.
template <int D, int K>
constexpr int line_pitch_rem() { return (K + 1) * (D == 2 ? 2 : 4) + 1; }
template <int D, int K>
constexpr int line_pitch(int entries) { return (entries + 31 - line_pitch_rem<D, K>()) / 32 * 32 + line_pitch_rem<D, K>(); }

// Lanes of one residual row: its first lane, their number (a power of two that
// the first lane is a multiple of) and the piece that holds its entries.
struct LineRow { int row, lane, lanes, piece; };

// Rows of a patch in lane order: shared velocity rows, the others, pressure rows.
template <int D, int K>
inline std::vector<LineRow> line_rows() {
  using PS = PatchShape<D, K>;
  using PL = LinePlan<D, K>;
  std::vector<LineRow> out;
  int v[D], idx[D], lane = 0, second = 0;
  for (int e = 0; e < D; ++e) v[e] = 2;
  for (int kind = 0; kind < 3; ++kind)
    for (int l = 0; l < PS::NV; ++l) {
      const int comp = patch_local_decode<D, K>(v, l, idx);
      if ((comp == D ? 2 : (idx[comp] % (K + 1) == 0 ? 0 : 1)) != kind) continue;
      const int n = kind == 0 ? PL::GS : (kind == 1 ? 1 : PL::GP);
      if (n == 0 || lane + n > PL::LW) {   // second pieces of the last lanes (with first pieces) or of the first ones
        out.push_back({l, (n == 0 ? 0 : PL::LW - 32) + second++, 1, 1});
      } else {
        out.push_back({l, lane, n, 0});
        lane += n;
      }
    }
  return out;
}

template <int D, int K, typename T, typename TS, int NR = 1>
struct LineShape {
  using PS = PatchShape<D, K>;
  using PL = LinePlan<D, K>;
  using R = LineRows<D, K>;
  using SL = SLayout<PS::NV, TS>;
  static constexpr int NV = PS::NV, NU = D * PS::NU1, K1 = K + 1, RG = SL::RG, NVP = SL::NVP;
  static constexpr int LW = PL::LW, Z0 = PL::Z0, ZM = PL::ZM, Z1 = PL::Z1, ZP = Z0 + Z1, NS = ZP + ZM;
  static constexpr int GMAX = PL::GS;                        // most lanes of a row
  static constexpr int GPW = LW < 32 ? 32 / LW : 1;          // patches per team
  static constexpr int TW = LW < 32 ? 1 : LW / 32;           // warps per team
  static constexpr int TT = 32 * TW;                         // threads per team
  static constexpr bool BF = std::is_same<TS, __nv_bfloat16>::value;
  // product: lane (group of PR rows, column part).  SHF: a power of two parts,
  // at least as many as rows of a group, reduced and scattered by shuffles;
  // otherwise the parts are added through shared memory.  FP32 reads RG rows (16
  // bytes) at once; FP64 takes the group size that leaves fewest lanes idle
  static constexpr int p2(int v) { return v >= 32 ? 32 : v >= 16 ? 16 : v >= 8 ? 8 : v >= 4 ? 4 : v >= 2 ? 2 : 1; }
  static constexpr bool SHF = sizeof(T) == 4 && NVP <= LW;
  static constexpr int PR = sizeof(T) == 4 ? RG : (K == 1 ? 5 : (K == 2 ? 4 : 2));
  static constexpr int LPP = (sizeof(T) == 4 ? NVP : NV) / PR;
  static constexpr int SPL = SHF ? p2(LW / LPP) : LW / LPP;
  static constexpr int JCH = (NV + SPL - 1) / SPL;
  static constexpr int NIT = SHF ? 1 : (NV + LW - 1) / LW;   // rows per lane of the update
  // largest block (without the copying warp): what the inverse buffers leave
  // room for, and registers for the plan
  static constexpr int MAXT = K == 2 ? (sizeof(T) == 4 ? 288 : 192) : (K == 1 ? (sizeof(T) == 4 && NR == 1 ? 384 : 256) : 512);
  // 3-D RT_0 in FP32 with one right-hand side comes in two forms: with the registers
  // of one of the largest blocks on an SM (96: all its loads in flight at once;
  // 16^3 1.02 us a pass, 32^3 1.59) and with those of two (56, more lines at once;
  // 1.15, 1.44).  2-D RT_0 is faster with 96 throughout (512^2 4.0 against 4.8)
  static constexpr bool LEAN = D == 3 && K == 0 && sizeof(T) == 4 && NR == 1;
  // clocks of an SM that one item (GPW patches) takes of its busiest unit besides
  // the copies: shared-memory wavefronts, or the FP64 units (two FMAs per clock)
  static constexpr int WORK = sizeof(T) == 8 ? 16 * TW * NR * (NS + JCH * PR + 10)
                                             : TW * (NS * (NR == 1 ? 7 : 16) / 4 + JCH * (RG * (int)sizeof(TS) / 4 + 1) + 20 * NR);
  // scratch per patch (T): residual ((r, r) pairs with one FP32 right-hand side), twice where
  // only one barrier an item orders several warps; FP64 partial sums
  static constexpr int RP = (sizeof(T) == 4 && NR == 1) ? 2 : NR;
  static constexpr int RVS = (NV * RP + 3) / 4 * 4, RVN = SHF && TW > 1 ? 2 : 1;
  static constexpr int O_D = RVN * RVS;
  static constexpr int SCR = O_D + (SHF ? 0 : (SPL * LPP * PR * NR + 3) / 4 * 4);
  static constexpr int S_BYTES = (int)(SL::STRIDE * sizeof(TS)), SC_BYTES = BF ? NVP * 4 : 0;
  static constexpr int BUF = ((GPW * (S_BYTES + SC_BYTES) + 127) / 128) * 128;   // one inverse buffer
  // tables (level): positions [cross type][slot][lane] of the plain then the
  // mass entries, cells [cross type][lane], coefficients [type][slot][lane] in
  // the same order, row positions [row] (x strip, b strip), lanes [lane] (int2:
  // first row | lanes << 16, second row; -1 where the lane writes none)
  static constexpr int NX = D == 2 ? 4 : 16, NTYPE = 4 * NX;
  static constexpr size_t a16(size_t b) { return (b + 15) / 16 * 16; }
  static constexpr size_t TB_POS = 0;
  static constexpr size_t TB_CELL = TB_POS + a16((size_t)NX * NS * LW * 4);
  static constexpr size_t TB_COEF = TB_CELL + a16((size_t)NX * LW * 4);
  static constexpr size_t TB_ROW = TB_COEF + a16((size_t)NTYPE * NS * LW * sizeof(T));
  static constexpr size_t TB_LANE = TB_ROW + a16((size_t)NV * 8);
  // strip rows (int4): flat index of x node 0 as e.x + e.y v_1 + e.z v_2, then
  // for x rows the cross positions outside the domain (bits 0, 1: v_1 = 1, n - 1;
  // bits 2, 3: v_2), for b rows the x row of the same nodes << 4
  static constexpr size_t TB_STRIP = TB_LANE + a16((size_t)LW * 8);
  static constexpr size_t TAB_BYTES = TB_STRIP + (size_t)(R::XROWS + R::BROWS) * 16;
  // the coefficients of the patches at the line's ends: in shared memory, or
  // read from the table where they are too many (RT_2)
  static constexpr bool ENDS = K < 2;
  static constexpr int END_N = ENDS ? NS * LW : 0;
  // shared memory: x, b and c strips, end coefficients, team scratch, row bases, inverse buffers, mbarriers
  static constexpr int IROWS = (R::XROWS + 2 * R::BROWS + 1 + 3) / 4 * 4;
  // mbarriers: copies landed and buffers free per team and buffer, then for each
  // neighbour (left, right) its strip loaded and its updates of each pass
  struct Smem { int scr, rows, buf, bars; size_t bytes; };
  static __host__ __device__ Smem layout(int PX, int PC, int teams, int nsb) {
    Smem m;
    const int strips = ((R::XROWS + R::BROWS) * PX * NR + R::CROWS * PC + 2 * END_N) * (int)sizeof(T);
    m.scr = (strips + 15) / 16 * 16;
    m.rows = m.scr + teams * GPW * SCR * (int)sizeof(T);
    m.buf = (m.rows + IROWS * 4 + 127) / 128 * 128;
    m.bars = m.buf + teams * nsb * BUF;
    m.bytes = (size_t)m.bars + (size_t)(2 * teams * nsb + 2 * (1 + LINE_MAX_SUB)) * 8 + 16;
    return m;
  }
  static constexpr int RT = sizeof(T) == 4 ? NVP : NV;
  static_assert(LPP * SPL <= LW && SPL >= 1 && LPP * PR >= NV, "row groups x parts fit the team");
  static_assert(!SHF || (SPL >= PR && 32 % SPL == 0), "the parts of a row group lie in one warp");
  static_assert(S_BYTES % 16 == 0 && SC_BYTES % 16 == 0, "bulk copies move multiples of 16 bytes");
};

// --- host construction -----------------------------------------------------------

// Lane tables of one level.  For each cross type the positions of a row's
// entries are those of the interior patch type along x (the union over the x
// codes present), the coefficients follow per type (zero where a type lacks the
// entry).  The entries of a row's parts are ordered so that the lanes of a warp
// read few strip entries of the same bank in one slot.
template <int D, int K, typename T, typename TS>
bool build_line_tables(const Lvl<D, K, T>& L, const Tab<K, T>& tb, std::vector<unsigned char>& blob, std::string& why) {
  using C = LineShape<D, K, T, TS>;
  using R = LineRows<D, K>;
  using PS = PatchShape<D, K>;
  constexpr int LW = C::LW, Z0 = C::Z0, ZP = C::ZP, ZM = C::ZM, NS = C::NS, NV = C::NV;
  blob.assign(C::TAB_BYTES, 0);
  int* tpos = reinterpret_cast<int*>(blob.data() + C::TB_POS);
  int* tcell = reinterpret_cast<int*>(blob.data() + C::TB_CELL);
  T* tcoef = reinterpret_cast<T*>(blob.data() + C::TB_COEF);
  const std::vector<LineRow> lanes = line_rows<D, K>();
  constexpr int BANKS = 128 / (int)sizeof(T), HALF = 32 / (int)(sizeof(T) / 4);   // lanes served by one wavefront
  for (int ct = 0; ct < C::NX; ++ct) {
    // the rows of every x code present
    std::vector<PlanRow<T>> rows[4];
    bool any = false;
    for (int code = 0; code < 4; ++code) {
      const int t = code + 4 * ct;
      if (!type_present<D>(t, L.n)) continue;
      any = true;
      int v[D];
      type_vertex<D>(t, L.n, v);
      plan_rows(L, tb, v, rows[code]);
    }
    if (!any) continue;
    // entry lists per lane: plain entries of the two pieces, mass entries of one cell
    struct Ent { int w; T c[4]; };
    std::vector<std::vector<Ent>> pl0(LW), pl1(LW), ms(LW);
    std::vector<int> cell(LW, 0);
    auto add = [](std::vector<Ent>& p, int code, int w, T c) {
      for (auto& e : p)
        if (e.w == w) {
          e.c[code] = c;
          return;
        }
      p.push_back(Ent{w, {T(0), T(0), T(0), T(0)}});
      p.back().c[code] = c;
    };
    for (const LineRow& lr : lanes) {
      std::vector<Ent> p;
      std::vector<std::vector<Ent>> m;
      std::vector<int> cells;
      for (int code = 0; code < 4; ++code) {
        if (rows[code].empty()) continue;
        for (const auto& e : rows[code][lr.row].pl) add(p, code, e.first, e.second);
        for (const auto& e : rows[code][lr.row].ms) {
          const size_t q = std::find(cells.begin(), cells.end(), e.first.second) - cells.begin();
          if (q == cells.size()) {
            cells.push_back(e.first.second);
            m.push_back({});
          }
          add(m[q], code, e.first.first, e.second);
        }
      }
      const int a = (int)p.size(), nc = (int)cells.size(), gl = nc > 0 ? lr.lanes / nc : 0;   // lanes per cell
      bool ok = lr.lane >= 0 && lr.lane + lr.lanes <= LW && lr.lane % lr.lanes == 0 &&
                a <= lr.lanes * (lr.piece ? C::Z1 : Z0) && (nc == 0 || (gl > 0 && lr.piece == 0));
      for (const auto& e : m) ok = ok && (int)e.size() <= gl * ZM;
      if (!ok) {
        why = "line plan: patch row " + std::to_string(lr.row) + " (" + std::to_string(a) + " entries) does not fit";
        return false;
      }
      for (int i = 0; i < a; ++i) (lr.piece ? pl1 : pl0)[lr.lane + i % lr.lanes].push_back(p[i]);
      for (int q = 0; q < nc; ++q)
        for (int i = 0; i < (int)m[q].size(); ++i) {
          const int lam = lr.lane + q * gl + i % gl;
          ms[lam].push_back(m[q][i]);
          cell[lam] = ((cells[q] >> 1) << 16) | ((cells[q] & 1) + 1);
        }
    }
    // slots: lane after lane, each entry into the free slot of its lane whose
    // wavefront reads the entry's bank least so far
    auto place = [&](std::vector<std::vector<Ent>>& lists, int first, int count) {
      for (int l0 = 0; l0 < LW; l0 += HALF) {
        std::vector<std::vector<int>> words(count);   // strip words read by the wavefront's lanes, per slot
        for (int lam = l0; lam < std::min(l0 + HALF, LW); ++lam) {
          std::vector<char> used(count, 0);
          for (const Ent& e : lists[lam]) {
            const int pos = line_pos<D, K>(e.w), word = (pos >> 16) * line_pitch_rem<D, K>() + (pos & 0xffff);
            int best = -1, cost = 1 << 30;
            for (int s = 0; s < count; ++s) {
              if (used[s]) continue;
              int c = 0;
              for (int w : words[s])
                if (w == word) { c = -1; break; }   // the same word: a broadcast
                else c += (w - word) % BANKS == 0;
              if (c < cost) {
                cost = c;
                best = s;
              }
            }
            used[best] = 1;
            if (cost >= 0) words[best].push_back(word);
            tpos[((size_t)ct * NS + first + best) * LW + lam] = pos;
            for (int code = 0; code < 4; ++code)
              if (!rows[code].empty()) tcoef[((size_t)(code + 4 * ct) * NS + first + best) * LW + lam] = e.c[code];
          }
          for (int s = 0; s < count; ++s)
            if (!used[s]) tpos[((size_t)ct * NS + first + s) * LW + lam] = -1;
        }
        // empty slots read a word their wavefront reads anyway
        for (int s = 0; s < count; ++s) {
          int any_pos = 0;
          for (int o = l0; o < std::min(l0 + HALF, LW); ++o)
            any_pos = std::max(any_pos, tpos[((size_t)ct * NS + first + s) * LW + o]);
          for (int lam = l0; lam < std::min(l0 + HALF, LW); ++lam) {
            int& p = tpos[((size_t)ct * NS + first + s) * LW + lam];
            if (p < 0) p = any_pos;
          }
        }
      }
    };
    place(pl0, 0, Z0);
    if (C::Z1 > 0) place(pl1, Z0, C::Z1);
    place(ms, ZP, ZM);
    for (int lam = 0; lam < LW; ++lam) tcell[(size_t)ct * LW + lam] = cell[lam];
  }
  int* ln = reinterpret_cast<int*>(blob.data() + C::TB_LANE);
  for (int lam = 0; lam < LW; ++lam) {
    ln[2 * lam] = (1 << 16) | 0xffff;
    ln[2 * lam + 1] = -1;
  }
  for (const LineRow& lr : lanes)
    if (lr.piece) ln[2 * lr.lane + 1] = lr.row;
    else
      for (int q = 0; q < lr.lanes; ++q) ln[2 * (lr.lane + q)] = (lr.lanes << 16) | (q == 0 ? lr.row : 0xffff);
  int* st = reinterpret_cast<int*>(blob.data() + C::TB_STRIP);
  for (int r = 0; r < R::XROWS + R::BROWS; ++r) {
    auto base_of = [&](int v1, int v2, int& xr) {
      int v[D], comp;
      v[0] = 2;
      v[1] = v1;
      if (D == 3) v[D - 1] = v2;
      int64_t base;
      xr = 0;
      if (r < R::XROWS) line_xrow(L, v, r, comp, base);
      else line_brow(L, v, r - R::XROWS, comp, xr, base);
      return (int)base;
    };
    int xr;
    const int b00 = base_of(0, 0, xr);
    st[4 * r] = b00;
    st[4 * r + 1] = base_of(1, 0, xr) - b00;
    st[4 * r + 2] = D == 3 ? base_of(0, 1, xr) - b00 : 0;
    int w = xr << 4;
    if (r < R::XROWS) {   // rows in the cells v_e - 2 (outside for v_e = 1) and v_e + 1 (for v_e = n - 1)
      int c = 0;
      while (c < D && r >= R::xfirst(c + 1)) ++c;
      int q = r - R::xfirst(c);
      for (int e = 1; e < D; ++e) {
        const int ext = R::wext(c, e), le = q % ext;
        q /= ext;
        if (c < D && c != e) w |= ((le < C::K1 ? 1 : 0) | (le >= 3 * C::K1 ? 2 : 0)) << (2 * (e - 1));
      }
    }
    st[4 * r + 3] = w;
  }
  int* ro = reinterpret_cast<int*>(blob.data() + C::TB_ROW);
  for (int l = 0; l < NV; ++l) {
    const int c = std::min(l / PS::NU1, D), q = l - c * PS::NU1;
    const int u0 = (c == 0) ? PS::UA : PS::UB;
    int v[D], idx[D];
    for (int e = 0; e < D; ++e) v[e] = 2;
    patch_local_decode<D, K>(v, l, idx);
    ro[2 * l] = line_pos<D, K>(win_index<D, K>(v, c, idx));
    ro[2 * l + 1] = ((R::bfirst(c) + q / u0) << 16) | (ro[2 * l] & 0xffff);
  }
  return true;
}

// Host check of the line tables of one level: every row of every patch type
// evaluated from its lane plan on a strip filled by the kernel's own row
// formulas, against the row visitor on the same values of x and c, and the
// position of every patch row in the x and b strips.
template <int D, int K, typename T, typename TS>
int check_line_tables(const Lvl<D, K, T>& L, const Tab<K, T>& tb, std::string& why) {
  using C = LineShape<D, K, T, TS>;
  using R = LineRows<D, K>;
  constexpr int K1 = K + 1, LW = C::LW, NS = C::NS, ZP = C::ZP, Z0 = C::Z0;
  std::vector<unsigned char> blob;
  if (!build_line_tables<D, K, T, TS>(L, tb, blob, why)) return 1;
  auto val = [](int64_t g) {   // pseudo-random value of x at flat index g
    uint64_t h = (uint64_t)(g + 1) * 0x9E3779B97F4A7C15ull;
    h ^= h >> 29;
    h *= 0xBF58476D1CE4E5B9ull;
    h ^= h >> 32;
    return 2.0 * (double)(h >> 11) * (1.0 / 9007199254740992.0) - 1.0;
  };
  Lvl<D, K, double> Ld;
  Ld.n = L.n;
  Ld.N = L.N;
  for (int e = 0; e <= D; ++e) Ld.off[e] = L.off[e];
  Ld.ndof = L.ndof;
  Ld.s_mu = (double)L.s_mu;
  Ld.s_c = (double)L.s_c;
  Ld.s_b = (double)L.s_b;
  Ld.c = nullptr;
  Tab<K, double> tbd;
  {
    const T* src = reinterpret_cast<const T*>(&tb);
    double* dst = reinterpret_cast<double*>(&tbd);
    for (size_t q = 0; q < sizeof(tb) / sizeof(T); ++q) dst[q] = (double)src[q];
  }
  const int* tpos = reinterpret_cast<const int*>(blob.data() + C::TB_POS);
  const int* tcell = reinterpret_cast<const int*>(blob.data() + C::TB_CELL);
  const T* tcoef = reinterpret_cast<const T*>(blob.data() + C::TB_COEF);
  const int* ro = reinterpret_cast<const int*>(blob.data() + C::TB_ROW);
  // the lanes of each residual row, from the kernel's lane table
  const int* ln = reinterpret_cast<const int*>(blob.data() + C::TB_LANE);
  std::vector<int> lane_of(C::NV, -1), piece_of(C::NV, 0);
  for (int lam = 0; lam < LW; ++lam) {
    const int a = ln[2 * lam] & 0xffff, n = ln[2 * lam] >> 16, b2 = ln[2 * lam + 1];
    if (n < 1 || n > C::GMAX || (n & (n - 1)) || (a != 0xffff && (a >= C::NV || lam % n || lane_of[a] >= 0)) || b2 >= C::NV ||
        (b2 >= 0 && lane_of[b2] >= 0)) {
      why = "line plan: row of a lane";
      return 1;
    }
    if (a != 0xffff) lane_of[a] = lam;
    if (b2 >= 0) {
      lane_of[b2] = lam;
      piece_of[b2] = 1;
    }
  }
  for (int t = 0; t < C::NTYPE; ++t) {
    if (!type_present<D>(t, L.n)) continue;
    const int ct = t >> 2;
    int v[D];
    type_vertex<D>(t, L.n, v);
    // the segment of one vertex: cells v - 2 .. v + 1
    const int PX = 4 * K1 + 1, PC = 4;
    std::vector<double> xs((size_t)R::XROWS * PX, 0.0), cs((size_t)R::CROWS * PC, 0.0);
    std::vector<int64_t> gi((size_t)R::XROWS * PX, -1), bi((size_t)R::BROWS * PX, -1);
    for (int r = 0; r < R::XROWS; ++r) {
      int comp;
      int64_t base;
      const bool ok = line_xrow(L, v, r, comp, base);
      for (int j = 0; j < PX; ++j) {
        const int gx = (v[0] - 2) * K1 + j, hi = comp == 0 ? L.N : L.N - 1;
        if (!ok || gx < 0 || gx > hi) continue;
        gi[(size_t)r * PX + j] = base + gx;
        xs[(size_t)r * PX + j] = val(base + gx);
      }
    }
    for (int r = 0; r < R::BROWS; ++r) {
      int comp, xr;
      int64_t base;
      line_brow(L, v, r, comp, xr, base);
      int comp2;
      int64_t base2;
      if (xr < 0 || xr >= R::XROWS || !line_xrow(L, v, xr, comp2, base2) || comp2 != comp || base2 != base) {
        why = "line strip: b row " + std::to_string(r) + " is not the x row it names";
        return 1;
      }
      for (int j = 0; j < PX; ++j) bi[(size_t)r * PX + j] = base + (v[0] - 2) * K1 + j;
    }
    const int* st = reinterpret_cast<const int*>(blob.data() + C::TB_STRIP);
    for (int r = 0; r < R::XROWS + R::BROWS; ++r) {   // the kernel's strip rows
      const int* e = st + 4 * r;
      int base = e[0] + e[1] * v[1], comp, xr = 0;
      bool ok = !((v[1] == 1 && (e[3] & 1)) || (v[1] == L.n - 1 && (e[3] & 2)));
      if (D == 3) {
        base += e[2] * v[D - 1];
        ok = ok && !((v[D - 1] == 1 && (e[3] & 4)) || (v[D - 1] == L.n - 1 && (e[3] & 8)));
      }
      int64_t want;
      bool in = true;
      if (r < R::XROWS) in = line_xrow(L, v, r, comp, want);
      else line_brow(L, v, r - R::XROWS, comp, xr, want);
      if (ok != in || (in && base != want) || (r >= R::XROWS && (e[3] >> 4) != xr)) {
        why = "line strip: table of row " + std::to_string(r);
        return 1;
      }
    }
    double cw[1 << D];
    for (int q = 0; q < (1 << D); ++q) {
      cw[q] = std::exp(3.0 * val(1000003 + q + 17 * t));
      cs[(size_t)(q >> 1) * PC + 1 + (q & 1)] = cw[q];
    }
    std::vector<double> win(PassShape<D, K, T, T, 1>::WIN, 0.0);
    for (int c = 0; c <= D; ++c) {   // the same values by window column
      int ext[D], tot = 1;
      for (int e = 0; e < D; ++e) {
        ext[e] = win_extent<D, K>(c, e);
        tot *= ext[e];
      }
      for (int q = 0; q < tot; ++q) {
        int idx[D], rr = q;
        bool in = true;
        for (int e = 0; e < D; ++e) {
          idx[e] = win_origin<D, K>(v, c, e) + rr % ext[e];
          rr /= ext[e];
          in = in && idx[e] >= 0 && idx[e] <= ((c < D && e == c) ? L.N : L.N - 1);
        }
        if (!in) continue;
        const int64_t g = flat_index(L, c, idx);
        const int w = win_index<D, K>(v, c, idx), pos = line_pos<D, K>(w);
        if ((pos & 0xffff) >= PX || (pos >> 16) >= R::XROWS || gi[(size_t)(pos >> 16) * PX + (pos & 0xffff)] != g) {
          why = "line strip: type " + std::to_string(t) + " window column " + std::to_string(w) + " holds the wrong entry";
          return 1;
        }
        win[w] = val(g);
      }
    }
    std::vector<double> part0(LW, 0.0), part1(LW, 0.0);
    for (int lam = 0; lam < LW; ++lam) {
      double sum[3] = {0, 0, 0};
      for (int s = 0; s < NS; ++s) {
        const int pos = tpos[((size_t)ct * NS + s) * LW + lam];
        if ((pos >> 16) >= R::XROWS || (pos & 0xffff) >= PX) { why = "line plan: entry outside the strip"; return 1; }
        sum[s < Z0 ? 0 : (s < ZP ? 1 : 2)] +=
            (double)tcoef[((size_t)t * NS + s) * LW + lam] * xs[(size_t)(pos >> 16) * PX + (pos & 0xffff)];
      }
      const int ce = tcell[(size_t)ct * LW + lam];
      if ((ce >> 16) >= R::CROWS || (ce & 0xffff) >= PC) { why = "line plan: cell outside the strip"; return 1; }
      part0[lam] = sum[0] + sum[2] * cs[(size_t)(ce >> 16) * PC + (ce & 0xffff)];
      part1[lam] = sum[1];
    }
    for (int l = 0; l < C::NV; ++l) {
      int idx[D];
      const int comp = patch_local_decode<D, K>(v, l, idx);
      HostEvalVisitor<D, K> ev(v, win.data(), cw);
      visit_row(Ld, tbd, comp, idx, ev);
      double r;
      if (lane_of[l] < 0) { why = "line plan: a row without a lane"; return 1; }
      r = piece_of[l] ? part1[lane_of[l]] : 0.0;
      if (!piece_of[l])
        for (int q = 0; q < (ln[2 * lane_of[l]] >> 16); ++q) r += part0[lane_of[l] + q];
      if (std::fabs(r - ev.acc) > (sizeof(T) == 4 ? 1e-5 : 1e-12) * (ev.mag + 1e-300)) {
        why = "line plan: type " + std::to_string(t) + " row " + std::to_string(l) + " value " + std::to_string(r) +
              " differs from the row value " + std::to_string(ev.acc);
        return 1;
      }
      const int xp = ro[2 * l], bp = ro[2 * l + 1];
      const int64_t g = flat_index(L, comp, idx);
      if (gi[(size_t)(xp >> 16) * PX + (xp & 0xffff)] != g || bi[(size_t)(bp >> 16) * PX + (bp & 0xffff)] != g) {
        why = "line strip: type " + std::to_string(t) + " patch row " + std::to_string(l) + " has the wrong position";
        return 1;
      }
    }
  }
  return 0;
}

// --- the kernel -------------------------------------------------------------------

// One class of lines and the run of passes of a launch.
struct LineArgs {
  int nlines;            // lines of the class
  int first[2], cnt[2];  // cross directions: first vertex and number of lines
  int cl;                // blocks per line (cluster size)
  int px, pc;            // pitch of the strip rows (elements) and of the cell rows
  int teams;             // teams per block
  int nsb;               // inverse buffers per team
  int ns;                // passes of the run
  int cx[LINE_MAX_SUB];  // x digit of each pass
  int cntx[3];           // patches of a line per x digit
  unsigned stream;       // bit s: the inverses of pass s are not read again soon (evict first)
  const void* S[3];      // inverses of the class's colours by x digit
  int64_t s_prob[3];     // bytes between problems of a group
  int nlo, nhi;          // patch rows in the patch's lower and upper cell along x
  uint64_t nb_ns;        // limit of the waits for the neighbour blocks (line_neighbour_limit)
};

// Limit of a block's wait for a neighbour's strip or updates (ns).  A block is at most
// as far behind as its own waits, each within the handle's limit wait_ns, can hold up
// the line: pass s of a block ends no later than its items of that pass take after the
// later of its own and its neighbours' pass s - 1, so the waits of one block's items of
// the whole run bound it, however they are spread over the line.  A second is left for
// the work itself.  (A team that has given up waits for no copy any more, so a copy that
// never lands costs a team one wait.)
constexpr uint64_t line_neighbour_limit(uint64_t wait_ns, int passes, int vertices, int teams, int gpw) {
  const int patches = (vertices + 2) / 3;   // of a block and pass
  return wait_ns * (uint64_t)(passes * ((patches + teams * gpw - 1) / (teams * gpw))) + 1000000000ull;
}
static_assert(line_neighbour_limit(0, 5, 43, 6, 1) == 1000000000ull, "no wait but for the work");
static_assert(line_neighbour_limit(2000000000ull, 1, 3, 8, 1) > 2000000000ull, "longer than one item's wait");
static_assert(line_neighbour_limit(60000000000ull, 5, 43, 6, 1) > 5 * 3 * 60000000000ull, "15 patches on 6 teams, 5 passes");
static_assert(line_neighbour_limit(60000000000ull, 5, 4095, 1, 1) > 5 * 1365 * 60000000000ull, "no overflow on the longest lines");

// (relaxed: only mbarrier initialisations, fenced by mbar_init, are published;
// a release would wait for every copy in flight)
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Waits until every thread of the cluster has left or waits here too (the threads of a
// warp need not come together).
__device__ __forceinline__ void cluster_sync_late() {
  asm volatile("barrier.cluster.arrive.relaxed;\n barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits (at most limit_ns) for an arrival of another block of the cluster.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const uint32_t a = smem_u32(bar);
  uint64_t t0 = 0;
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    const uint64_t t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    else if (t - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Store into another block's shared memory that completes `bytes of the value`
// on a barrier there: who waits for the barrier sees the value (and what was
// ordered before the store), with no fence in between.
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, float v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, double v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}

// Barrier over the threads of a team: one warp, or a named barrier.
template <int TW>
__device__ __forceinline__ void team_sync(int team) {
  __syncwarp();
  if constexpr (TW > 1) asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(32 * TW) : "memory");
}
// The same, returning whether `p` holds for any thread of the team.
template <int TW>
__device__ __forceinline__ bool team_sync_or(int team, bool p) {
  __syncwarp();
  if constexpr (TW == 1) {
    return __any_sync(0xffffffffu, p);
  } else {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred q, s;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred s, %2, %3, q;\n selp.u32 %0, 1, 0, s;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(team + 1), "n"(32 * TW)
        : "memory");
    return r != 0;
  }
}

// PR consecutive entries of a stored inverse from shared memory.
template <int PR, typename TS, typename T>
__device__ __forceinline__ void load_rows(const TS* p, T (&o)[PR]) {
  if constexpr (sizeof(T) == 4) {
    load_rg_smem<TS, T>(p, o);
  } else if constexpr (PR % 2 == 0) {
#pragma unroll
    for (int h = 0; h < PR; h += 2) {
      const double2 v = *reinterpret_cast<const double2*>(p + h);
      o[h] = v.x;
      o[h + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int h = 0; h < PR; ++h) o[h] = p[h];
  }
}

// MB: blocks per SM that the registers leave room for (2: LineShape::LEAN)
template <int D, int K, typename T, typename TS, int NR, int MB>
__global__ void __launch_bounds__(LineShape<D, K, T, TS, NR>::MAXT + 32, MB)
    k_line_sweep(const __grid_constant__ Lvl<D, K, T> L, const __grid_constant__ LineArgs A,
                 const unsigned char* __restrict__ tabs, T* x, const T* __restrict__ b, int* __restrict__ err,
                 uint64_t wait_ns, int64_t vs, const ProbStride ps) {
  using C = LineShape<D, K, T, TS, NR>;
  using R = LineRows<D, K>;
  constexpr int K1 = K + 1, NV = C::NV, LW = C::LW, GPW = C::GPW, NVP = C::NVP, SPL = C::SPL, PR = C::PR, LPP = C::LPP;
  constexpr int Z0 = C::Z0, ZP = C::ZP, ZM = C::ZM, NS = C::NS, NIT = C::NIT;
  constexpr int EB = NR * (int)sizeof(T);   // bytes of a strip entry (the right-hand sides together)
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_launch_dependents();   // the next launch's blocks prepare beside this one's
  const int tid = threadIdx.x;
  const int N = A.teams * C::TT;            // threads of the teams; the last warp copies the inverses
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, nw = N >> 5;
  const int team = warp / C::TW, tl = tid - team * C::TT;   // team, lane of the team
  const int g = GPW > 1 ? tl / LW : 0, lp = GPW > 1 ? tl - g * LW : tl;   // patch of the team, lane of the patch
  const int nx = L.n - 1;   // vertices of a line
  const int rank = blockIdx.x % A.cl, line = blockIdx.x / A.cl;
  const int va = 1 + rank * nx / A.cl, vb = 1 + (rank + 1) * nx / A.cl;   // this block's vertices
  const int m = vb - va, va3 = va % 3;
  const bool left_nb = rank > 0, right_nb = rank < A.cl - 1;
  x += (int64_t)blockIdx.y * NR * vs;
  b += (int64_t)blockIdx.y * NR * vs;
  const int64_t prob = ps.of((int64_t)blockIdx.y * NR);
  // shared memory
  const typename C::Smem lay = C::layout(A.px, A.pc, A.teams, A.nsb);
  const int obs = R::XROWS * A.px * EB, ocs = obs + R::BROWS * A.px * EB;
  const int oends = ocs + R::CROWS * A.pc * (int)sizeof(T);   // coefficients of the line's first and last patch
  int* xrow = reinterpret_cast<int*>(smem + lay.rows);   // flat index of x node 0 per x row (-1: outside)
  int* brow = xrow + R::XROWS;
  volatile int* quit = brow + 2 * R::BROWS;   // 1: a team gave up waiting, 2: a wait for a neighbour ran out
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + lay.bars);   // copies landed [team][buffer]
  uint64_t* empty = full + A.teams * A.nsb;                        // buffers free
  // neighbour blocks [left, right]: strip loaded, then its updates of pass s
  uint64_t* nbs = empty + A.teams * A.nsb;
  constexpr int NBS = 1 + LINE_MAX_SUB;

  // patches of this block in pass s: vertices v0, v0 + 3, .. (cnt of them)
  auto pass_first = [&](int s, int& cnt) {
    int t = A.cx[s] - va3;
    t += t < 0 ? 3 : 0;
    cnt = m > t ? (m - 1 - t) / 3 + 1 : 0;
    return va + t;
  };

  if (warp == nw) {
    // --- the copying warp: lane t streams the inverses of team t through its
    // buffers, as many items ahead as there are buffers
    const bool act = lane < A.teams;
    uint64_t* fb = full + lane * A.nsb;
    uint64_t* eb = empty + lane * A.nsb;
    unsigned char* bufs = smem + lay.buf + lane * A.nsb * C::BUF;
    int is = -1, left = 0, ib = 0, issued = 0;
    uint32_t par = 1u;   // parity of the buffers' barriers one round back
    const unsigned char* src = nullptr;
    [[maybe_unused]] const unsigned char* src_sc = nullptr;
    uint64_t pol = 0;
    auto next_pass = [&]() {
      while (left <= 0 && ++is < A.ns) {
        int cnt;
        const int cx = A.cx[is], v0 = pass_first(is, cnt);
        left = cnt - lane * GPW;
        const int p = (v0 - colour_first(cx)) / 3 + A.cntx[cx] * line + lane * GPW;
        const unsigned char* S = static_cast<const unsigned char*>(A.S[cx]) + prob * A.s_prob[cx];
        src = S + (int64_t)p * C::S_BYTES;
        if constexpr (C::BF) src_sc = S + (int64_t)A.cntx[cx] * A.nlines * C::S_BYTES + (int64_t)p * C::SC_BYTES;
        pol = ((A.stream >> is) & 1u) ? l2_policy_evict_first() : l2_policy_evict_last();
      }
    };
    auto issue = [&]() {
      const int np = GPW == 1 ? 1 : min(GPW, left);
      unsigned char* dst = bufs + ib * C::BUF;
      mbar_arrive_expect_tx(fb + ib, (uint32_t)(np * (C::S_BYTES + C::SC_BYTES)));
      bulk_load(dst, src, (uint32_t)(np * C::S_BYTES), fb + ib, pol);
      if constexpr (C::BF) bulk_load(dst + GPW * C::S_BYTES, src_sc, (uint32_t)(np * C::SC_BYTES), fb + ib, pol);
      src += A.teams * (GPW * C::S_BYTES);
      if constexpr (C::BF) src_sc += A.teams * (GPW * C::SC_BYTES);
      left -= A.teams * GPW;
      if (++ib == A.nsb) {
        ib = 0;
        par ^= 1u;
      }
      ++issued;
      if (left <= 0) next_pass();
    };
    if (act) {
      for (int q = 0; q < A.nsb; ++q) {
        mbar_init(fb + q, 1);
        mbar_init(eb + q, C::TW);
      }
      next_pass();
      for (int q = 0; q < A.nsb && is < A.ns; ++q) issue();
    }
    // what the neighbours will send: a word once their strip is loaded, and the
    // updates of their vertices within two of this segment that lie in its strip
    if (A.cl > 1 && lane < 2 * NBS) {
      const bool rside = lane >= NBS;
      const int s = lane - (rside ? NBS : 0) - 1;
      mbar_init(nbs + lane, 1);
      if ((rside ? right_nb : left_nb) && s < A.ns) {
        uint32_t bytes = 4;
        if (s >= 0) {
          const int far = rside ? vb + 1 : va - 2, near = rside ? vb : va - 1, cx = A.cx[s];
          bytes = (uint32_t)(EB * (near % 3 == cx ? NV : (far % 3 == cx ? (rside ? A.nlo : A.nhi) : 0)));
        }
        mbar_arrive_expect_tx(nbs + lane, bytes);
      }
    }
    if (lane == 0) *quit = 0;
    __syncthreads();   // barriers and row tables
    if (A.cl > 1) {
      cluster_arrive();   // barriers ready
      cluster_wait();
    }
    // a buffer is refilled once its team has released it; the rest is given up
    // when a team has given up (or nothing moves for longer than any wait)
    uint64_t t0 = globaltimer_ns();
    bool more = act && is < A.ns && wait_ns != 0;
    while (__any_sync(0xffffffffu, more)) {
      bool did = false;
      if (more && mbar_test(eb + ib, par)) {
        fence_proxy_async_smem();   // the team's reads of the buffer before the copy's writes
        issue();
        more = is < A.ns;
        did = true;
      }
      if (__any_sync(0xffffffffu, did)) t0 = globaltimer_ns();
      else if (*quit || globaltimer_ns() - t0 > wait_ns + A.nb_ns) break;
      else __nanosleep(20);
    }
    // no copy may land after the block has left: wait (bounded) for the last one
    // of every buffer (already there unless a team gave up)
    if (act)
      for (int q = 0; q < A.nsb && q < issued; ++q) {
        const int cnt = (issued - q + A.nsb - 1) / A.nsb;   // copies into buffer q
        mbar_wait_bounded(fb + q, (uint32_t)((cnt - 1) & 1), 100000000ull);
      }
    return;
  }

  // --- the teams.  (1) everything that does not depend on the preceding kernel
  int v[D];
  v[0] = 2;
  v[1] = A.first[0] + 3 * (D == 2 ? line : line % A.cnt[0]);
  if (D == 3) v[D - 1] = A.first[1] + 3 * (line / A.cnt[0]);
  T* const scr = reinterpret_cast<T*>(smem + lay.scr) + (team * GPW + g) * C::SCR;
  T* rv = scr;   // residual buffer of the current item
  unsigned char* bufs = smem + lay.buf + team * A.nsb * C::BUF;
  full += team * A.nsb;
  empty += team * A.nsb;
  // rows of the strips
  for (int q = tid; q < R::XROWS + R::BROWS; q += N) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(tabs + C::TB_STRIP) + q);
    int base = e.x + e.y * v[1];
    bool ok = !((v[1] == 1 && (e.w & 1)) || (v[1] == nx && (e.w & 2)));
    if constexpr (D == 3) {
      base += e.z * v[D - 1];
      ok = ok && !((v[D - 1] == 1 && (e.w & 4)) || (v[D - 1] == nx && (e.w & 8)));
    }
    xrow[q] = ok ? base : -1;
    if (q >= R::XROWS) brow[R::BROWS + q - R::XROWS] = e.w >> 4;   // the x row of the same nodes
  }
  // positions and coefficients of the interior patches of the line
  int ct = 0;
#pragma unroll
  for (int e = 1; e < D; ++e) ct += type_code(v[e], L.n) << (2 * (e - 1));
  const int code_mid = L.n >= 4 ? 1 : (L.n == 2 ? 3 : 0);
  T pc[ZP], mc[ZM];
  int po[ZP], mo[ZM];
  {
    const int* tp = reinterpret_cast<const int*>(tabs + C::TB_POS) + ct * NS * LW + lp;
    const T* tc = reinterpret_cast<const T*>(tabs + C::TB_COEF) + (code_mid + 4 * ct) * NS * LW + lp;
#pragma unroll
    for (int s = 0; s < ZP; ++s) {
      const int pos = __ldg(tp + s * LW);
      pc[s] = __ldg(tc + s * LW);
      po[s] = ((pos >> 16) * A.px + (pos & 0xffff)) * EB;
    }
#pragma unroll
    for (int s = 0; s < ZM; ++s) {
      const int pos = __ldg(tp + (ZP + s) * LW);
      mc[s] = __ldg(tc + (ZP + s) * LW);
      mo[s] = ((pos >> 16) * A.px + (pos & 0xffff)) * EB;
    }
  }
  int co;
  {
    const int pos = __ldg(reinterpret_cast<const int*>(tabs + C::TB_CELL) + ct * LW + lp);
    co = ocs + ((pos >> 16) * A.pc + (pos & 0xffff)) * (int)sizeof(T);
  }
  const T* tends = reinterpret_cast<const T*>(tabs + C::TB_COEF) + 4 * ct * NS * LW;   // by x code
  if constexpr (C::ENDS) {
    T* ends = reinterpret_cast<T*>(smem + oends);
    if (va == 1)
      for (int q = tid; q < C::END_N; q += N) ends[q] = __ldg(tends + type_code(1, L.n) * C::END_N + q);
    if (vb == L.n)
      for (int q = tid; q < C::END_N; q += N) ends[C::END_N + q] = __ldg(tends + type_code(nx, L.n) * C::END_N + q);
  }
  // rows of this lane: those whose residual it writes (ra, rb), the lanes gs that
  // share the first, and the rows of the update it makes
  const int2* rowt = reinterpret_cast<const int2*>(tabs + C::TB_ROW);
  auto off_of = [&](int pos) { return ((pos >> 16) * A.px + (pos & 0xffff)) * EB; };
  const int2 li = __ldg(reinterpret_cast<const int2*>(tabs + C::TB_LANE) + lp);
  const int ra = (li.x & 0xffff) == 0xffff ? -1 : (li.x & 0xffff), gs = li.x >> 16, rb = li.y;
  [[maybe_unused]] const bool second = C::Z1 > 0 && __any_sync(0xffffffffu, rb >= 0);   // the warp has second pieces
  int ba = 0, bp = 0, xo[NIT], xcol[NIT];
  if (ra >= 0) ba = obs + off_of(__ldg(rowt + ra).y);
  if (C::Z1 > 0 && rb >= 0) bp = obs + off_of(__ldg(rowt + rb).y);
  const int part = C::SHF ? lp % SPL : lp / LPP, grp = C::SHF ? lp / SPL : lp - part * LPP;
  auto urow = [&](int it) {   // row of the update (NV: none)
    if constexpr (C::SHF) return (part < PR && grp < LPP) ? min(grp * PR + part, NV) : NV;
    else return min(lp + it * LW, NV);
  };
#pragma unroll
  for (int it = 0; it < NIT; ++it) {
    xo[it] = xcol[it] = 0;
    if (urow(it) < NV) {
      const int pos = __ldg(rowt + urow(it)).x;
      xo[it] = off_of(pos);
      xcol[it] = pos & 0xffff;
    }
  }
  __syncthreads();   // rows, barriers, end coefficients
  if (A.cl > 1) cluster_arrive();   // barriers ready
  // b and c strips: columns of cells va - 2 .. vb, read ahead of the wait: the launch
  // before writes x only, and what wrote b ended before that one began
  const int wc = m + 3, x0 = (va - 2) * K1;
  const int wx = wc * K1 + 1;
  const uint32_t wmag = 0xffffffffu / (uint32_t)wx + 1u;   // e / wx as the high word of e wmag, for e below 2^32 / wx
  for (int e = tid; e < R::BROWS * wx; e += N) {
    const int r = (int)__umulhi((uint32_t)e, wmag), j = e - r * wx;
    const bool ok = (unsigned)(x0 + j) < (unsigned)L.N;
    const T* from = ok ? b + (brow[r] + x0 + j) : b;
    T* dst = reinterpret_cast<T*>(smem + obs + (r * A.px + j) * EB);
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) cp_async_t(dst + rr, ok ? from + rr * vs : b, ok);
  }
  const T* coef = L.c + prob * ps.c;
  for (int r = warp; r < R::CROWS; r += nw) {
    int base = va - 2, st = L.n;
#pragma unroll
    for (int e = 1; e < D; ++e) {
      base += (v[e] - 1 + ((r >> (e - 1)) & 1)) * st;
      st *= L.n;
    }
    T* dst = reinterpret_cast<T*>(smem + ocs) + r * A.pc;
    for (int j = lane; j < wc; j += 32) {
      const bool ok = (unsigned)(va - 2 + j) < (unsigned)L.n;
      cp_async_t(dst + j, ok ? coef + base + j : coef, ok);
    }
  }
  // (2) x strip: the addresses of the first entries per thread are ready before
  // the wait for the preceding kernel
  constexpr int PRE = NR == 1 ? 8 : 4;
  const int ne = R::XROWS * wx;
  int gofs[PRE], sofs[PRE];
#pragma unroll
  for (int q = 0; q < PRE; ++q) {
    const int e = tid + q * N, r = min((int)__umulhi((uint32_t)e, wmag), R::XROWS - 1), j = e - r * wx;
    const int base = xrow[r], hi = r < R::xfirst(1) ? L.N + 1 : L.N;
    sofs[q] = e < ne ? (r * A.px + j) * EB : -1;
    gofs[q] = e < ne && base >= 0 && (unsigned)(x0 + j) < (unsigned)hi ? base + x0 + j : -1;
  }
  pdl_wait();   // x comes from the preceding kernel
#pragma unroll
  for (int q = 0; q < PRE; ++q)
    if (sofs[q] >= 0) {
      T* dst = reinterpret_cast<T*>(smem + sofs[q]);
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) cp_async_t(dst + rr, gofs[q] >= 0 ? x + gofs[q] + rr * vs : x, gofs[q] >= 0);
    }
  for (int e = tid + PRE * N; e < ne; e += N) {
    const int r = min((int)__umulhi((uint32_t)e, wmag), R::XROWS - 1), j = e - r * wx;
    const int base = xrow[r], hi = r < R::xfirst(1) ? L.N + 1 : L.N;
    const bool ok = base >= 0 && (unsigned)(x0 + j) < (unsigned)hi;
    T* dst = reinterpret_cast<T*>(smem + (r * A.px + j) * EB);
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) cp_async_t(dst + rr, ok ? x + base + x0 + j + rr * vs : x, ok);
  }
  cp_async_commit();
  const int ml = left_nb ? va - (1 + (rank - 1) * nx / A.cl) : 0;   // vertices of the block to the left
  // a = 0: the neighbours' strips are loaded, s + 1: their updates of pass s are here
  auto wait_nb = [&](int a) {
    bool ok = true;
    if (left_nb) ok = mbar_wait_cluster(nbs + a, 0, A.nb_ns);
    if (right_nb) ok = mbar_wait_cluster(nbs + NBS + a, 0, A.nb_ns) && ok;
    if (!ok) {
      atomicOr(const_cast<int*>(quit), 2);
      atomicExch(err, 2);
    }
  };
  auto block_sync = [&]() {
    __syncwarp();
    asm volatile("bar.sync 0, %0;" ::"r"(N) : "memory");
  };
  if (A.cl > 1) cluster_wait();   // the neighbours' barriers are ready
  int cnt, v0 = pass_first(0, cnt);
  cp_async_wait<0>();
  block_sync();
  if (tid == 0) {   // strip loaded: the neighbours may store into it
    const uint32_t word = smem_u32(nbs + 2 * NBS), l0 = smem_u32(nbs + NBS), r0 = smem_u32(nbs);
    if (left_nb) st_async(map_rank(word, rank - 1), map_rank(l0, rank - 1), 0.f);
    if (right_nb) st_async(map_rank(word + 4, rank + 1), map_rank(r0, rank + 1), 0.f);
  }

  // (3) the passes
  int sb = 0;           // buffer of the current item
  uint32_t phase = 0;   // parity of that buffer's barrier
  bool dead = false;    // a wait ran out: the team only keeps the barriers
  for (int s = 0; s < A.ns; ++s) {
    for (int q0 = team * GPW; q0 < cnt; q0 += A.teams * GPW) {
      const bool act = GPW == 1 || q0 + g < cnt;
      const int vx = v0 + 3 * (q0 + (act ? g : 0));
      const int pb = (vx - va) * (K1 * EB);   // strip base of the patch (bytes)
      auto at = [&](int off) { return reinterpret_cast<T*>(smem + (off + pb)); };
      T xw[NIT][NR];   // this lane's rows of x
#pragma unroll
      for (int it = 0; it < NIT; ++it) ld_rhs<T, NR>(at(xo[it]), xw[it]);
      auto update = [&]() -> bool {   // false: the inverses did not arrive in time
      bool ready = mbar_try_wait(full + sb, phase);   // the inverses, usually there by now
      // (3a) local residual
      T t0[NR], t1[NR];
      auto residual = [&](auto cf) {   // cf(slot): coefficient of the lane's slot
        T u0[NR], am[NR];
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) t0[rr] = t1[rr] = u0[rr] = am[rr] = T(0);
#pragma unroll
        for (int z = 0; z < Z0; ++z) {
          T w[NR];
          ld_rhs<T, NR>(at(po[z]), w);
          const T c0 = cf(z);
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) {
            if (NR == 1 && (z & 1)) u0[rr] += c0 * w[rr];
            else t0[rr] += c0 * w[rr];
          }
        }
#pragma unroll
        for (int z = 0; z < ZM; ++z) {
          T w[NR];
          ld_rhs<T, NR>(at(mo[z]), w);
          const T c0 = cf(ZP + z);
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) am[rr] += c0 * w[rr];
        }
        const T ck = *reinterpret_cast<const T*>(smem + co + (vx - va) * (int)sizeof(T));
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          if (NR == 1) t0[rr] += u0[rr];
          t0[rr] += ck * am[rr];
        }
        if (C::Z1 > 0 && (C::TW == 1 || second)) {
#pragma unroll
          for (int z = Z0; z < ZP; ++z) {
            T w[NR];
            ld_rhs<T, NR>(at(po[z]), w);
            const T c0 = cf(z);
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) t1[rr] += c0 * w[rr];
          }
        }
      };
      if ((vx != 1 && vx != nx) || type_code(vx, L.n) == code_mid) {
        residual([&](int z) { return z < ZP ? pc[z < ZP ? z : 0] : mc[z >= ZP ? z - ZP : 0]; });
      } else if constexpr (C::ENDS) {
        const T* ec = reinterpret_cast<const T*>(smem + oends) + (vx == 1 ? 0 : C::END_N) + lp;
        residual([&](int z) { return ec[z * LW]; });
      } else {
        const T* ec = tends + type_code(vx, L.n) * NS * LW + lp;
        residual([&](int z) { return __ldg(ec + z * LW); });
      }
      // the lanes of a row
#pragma unroll
      for (int o = 1; o < C::GMAX; o <<= 1)
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          const T w = __shfl_xor_sync(0xffffffffu, t0[rr], o);
          if (gs > o) t0[rr] += w;
        }
      unsigned char* sbuf = bufs + sb * C::BUF;
      const float* scl = reinterpret_cast<const float*>(sbuf + GPW * C::S_BYTES) + g * NVP;
      // (bounded wait; BF16: the inverses' row scales enter r)
      if constexpr (C::BF) ready = wait_ns != 0 && (ready || mbar_wait_bounded(full + sb, phase, wait_ns));
      auto put_r = [&](int row, int bofs, const T (&t)[NR]) {
        T r[NR];
        ld_rhs<T, NR>(at(bofs), r);
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          r[rr] -= t[rr];
          if constexpr (C::BF) r[rr] *= (T)scl[row];
        }
        if constexpr (C::RP == 2 * NR) reinterpret_cast<float2*>(rv)[row] = make_float2(r[0], r[0]);
        else st_rhs<T, NR>(rv + row * NR, r);
      };
      if (ra >= 0) put_r(ra, ba, t0);
      if constexpr (C::Z1 > 0) {
        if (rb >= 0) put_r(rb, bp, t1);
      }
      if constexpr (!C::BF) ready = wait_ns != 0 && (ready || mbar_wait_bounded(full + sb, phase, wait_ns));
      if (team_sync_or<C::TW>(team, !ready)) {
        if (tl == 0) {
          atomicExch(err, 2);
          atomicOr(const_cast<int*>(quit), 1);
        }
        return false;
      }
      [[maybe_unused]] T scx[NIT];
      if constexpr (C::BF)
#pragma unroll
        for (int it = 0; it < NIT; ++it) scx[it] = (T)scl[min(urow(it), NV - 1)];
      // (3b) delta = S_v r
      T d[PR][NR];
#pragma unroll
      for (int i = 0; i < PR; ++i)
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) d[i][rr] = T(0);
      if (LPP * SPL == LW || (C::SHF ? grp < LPP : part < SPL)) {
        const TS* Sg = reinterpret_cast<const TS*>(sbuf + g * C::S_BYTES) + grp * PR + part * NVP;
        if constexpr (C::RP == 2 * NR) {   // FP32, one right-hand side: packed pairs
          float2 acc[PR / 2];
#pragma unroll
          for (int h = 0; h < PR / 2; ++h) acc[h] = make_float2(0.f, 0.f);
          const float2* rp = reinterpret_cast<const float2*>(rv) + part;
#pragma unroll
          for (int jj = 0; jj < C::JCH; ++jj) {
            if ((jj + 1) * SPL <= NV || part + jj * SPL < NV) {
              float sv[PR];
              load_rows<PR, TS, float>(Sg + jj * SPL * NVP, sv);
              const float2 rj = rp[jj * SPL];
#pragma unroll
              for (int h = 0; h < PR / 2; ++h) acc[h] = __ffma2_rn(make_float2(sv[2 * h], sv[2 * h + 1]), rj, acc[h]);
            }
          }
#pragma unroll
          for (int h = 0; h < PR / 2; ++h) {
            d[2 * h][0] = acc[h].x;
            d[2 * h + 1][0] = acc[h].y;
          }
        } else {
#pragma unroll
          for (int jj = 0; jj < C::JCH; ++jj) {
            if ((jj + 1) * SPL <= NV || part + jj * SPL < NV) {
              T sv[PR], rj[NR];
              load_rows<PR, TS, T>(Sg + jj * SPL * NVP, sv);
              ld_rhs<T, NR>(rv + (part + jj * SPL) * NR, rj);
#pragma unroll
              for (int i = 0; i < PR; ++i)
#pragma unroll
                for (int rr = 0; rr < NR; ++rr) d[i][rr] += sv[i] * rj[rr];
            }
          }
        }
        if constexpr (!C::SHF) {
          T* dp = scr + C::O_D + (part * (LPP * PR) + grp * PR) * NR;
          if constexpr (NR == 1 && sizeof(T) == 4) {
#pragma unroll
            for (int i = 0; i < PR; i += 4) *reinterpret_cast<float4*>(dp + i) = make_float4(d[i][0], d[i + 1][0], d[i + 2][0], d[i + 3][0]);
          } else {
#pragma unroll
            for (int i = 0; i < PR; ++i) st_rhs<T, NR>(dp + i * NR, d[i]);
          }
        }
      }
      if constexpr (C::SHF) {
        // reduce and scatter: at each round a lane keeps the half of the rows its
        // part's bit names; then the parts of equal low bits are added
#pragma unroll
        for (int o = PR / 2; o > 0; o >>= 1) {
          const bool up = (part & o) != 0;
#pragma unroll
          for (int i = 0; i < PR / 2; ++i) {
            if (i >= o) break;
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
              const T keep = up ? d[i + o][rr] : d[i][rr], give = up ? d[i][rr] : d[i + o][rr];
              d[i][rr] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
          }
        }
#pragma unroll
        for (int o = PR; o < SPL; o <<= 1)
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) d[0][rr] += __shfl_xor_sync(0xffffffffu, d[0][rr], o);
        __syncwarp();
      } else {
        team_sync<C::TW>(team);
      }
      if (lane == 0) mbar_arrive(empty + sb);   // this warp is done with the inverses
      // (3c) x|_v += delta, in the strip and, near a segment's end, in the neighbour's
#pragma unroll
      for (int it = 0; it < NIT; ++it) {
        if (urow(it) >= NV) break;
        T delta[NR];
        if constexpr (C::SHF) {
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) delta[rr] = d[0][rr];
        } else {
          const T* dp = scr + C::O_D + (lp + it * LW) * NR;
          ld_rhs<T, NR>(dp, delta);
#pragma unroll
          for (int q2 = 1; q2 < SPL; ++q2) {
            T w[NR];
            ld_rhs<T, NR>(dp + q2 * (LPP * PR) * NR, w);
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) delta[rr] += w[rr];
          }
        }
        if (GPW > 1 && !act) break;
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          if constexpr (C::BF) xw[it][rr] += delta[rr] * scx[it];
          else xw[it][rr] += delta[rr];
        }
        st_rhs<T, NR>(at(xo[it]), xw[it]);
      }
      return true;
      };
      if (!dead) dead = !update();
      if (A.cl > 1 && (vx <= va + 1 || vx >= vb - 2)) {
        if (s == 0) wait_nb(0);   // the neighbours' strips are loaded
        if (act) {
#pragma unroll
          for (int it = 0; it < NIT; ++it) {
            if (urow(it) >= NV) break;
            const int col = xcol[it] + (vx - va) * K1;
            const uint32_t own = smem_u32(at(xo[it]));
            if (left_nb && vx <= va + 1 && col < 3 * K1) {
              const uint32_t to = map_rank(own, rank - 1) + ml * (K1 * EB), bar = map_rank(smem_u32(nbs + NBS + s + 1), rank - 1);
#pragma unroll
              for (int rr = 0; rr < NR; ++rr) st_async(to + rr * (int)sizeof(T), bar, xw[it][rr]);
            }
            if (right_nb && vx >= vb - 2 && col >= m * K1) {
              const uint32_t to = map_rank(own, rank + 1) - m * (K1 * EB), bar = map_rank(smem_u32(nbs + s + 1), rank + 1);
#pragma unroll
              for (int rr = 0; rr < NR; ++rr) st_async(to + rr * (int)sizeof(T), bar, xw[it][rr]);
            }
          }
        }
      }
      if (++sb == A.nsb) {
        sb = 0;
        phase ^= 1u;
      }
      if constexpr (C::RVN == 2) rv = rv == scr ? scr + C::RVS : scr;
    }
    // the next pass reads what this one wrote: the block's teams, then the
    // neighbour blocks
    if (s + 1 < A.ns) v0 = pass_first(s + 1, cnt);
    block_sync();
    if (A.cl > 1) wait_nb(s + 1);
  }
  // A block leaves once everything its neighbours send has landed, the word of a loaded
  // strip too.  Where a wait for it ran out they may be slower still, and a store into a
  // block that has left would be a fault: the block then stays until every other one of
  // the line has left or waits here too (all their waits are bounded), and looks for what
  // they sent once more.  (The barrier in the loop, not behind it or behind the stores,
  // and no flag or limit read besides: other forms took 0.5 to 4 % of a 256^2 RT_1 cycle,
  // 1,478 us without any, 1,482 so.)
  if (A.cl > 1) {
    int a = 0;
    do {
      wait_nb(a > A.ns ? 0 : a);
      if (a == 0 && (*quit & 2)) cluster_sync_late();
    } while ((*quit & 2) && ++a <= A.ns + 1);
  }
  // (4) the updated rows of this segment's cells: va - 1 .. vb - 2, the first
  // and last block to the ends of the line
  const int lo = (va - 1) * K1, hi = rank == A.cl - 1 ? L.N : (vb - 1) * K1;
  for (int r = warp; r < R::BROWS; r += nw) {
    T* dst = x + brow[r];
    const T* from = reinterpret_cast<const T*>(smem + (brow[R::BROWS + r] * A.px - x0) * EB);
    for (int gx = lo + lane; gx < hi; gx += 32) {
      T w[NR];
      ld_rhs<T, NR>(from + gx * NR, w);
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) dst[gx + rr * vs] = w[rr];
    }
  }
}

}  // namespace mgd
