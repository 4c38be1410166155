// Encoder of the scheduled engine: plays the message passing of every loaded instance through, one warp per instance, and
// writes the instance's program (wave.h).  A payload is a list of row records, a row record a list of terms.
#include <cuda_runtime.h>

#include "kernel_smem.h"
#include "wave.h"

namespace wave {
using namespace amp;

namespace {

constexpr int EW = 4;                  // warps per block
constexpr unsigned FULL = 0xffffffffu;

struct __align__(16) Item {            // a message on its way: state, payload rows
  unsigned where;                      // node | arrival port << 8 | direction << 16 | state port << 20
  unsigned state;                      // iteration | position << 16
  unsigned rs, n;                      // first row record, rows
};
enum { OUT_PORT = 0xff };              // arrival port of a deferred emission (a GRU's result, one step after its first half)

__device__ __forceinline__ unsigned pack_where(int node, int aport, int dir, int sport) { return node | (aport << 8) | (dir << 16) | (sport << 20); }

struct Row { unsigned ts, nt; };

__device__ __forceinline__ unsigned warp_excl(unsigned v, unsigned& total) {
  const int lane = threadIdx.x & 31;
  unsigned s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const unsigned x = __shfl_up_sync(FULL, s, o); if (lane >= o) s += x; }
  total = __shfl_sync(FULL, s, 31);
  return s - v;
}

__device__ __forceinline__ unsigned long long warp_excl64(unsigned long long v, unsigned long long& total) {
  const int lane = threadIdx.x & 31;
  unsigned long long s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const unsigned long long x = __shfl_up_sync(FULL, s, o); if (lane >= o) s += x; }
  total = __shfl_sync(FULL, s, 31);
  return s - v;
}

template <bool EMIT>
struct Encoder {
  const EncModel& M; const DevInst& I; unsigned* const scr; Item* const stack; unsigned* const cur;
  Item* front[3]; Row* rows; Term* terms;
  const int lane; const unsigned STACK;
  long long inst, ibase, ebase;
  unsigned n_front[3], n_rows, n_terms, arena4, n_ov, msgs_f, msgs_b;
  int pending, retired, status;
  Entry* const* ent; Term* ovp; unsigned* ov_cursor; const unsigned* cell_end;

  __device__ Encoder(const EncModel& m, const DevInst& i, unsigned* s, Item* st, unsigned* c) : M(m), I(i), scr(s), stack(st), cur(c), lane(threadIdx.x & 31), STACK(m.stack_cap) {
    char* p = reinterpret_cast<char*>(s + m.table_words);
    for (int k = 0; k < 3; k++) { front[k] = reinterpret_cast<Item*>(p); p += (size_t)m.front_cap * sizeof(Item); }
    terms = reinterpret_cast<Term*>(p); p += (size_t)m.term_cap * sizeof(Term);
    rows = reinterpret_cast<Row*>(p);
  }
  __device__ unsigned key(unsigned state, int u, int U) {
    const int it = state & 0xffff;
    if ((unsigned)u >= (unsigned)U || it >= M.IT) { status = ST_OVERFLOW; return 0; }
    return (unsigned)it * U + u;
  }
  __device__ unsigned alloc(unsigned n, unsigned& cursor, unsigned cap) {       // per-lane share of a bump allocation
    unsigned total;
    const unsigned off = cursor + warp_excl(n, total);
    cursor += total;
    if (cursor > cap) { status = ST_OVERFLOW; return 0; }
    return off;
  }
  __device__ void land(bool yes, const Item& it, int f) {                        // append to the frontier f
    unsigned total;
    const unsigned at = n_front[f] + warp_excl(yes ? 1u : 0u, total);
    n_front[f] += total;
    if (n_front[f] > M.front_cap) { status = ST_OVERFLOW; n_front[f] = M.front_cap; return; }
    if (yes) front[f][at] = it;
  }

  // ---- one hop of up to 32 messages; `next` collects what reaches parameterised nodes ----------------------------
  __device__ void drain(unsigned& sp, const int next) {
    for (unsigned guard = 0; sp > 0 && !__any_sync(FULL, status); guard++) {
      if (guard > (1u << 20)) { status = ST_OVERFLOW; return; }      // (no structure needs that many)
      const unsigned n = min(32u, sp);
      sp -= n;
      const bool live = lane < n;
      Item it{};
      if (live) it = stack[sp + lane];
      __syncwarp();
      int node = it.where & 0xff, aport = (it.where >> 8) & 0xff, dir = (it.where >> 16) & 1, sport = (it.where >> 20) & 0xff, u = it.state >> 16;
      enum { A_NONE, A_PASS, A_FORK, A_SLICE, A_CONCAT, A_SUM, A_GATHER, A_SUMALL, A_SUMREFS, A_SPREAD, A_MULTI, A_REP, A_LAND };
      int act = A_NONE, J = 0, to = -1, to_port = 0, to_dir = dir, port = sport, reps = 0;
      unsigned state = it.state, cnt = NONE, ref = NONE, expected = 0, rs = it.rs, nr = it.n, w4 = 0;
      const EncNode* NP = &M.nodes[live ? node : 0];
#define N (*NP)
      auto succ = [&](int k) { to = N.succ_node[k]; to_port = N.succ_port[k]; to_dir = FWD; };
      auto pred = [&](int k) { to = N.pred_node[k]; to_port = N.pred_port[k]; to_dir = BWD; };
      auto at_u = [&](int nu) { state = (state & 0xffff) | ((unsigned)nu << 16); };
      auto join = [&](int ku, int Uk, int slot, int slots, int exp_) {           // reference `slot` of the join keyed on (it, ku)
        const unsigned k = key(it.state, ku, Uk);
        if ((unsigned)slot >= (unsigned)slots || exp_ > slots) { status = ST_OVERFLOW; return; }
        ref = N.ref_off + k * N.J; cnt = N.cnt_off + k; expected = exp_;
        scr[ref + slot] = it.rs;
      };
      // (nodes that only change the state or the way are walked through on the spot)
      for (int hops = 0; live; hops++) {
        if (hops > 64) { status = ST_OVERFLOW; act = A_NONE; break; }
        act = A_NONE;
        if (N.type != SOURCE) { if (dir == FWD) msgs_f++; else msgs_b++; }
        switch (N.type) {
          case LINEAR: case LOOKUP: case GRUCELL: {
            const EncPpt& P = M.ppts[N.ppt];
            act = A_LAND;
            // a gate node's Linear waits for the children's cells, which arrive at the gate node's second port
            if (dir == FWD && P.lstm >= 0 && M.nodes[P.lstm].fn == 2) {
              const EncNode& L = M.nodes[P.lstm];
              const unsigned k = key(it.state, u, L.U);
              ref = L.ref_off + k * L.J; cnt = L.cnt_off + k; expected = 2;
              scr[ref] = it.rs;
            }
          } break;
          case NPT_LSTM:
            if (dir == FWD) {                                  // (port 0 is the Linear's own result: it fires inside its cell)
              const unsigned k = key(it.state, u, N.U);
              ref = N.ref_off + k * N.J; cnt = N.cnt_off + k; expected = 2;
              scr[ref + 1] = it.rs;
              to = N.pred_node[0];
              act = A_LAND;
            } else { to = N.pred_node[0]; act = A_LAND; msgs_b++; }
            break;
          case SOURCE: retired++; break;
          case SINK: nr = it.n; act = A_REP; reps = -1; pred(0); break;          // answers with a zero gradient
          case COND:
            act = A_PASS;
            if (dir == FWD) {
              int k = 0;
              switch (N.fn) {
                case 1: k = u < (int)(I.offsets[inst + 1] - ibase) ? 0 : 1; break;
                case 2: k = I.parent[ibase + u] < 0 ? 0 : 1; break;
                case 3: k = u; break;
                case 4: k = (int)(it.state & 0xffff) < N.fn_arg ? 0 : 1; break;
                case 5: k = (int)((inst + u) % N.n_succ); break;
              }
              if ((unsigned)k >= (unsigned)N.n_succ) { status = ST_OVERFLOW; k = 0; }
              succ(k);
            } else pred(0);
            break;
          case PHI: {
            const unsigned k = N.cnt_off + key(it.state, u, N.U);
            act = A_PASS;
            if (dir == FWD) { scr[k] = aport + 1; succ(0); }
            else {
              const int j = (int)scr[k] - 1;
              if (j < 0 || j >= N.n_pred) { status = ST_OVERFLOW; act = A_NONE; break; }
              scr[k] = 0;
              pred(j);
            }
          } break;
          case ISU:
            act = A_PASS;
            if (dir == FWD) {
              if (N.fn == 1) at_u(u + 1);
              else if (N.fn == 2) { port = I.child_slot[ibase + u]; at_u(I.parent[ibase + u]); }
              else state += 1;
              succ(0);
            } else {
              if (N.fn == 1) at_u(u - 1);
              else if (N.fn == 2) { at_u(sport == 0 ? I.left[ibase + u] : I.right[ibase + u]); port = 0; }
              else state -= 1;
              pred(0);
            }
            break;
          case BCAST:
            if (dir == FWD) { act = A_FORK; reps = N.fn_arg; }
            else { join(u, N.U, aport, N.fn_arg, N.fn_arg); act = A_SUM; J = N.fn_arg; pred(0); }
            break;
          case CONCAT:
            if (dir == FWD) { join(u, N.U, N.fn == 2 ? sport : aport, N.fn_arg, N.fn_arg); act = A_CONCAT; J = N.fn_arg; w4 = N.w4; port = 0; succ(0); }
            else { act = A_SLICE; J = N.fn_arg; w4 = N.w4; }
            break;
          case SPLIT:
            if (dir == FWD) { act = A_SLICE; J = N.fn_arg; w4 = N.w4; }
            else { join(u, N.U, aport, N.fn_arg, N.fn_arg); act = A_CONCAT; J = N.fn_arg; w4 = N.w4; pred(0); }
            break;
          case GROUP:
            if (dir == FWD) {
              int k = 0, member = u, count = 1;
              if (N.fn == 1) { k = I.etype[ebase + u]; member = I.rank_type[ebase + u]; const long long* o = I.type_off + inst * I.NT + k; count = (int)(o[1] - o[0]); }
              else if (N.fn == 2) { k = I.edst[ebase + u]; member = I.rank_in[ebase + u]; count = (int)(I.in_off[ibase + k + 1] - I.in_off[ibase + k]); }
              else count = (int)(I.offsets[inst + 1] - ibase);
              join(k, N.U, member, N.J, count);
              at_u(k);
              act = A_GATHER; succ(0);
            } else { act = A_SPREAD; reps = it.n; }
            break;
          case UNGROUP:
            if (dir == FWD) { act = A_SPREAD; reps = it.n; }
            else {
              int k = 0, row = u, count = 1;
              if (N.fn == 2) { k = I.etype[ebase + u]; row = I.rank_type[ebase + u]; const long long* o = I.type_off + inst * I.NT + k; count = (int)(o[1] - o[0]); }
              else if (N.fn == 3) {
                const long long l0 = I.leaf_off[inst];
                count = (int)(I.leaf_off[inst + 1] - l0);
                int lo = 0, hi = count - 1;
                while (lo < hi) { const int mid = (lo + hi) >> 1; if (I.leaf_ids[l0 + mid] < u) lo = mid + 1; else hi = mid; }
                row = lo;
              } else count = (int)(I.offsets[inst + 1] - ibase);
              join(k, N.U, row, N.J, count);
              at_u(k);
              act = A_GATHER; pred(0);
            }
            break;
          case FLATMAP:
            if (dir == FWD) { act = A_MULTI; reps = (int)(I.out_off[ibase + u + 1] - I.out_off[ibase + u]); }
            else {
              const int v = I.esrc[ebase + u], deg = (int)(I.out_off[ibase + v + 1] - I.out_off[ibase + v]);
              join(v, N.U, I.rank_out[ebase + u], N.J, deg);
              at_u(v);
              act = A_SUMREFS; J = deg; pred(0);
            }
            break;
          case NPT_SUMROWS: {
            const unsigned k = N.cnt_off + key(it.state, u, N.U);
            if (dir == FWD) { scr[k] = it.n; act = A_SUMALL; succ(0); }
            else { act = A_REP; reps = (int)scr[k]; scr[k] = 0; pred(0); }
          } break;
          default: status = ST_OVERFLOW;
        }
        if (act != A_PASS || status) break;
        node = to; aport = to_port; dir = to_dir; sport = port; u = state >> 16;
        it.where = pack_where(node, aport, dir, sport); it.state = state;
        NP = &M.nodes[node];
      }
      if (__any_sync(FULL, status)) return;                    // (a failed join left no reference)
      if (cnt != NONE) {                                       // joins: references first (above), then the counters
        const unsigned old = atomicAdd(&scr[cnt], 1u);
        if (old == 0) pending++;
        if (old + 1 == expected) { scr[cnt] = 0; pending--; } else act = A_NONE;
      }
      __syncwarp();
      // ---- sizes of what this lane builds ------------------------------------------------------------------
      unsigned want_rows = 0, want_terms = 0, pushes = 0;
      auto nt_of = [&](unsigned r) { const Row x = rows[r]; return x.nt == NONE ? 0u : x.nt; };
      switch (act) {
        case A_PASS: pushes = 1; break;
        case A_FORK: case A_SPREAD: case A_MULTI: pushes = reps; break;
        case A_SLICE:
          pushes = J; want_rows = J * nr;
          for (unsigned r = 0; r < nr; r++) {
            const Row x = rows[rs + r];
            for (unsigned q = 0; q < x.nt; q++) { const Term t = terms[x.ts + q]; want_terms += (t.col4 + t.w4 + w4 - 1) / w4 - t.col4 / w4; }
          }
          break;
        case A_CONCAT: case A_SUM:
          pushes = 1; want_rows = nr;
          for (int j = 0; j < J; j++) for (unsigned r = 0; r < nr; r++) want_terms += nt_of(scr[ref + j] + r);
          break;
        case A_GATHER: pushes = 1; want_rows = expected; nr = expected; break;
        case A_SUMALL: pushes = 1; want_rows = 1; for (unsigned r = 0; r < nr; r++) want_terms += nt_of(rs + r); break;
        case A_SUMREFS: pushes = 1; want_rows = 1; for (int j = 0; j < J; j++) want_terms += nt_of(scr[ref + j]); break;
        case A_REP: pushes = 1; if (reps >= 0) nr = reps; want_rows = nr; break;
        default: break;
      }
      if (want_rows > 2000 || want_terms > 2000 || pushes > 1000) status = ST_OVERFLOW;
      // one scan for everything: row records and terms, messages to push and to land (sixteen bits each)
      unsigned sa = want_rows | (want_terms << 16), sb = pushes | (act == A_LAND ? 1u << 16 : 0u);
      const unsigned wa = sa, wb = sb;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(FULL, sa, o), y = __shfl_up_sync(FULL, sb, o);
        if (lane >= o) { sa += x; sb += y; }
      }
      const unsigned ta = __shfl_sync(FULL, sa, 31), tb = __shfl_sync(FULL, sb, 31);
      sa -= wa; sb -= wb;
      const unsigned r0 = n_rows + (sa & 0xffffu), t0 = n_terms + (sa >> 16), push_at = sp + (sb & 0xffffu), land_at = n_front[next] + (sb >> 16);
      n_rows += ta & 0xffffu; n_terms += ta >> 16;
      if (n_rows > M.row_cap || n_terms > M.term_cap || sp + (tb & 0xffffu) > STACK || n_front[next] + (tb >> 16) > M.front_cap) status = ST_OVERFLOW;
      if (__any_sync(FULL, status)) return;
      // ---- build ---------------------------------------------------------------------------------------------
      unsigned tc = t0;
      switch (act) {
        case A_SLICE:
          for (int k = 0; k < J; k++)
            for (unsigned r = 0; r < nr; r++) {
              const Row x = rows[rs + r];
              const unsigned first = tc;
              for (unsigned q = 0; q < x.nt; q++) {
                const Term t = terms[x.ts + q];
                const unsigned lo = max((unsigned)t.col4, k * w4), hi = min((unsigned)t.col4 + t.w4, (k + 1) * w4);
                if (lo < hi) terms[tc++] = Term{t.src4 + (lo - t.col4), (unsigned short)(lo - k * w4), (unsigned short)(hi - lo)};
              }
              rows[r0 + k * nr + r] = Row{first, tc - first};
            }
          break;
        case A_CONCAT: case A_SUM:
          for (unsigned r = 0; r < nr; r++) {
            const unsigned first = tc;
            for (int j = 0; j < J; j++) {
              const Row x = rows[scr[ref + j] + r];
              for (unsigned q = 0; q < x.nt; q++) { Term t = terms[x.ts + q]; if (act == A_CONCAT) t.col4 += (unsigned short)(j * w4); terms[tc++] = t; }
            }
            rows[r0 + r] = Row{first, tc - first};
          }
          rs = r0;
          break;
        case A_GATHER: for (unsigned r = 0; r < nr; r++) rows[r0 + r] = rows[scr[ref + r]]; rs = r0; break;
        case A_SUMALL: case A_SUMREFS: {
          const int m = act == A_SUMALL ? (int)nr : J;
          for (int j = 0; j < m; j++) {
            const Row x = rows[act == A_SUMALL ? rs + j : scr[ref + j]];
            for (unsigned q = 0; q < x.nt; q++) terms[tc++] = terms[x.ts + q];
          }
          rows[r0] = Row{t0, tc - t0};
          rs = r0; nr = 1;
        } break;
        case A_REP: { const Row x = reps >= 0 ? rows[rs] : Row{0, 0}; for (unsigned r = 0; r < nr; r++) rows[r0 + r] = x; rs = r0; } break;
        default: break;
      }
      // ---- push ------------------------------------------------------------------------------------------------
      for (unsigned k = 0; k < pushes; k++) {
        Item o{pack_where(to, to_port, to_dir, port), state, rs, nr};
        switch (act) {
          case A_FORK: o.where = pack_where(N.succ_node[k], N.succ_port[k], FWD, port); break;
          case A_SLICE:
            o.rs = r0 + k * nr;
            if (dir == FWD) o.where = pack_where(N.succ_node[k], N.succ_port[k], FWD, port);                       // SPLIT
            else if (N.fn == 2) o.where = pack_where(N.pred_node[0], N.pred_port[0], BWD, k);
            else o.where = pack_where(N.pred_node[k], N.pred_port[k], BWD, port);
            break;
          case A_SPREAD: {
            int mu = k;
            if (N.type == GROUP) { if (N.fn == 1) mu = I.type_list[I.type_off[inst * I.NT + u] + k]; else if (N.fn == 2) mu = I.in_list[I.in_off[ibase + u] + k]; }
            else mu = N.fn == 2 ? I.type_list[I.type_off[inst * I.NT + u] + k] : N.fn == 3 ? I.leaf_ids[I.leaf_off[inst] + k] : (int)k;
            o.rs = rs + k; o.n = 1; o.state = (it.state & 0xffff) | ((unsigned)mu << 16);
            if (dir == FWD) o.where = pack_where(N.succ_node[0], N.succ_port[0], FWD, port); else o.where = pack_where(N.pred_node[0], N.pred_port[0], BWD, port);
          } break;
          case A_MULTI:
            o.where = pack_where(N.succ_node[0], N.succ_port[0], FWD, port);
            o.state = (it.state & 0xffff) | ((unsigned)I.out_list[I.out_off[ibase + u] + k] << 16);
            break;
          default: break;
        }
        stack[push_at + k] = o;
      }
      sp += tb & 0xffffu;
      // ---- landings at parameterised nodes -----------------------------------------------------------------------
      Item ev = it;
      if (act == A_LAND) {
        if (N.type == NPT_LSTM) {
          ev.where = pack_where(to, 0, dir, 0);
          if (dir == FWD) ev.rs = scr[ref];
        }
      }
      if (act == A_LAND) front[next][land_at] = ev;
      n_front[next] += tb >> 16;
      __syncwarp();
    }
#undef N
  }

  // ---- step t: the messages of frontier f; what they cause goes to the next frontier ------------------------------------
  __device__ void entry(const bool yes, const int cell, Entry e, const unsigned trs, const bool with_terms) {
    // (all lanes; rank among the lanes that write to the same cell)
    const unsigned mine = yes ? (unsigned)cell : 0x80u;
    const unsigned peers = __match_any_sync(FULL, mine);
    const unsigned rank = __popc(peers & ((1u << lane) - 1u));
    unsigned base = 0;
    if (yes) base = cur[cell];
    __syncwarp();
    if (yes && rank == 0) cur[cell] = base + __popc(peers);
    __syncwarp();
    if (!yes) return;
    unsigned nt = 0;
    Row x{0, 0};
    if (with_terms) { x = rows[trs]; nt = x.nt; }
    if (nt == NONE) { e.meta |= E_DENSE; nt = 0; }
    if (nt > 0xff) { status = ST_OVERFLOW; return; }
    e.meta |= nt;
    if (nt > 4) {
      n_ov += nt;
      if (EMIT && !ovp) { status = ST_OVERFLOW; return; }
      if (EMIT) {
        const unsigned o = atomicAdd(ov_cursor, nt);
        for (unsigned q = 0; q < nt; q++) ovp[o + q] = terms[x.ts + q];
        e.meta |= E_OVERFLOW; e.t[0].src4 = o;
      }
    } else if (EMIT) for (unsigned q = 0; q < nt; q++) e.t[q] = terms[x.ts + q];
    if (EMIT && base + rank < cell_end[cell]) ent[cell][base + rank] = e;
  }

  __device__ void step(const int f) {
    const int next = f == 2 ? 0 : f + 1;
    unsigned nf = n_front[f];
    for (unsigned b0 = 0; b0 < nf && !__any_sync(FULL, status); b0 += 32) {
      const bool live = b0 + lane < nf;
      Item ev{};
      if (live) ev = front[f][b0 + lane];
      const int node = ev.where & 0xff, dir = (ev.where >> 16) & 1;
      const bool deferred = live && ((ev.where >> 8) & 0xff) == OUT_PORT;
      const EncPpt& P = M.ppts[live ? M.nodes[node].ppt : 0];
      const bool gru = P.kind == GRUCELL, lookup = P.kind == LOOKUP, head = P.head >= 0, lstm = P.lstm >= 0;
      const int u = ev.state >> 16;
      const unsigned k = live ? key(ev.state, u, P.U) : 0;
      if (__any_sync(FULL, status)) return;
      // arena rows of this message, row records of what it emits
      const int H4 = P.out4;
      unsigned size4 = 0;
      bool emits = false;
      if (live && !deferred) {
        if (lookup) { size4 = dir == FWD ? P.out4 : 0; emits = dir == FWD; }
        else if (gru) { size4 = dir == FWD ? 7 * H4 + 1 : 8 * H4; emits = true; }
        else if (lstm) { size4 = dir == FWD ? P.gates4 + 2 * H4 + 1 + (M.nodes[P.lstm].fn == 2 ? 2 * H4 : 0) : P.in4 + P.gates4 + 2 * H4; emits = true; }
        else if (head) { size4 = P.in4 + P.out4 + (P.xstore ? P.in4 : 0); emits = !P.source_adj; }
        else if (dir == FWD) { size4 = P.out4 + 1 + (P.xstore ? P.in4 : 0); emits = true; }
        else { size4 = P.source_adj ? 0 : P.in4 + P.out4; emits = !P.source_adj; }
      }
      const unsigned n = (live && !deferred) ? ev.n : 0;
      unsigned base4, total4;
      base4 = arena4 + warp_excl(n * size4, total4);
      arena4 += total4;
      const int streams = (lstm && dir == BWD && M.nodes[P.lstm >= 0 ? P.lstm : 0].fn == 2) ? 2 : 1;
      const unsigned r0 = alloc(emits ? n * streams : 0, n_rows, M.row_cap), t0 = alloc(emits ? n * streams : 0, n_terms, M.term_cap);
      if (__any_sync(FULL, status)) return;
      unsigned fwd4 = 0, xrs = 0, crs = 0;
      if (live && !deferred) {
        if (dir == FWD && lstm && M.nodes[P.lstm].fn == 2) crs = scr[M.nodes[P.lstm].ref_off + key(ev.state, u, M.nodes[P.lstm].U) * M.nodes[P.lstm].J + 1];
        if (dir == FWD) { scr[P.save_off + k * 3] = base4; scr[P.save_off + k * 3 + 1] = ev.rs; fwd4 = base4; xrs = ev.rs; }
        else { fwd4 = scr[P.save_off + k * 3]; xrs = scr[P.save_off + k * 3 + 1]; }
        if (head) msgs_b++, msgs_f++;                          // the Loss and the backward message it answers with
      }
      // ---- entries, row by row ----------------------------------------------------------------------------------------
      unsigned total, first = warp_excl(n, total);
      for (unsigned j0 = 0; j0 < total; j0 += 32) {
        const unsigned j = j0 + lane;
        int src = 0;                                           // lane whose message row j belongs to
#pragma unroll
        for (int o = 16; o; o >>= 1) { const unsigned v = __shfl_sync(FULL, first, min(src + o, 31)); if (src + o < 32 && v <= j) src += o; }
        // (lanes without rows share `first` with the next one that has some; the search ends at the last such lane)
        const unsigned row = j - __shfl_sync(FULL, first, src), rn = __shfl_sync(FULL, n, src);
        const bool on = j < total;
        const int snode = __shfl_sync(FULL, node, src), sdir = __shfl_sync(FULL, dir, src), su = __shfl_sync(FULL, u, src);
        const unsigned sbase = __shfl_sync(FULL, base4, src) + row * __shfl_sync(FULL, size4, src), srs = __shfl_sync(FULL, ev.rs, src) + row;
        const unsigned sr0 = __shfl_sync(FULL, r0, src) + row, st0 = __shfl_sync(FULL, t0, src) + row, sxrs = __shfl_sync(FULL, xrs, src) + row, scrs = __shfl_sync(FULL, crs, src) + row;
        const unsigned sfwd = __shfl_sync(FULL, fwd4, src);
        const bool semits = __shfl_sync(FULL, emits, src);
        const EncPpt& Q = M.ppts[M.nodes[snode].ppt];
        const unsigned end = row + 1 == rn ? E_MSG_END : 0u;
        const int h4 = Q.out4;
        Entry e{}, e2{};
        int cell = -1, cell2 = -1;
        bool terms1 = true, terms2 = false;
        unsigned trs = srs, trs2 = 0, out4 = sbase, out_w = 0;
        e.meta = e2.meta = end;
        bool three = false;                                     // GRU: a third and fourth entry of the same block
        Entry e3{}, e4{};
        if (on) {
          if (Q.kind == LOOKUP) {
            cell = Q.cell[sdir];
            long long pos = ibase + su;
            if (Q.src_fn == 5) pos = ibase + row;
            else if (Q.src_fn == 6) pos = ibase + I.leaf_ids[I.leaf_off[inst] + row];
            e.b4 = (unsigned)I.tokens[pos];
            e.out4 = sbase; out_w = Q.out4;
            terms1 = sdir == BWD;
          } else if (Q.kind == GRUCELL) {
            const unsigned fblk = sdir == FWD ? sbase : sfwd + row * (7 * h4 + 1);
            e.out4 = e2.out4 = fblk;
            e.a4 = e2.a4 = sbase;
            if (sdir == FWD) {
              cell = Q.cell[0]; cell2 = Q.cell[1]; out4 = fblk + 6 * h4; out_w = h4;
              e2.t[0] = Term{fblk, 0, (unsigned short)h4}; e2.t[1] = Term{fblk + 4 * h4, (unsigned short)h4, (unsigned short)h4}; e2.meta |= 2;
            }
            else {
              cell = Q.cell[2]; cell2 = Q.cell[3]; out4 = sbase + 6 * h4; out_w = 2 * h4;
              three = true;
              e3.meta = e4.meta = end; e3.a4 = e4.a4 = fblk + 7 * h4;
              e3.out4 = sbase + 3 * h4; e3.t[0] = Term{fblk, 0, (unsigned short)h4}; e3.t[1] = Term{fblk + 4 * h4, (unsigned short)h4, (unsigned short)h4}; e3.meta |= 2;
              e4.out4 = sbase + h4; e4.t[0] = Term{fblk, 0, (unsigned short)(2 * h4)}; e4.meta |= 1;
            }
          } else if (Q.lstm >= 0) {
            const bool br = M.nodes[Q.lstm].fn == 2;
            const unsigned fsize = Q.gates4 + 2 * h4 + 1 + (br ? 2 * h4 : 0), fblk = sdir == FWD ? sbase : sfwd + row * fsize;
            e.a4 = fblk;
            if (sdir == FWD) { cell = Q.cell[0]; e.out4 = fblk; out4 = fblk + Q.gates4; out_w = 2 * h4; }
            else {
              cell = Q.cell[1]; e.out4 = sbase; out_w = Q.in4;
              cell2 = Q.cell[2]; e2.out4 = sbase + Q.in4; e2.a4 = fblk + Q.gates4 + 2 * h4; terms2 = true; trs2 = sxrs;
            }
          } else if (Q.head >= 0) {
            cell = Q.cell[0]; e.out4 = sbase; e.a4 = sbase + Q.in4; out_w = Q.in4;
            const EncNode& L = M.nodes[Q.head];
            e.b4 = L.type == LOSS_CE ? (unsigned)I.labels_i[I.labels_per_node ? ibase + su : inst] : __float_as_uint(I.labels_f[inst]);
            cell2 = Q.cell[1]; e2.out4 = e.a4; e2.a4 = NONE; terms2 = true; trs2 = srs;
          } else if (sdir == FWD) {
            cell = Q.cell[0]; e.out4 = sbase; e.a4 = Q.xstore ? sbase + Q.out4 + 1 : NONE; out_w = Q.out4;
          } else {
            const unsigned y = sfwd + row * (Q.out4 + 1 + (Q.xstore ? Q.in4 : 0));
            if (Q.source_adj) {                                 // no input gradient: the accumulator takes the gradient itself
              cell = Q.cell[2]; e.out4 = NONE; e.a4 = y; e.meta |= E_RAW;
            } else {
              cell = Q.cell[1]; e.out4 = sbase; e.a4 = y; e.b4 = sbase + Q.in4; out_w = Q.in4;
              cell2 = Q.cell[2]; e2.out4 = e.b4; e2.a4 = y + Q.out4; terms2 = true; trs2 = sxrs;
            }
          }
        }
        // an input that was summed is kept as a row of its own: the accumulator reads that one
        const bool kept = on && Q.xstore && cell2 >= 0 && terms2;
        if (kept) {
          terms2 = false;
          const unsigned x4 = Q.head >= 0 ? sbase + Q.in4 + Q.out4 : e2.a4 + 1;
          e2.t[0] = Term{x4, 0, (unsigned short)Q.in4};
          e2.meta |= 1;
        }
        if (on && Q.kind == LINEAR && Q.lstm >= 0 && sdir == FWD && M.nodes[Q.lstm].fn == 2) {
          // input terms, then the children's cells': at most two each (a Concat of two copies)
          const Row a = rows[srs], c = rows[scrs];
          if (a.nt + c.nt > 4) status = ST_OVERFLOW;
          else {
            for (unsigned q = 0; q < a.nt; q++) e.t[q] = terms[a.ts + q];
            for (unsigned q = 0; q < c.nt; q++) e.t[a.nt + q] = terms[c.ts + q];
            e.meta |= a.nt | (c.nt << 16);
            terms1 = false;
          }
        }
        entry(on && cell >= 0, cell, e, trs, terms1);
        entry(on && cell2 >= 0, cell2, e2, trs2, terms2);
        if (__any_sync(FULL, three)) {
          entry(three, Q.cell[4], e3, 0, false);
          entry(three, Q.cell[5], e4, 0, false);
        }
        if (on && semits) {
          terms[st0] = Term{out4, 0, (unsigned short)out_w};
          rows[sr0] = Row{st0, 1};
          if (Q.lstm >= 0 && sdir == BWD && M.nodes[Q.lstm].fn == 2) {      // second stream: the children's cells' gradient
            terms[st0 + rn] = Term{sbase + Q.in4 + Q.gates4, 0, (unsigned short)(2 * h4)};
            rows[sr0 + rn] = Row{st0 + rn, 1};
          }
        }
      }
      // ---- emissions -------------------------------------------------------------------------------------------------
      Item o = ev;
      o.rs = deferred ? ev.rs : r0;
      const bool late = live && gru && !deferred;               // a GRU's result is there one step later
      const bool out_fwd = dir == FWD && !head;
      Item d = o;
      d.where = pack_where(node, OUT_PORT, dir, (ev.where >> 20) & 0xff);
      land(late, d, next);
      unsigned sp = 0;
      const bool push = live && (deferred || (emits && !gru)), home = live && !deferred && !emits && (dir == BWD || head);
      if (push) {
        const EncNode& N = M.nodes[node];
        const EncNode& S = lstm ? M.nodes[P.lstm] : N;          // the gate node emits for its Linear
        const int sport = (ev.where >> 20) & 0xff;
        o.where = out_fwd ? pack_where(S.succ_node[0], S.succ_port[0], FWD, sport) : pack_where(N.pred_node[0], N.pred_port[0], BWD, sport);
        if (lstm && dir == FWD) { msgs_f++; }
      }
      unsigned cnt;
      const unsigned at = warp_excl(push ? 1u : 0u, cnt);
      if (push) stack[at] = o;
      sp = cnt;
      const bool second = push && streams == 2;
      const unsigned at2 = warp_excl(second ? 1u : 0u, cnt);
      if (second) { const EncNode& S = M.nodes[P.lstm]; Item c = o; c.where = pack_where(S.pred_node[1], S.pred_port[1], BWD, (ev.where >> 20) & 0xff); c.rs = r0 + n; stack[sp + at2] = c; }
      sp += cnt;
      if (home) retired++;                                      // a source-fed node answers the controller
      __syncwarp();
      drain(sp, next);
    }
    n_front[f] = 0;
  }

  // ---- the source messages --------------------------------------------------------------------------------------------
  __device__ int pump() {
    int pumped = 0;
    for (int s = 0; s < M.n_sources; s++) {
      const EncNode& N = M.nodes[M.sources[s]];
      const int to = N.succ_node[0], tp = N.succ_port[0];
      int count = 1, rows_each = 1;
      if (N.fn == 2) count = (int)(I.offsets[inst + 1] - ibase);
      else if (N.fn == 4) count = (int)(I.leaf_off[inst + 1] - I.leaf_off[inst]);
      else if (N.fn == 5) rows_each = (int)(I.offsets[inst + 1] - ibase);
      else if (N.fn == 6) rows_each = (int)(I.leaf_off[inst + 1] - I.leaf_off[inst]);
      pumped += count;
      const bool token = N.fn != 1 && N.fn != 3;
      for (int c0 = 0; c0 < count && !__any_sync(FULL, status); c0 += 32) {
        const bool live = c0 + lane < count;
        const unsigned r0 = alloc(live && !token ? 1 : 0, n_rows, M.row_cap);
        if (live && !token) rows[r0] = Row{0, N.fn == 1 ? NONE : 0u};
        const int u = N.fn == 4 && live ? I.leaf_ids[I.leaf_off[inst] + c0 + lane] : N.fn == 2 ? c0 + lane : 0;
        const Item it{pack_where(to, tp, FWD, 0), (unsigned)u << 16, r0, (unsigned)rows_each};
        unsigned cnt;
        const unsigned at = warp_excl(live ? 1u : 0u, cnt);
        if (live) stack[at] = it;
        unsigned sp = cnt;
        __syncwarp();
        drain(sp, 0);
      }
    }
    return pumped;
  }

  __device__ void run(long long i, InstHdr& H, unsigned tab0, unsigned* const* tab, int& left) {
    inst = i;
    ibase = I.offsets ? I.offsets[i] : 0;
    ebase = I.edge_off ? I.edge_off[i] : 0;
    n_front[0] = n_front[1] = n_front[2] = 0;
    n_rows = n_terms = 0; arena4 = 0; n_ov = 0; msgs_f = msgs_b = 0; pending = retired = status = 0;
    const unsigned my0 = lane < M.n_cells ? cur[lane] : 0;      // entries before this instance
    int steps = 0, steps_eval = 0;
    const int last_steps = EMIT ? H.steps : 0;
    if (EMIT && lane < M.n_cells) for (int d = 0; d <= M.delay[lane]; d++) if (d <= last_steps) tab[lane][tab0 + d] = my0;
    __syncwarp();
    const int pumped = pump();
    int t = 0, f = 0;
    for (; n_front[f] > 0 && !__any_sync(FULL, status); t++) {
      const unsigned before = lane < M.n_cells ? cur[lane] : 0;
      __syncwarp();
      step(f);
      f = f == 2 ? 0 : f + 1;
      if (lane < M.n_cells) {
        const unsigned now = cur[lane];
        const int at = t + M.delay[lane] + 1;
        if (now != before) { steps = at; if (M.forward[lane]) steps_eval = at; }
        if (EMIT && at <= last_steps) tab[lane][tab0 + at] = now;
      }
      __syncwarp();
      if (t > 60000) { status = ST_OVERFLOW; }
    }
    auto sum = [&](int v) { for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o); return v; };
    auto most = [&](int v) { for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(FULL, v, o)); return v; };
    left = sum(pending) + (pumped - sum(retired));
    status = most(status);
    H.msgs = (unsigned)sum((int)(msgs_f + msgs_b)); H.msgs_eval = (unsigned)sum((int)msgs_f);
    steps = most(steps); steps_eval = most(steps_eval);
    if (EMIT && lane < M.n_cells) for (int s = t + M.delay[lane] + 1; s <= min(steps, last_steps); s++) tab[lane][tab0 + s] = cur[lane];
    if (EMIT && steps > last_steps) status = ST_OVERFLOW;
    if (steps > 65000) status = ST_OVERFLOW;
    H.steps = (unsigned short)steps; H.steps_eval = (unsigned short)steps_eval;
    n_ov = (unsigned)sum((int)n_ov);
    __syncwarp();
  }
};

__device__ void summarise(EncTotals* totals, const InstHdr& H, unsigned arena4, unsigned n_ov, int status, int left) {
  if (status || left) atomicCAS(&totals->status, 0, status ? status : -1);               // every message must be answered
  if (n_ov) atomicAdd(&totals->ov, (unsigned long long)n_ov);
  atomicMax(&totals->arena4_max, arena4);
  atomicMin(&totals->steps_min, (unsigned)H.steps); atomicMin(&totals->steps_eval_min, (unsigned)H.steps_eval);
  atomicAdd(&totals->steps_sum, (unsigned long long)H.steps); atomicAdd(&totals->steps_eval_sum, (unsigned long long)H.steps_eval);
}

__global__ void __launch_bounds__(EW * 32) encode_kernel(const __grid_constant__ EncModel M, const __grid_constant__ DevInst I, unsigned* scratch, const __grid_constant__ Program prog,
                                                         InstHdr* hdr, unsigned* counts, Term* ov, EncTotals* totals, const int emit) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ unsigned cursors[EW][MAX_CELLS];
  __shared__ Entry* ents[MAX_CELLS];
  __shared__ unsigned ends[MAX_CELLS];
  __shared__ unsigned* tabs[MAX_CELLS];
  __shared__ EncModel SM;                // (node tables are indexed by message: not from the constant bank)
  for (unsigned k = threadIdx.x; k < sizeof(EncModel) / 4; k += blockDim.x) reinterpret_cast<unsigned*>(&SM)[k] = reinterpret_cast<const unsigned*>(&M)[k];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (threadIdx.x < MAX_CELLS) { ents[threadIdx.x] = const_cast<Entry*>(prog.ent[threadIdx.x]); tabs[threadIdx.x] = const_cast<unsigned*>(prog.tab[threadIdx.x]); ends[threadIdx.x] = emit == 2 && threadIdx.x < M.n_cells ? M.bound[threadIdx.x] * (unsigned)I.n : 0xffffffffu; }
  __syncthreads();
  Item* const stack = reinterpret_cast<Item*>(dyn) + (size_t)warp * M.stack_cap;
  unsigned* const cur = cursors[warp];
  const long long gw = (long long)blockIdx.x * warps + warp, nw = (long long)gridDim.x * warps;
  unsigned* const scr = M.near_scratch ? reinterpret_cast<unsigned*>(dyn + (size_t)warps * M.stack_cap * sizeof(Item)) + (size_t)warp * M.scratch_words : scratch + (size_t)gw * M.scratch_words;
  if (M.near_scratch) { for (unsigned k = lane; k < M.table_words; k += 32) scr[k] = 0; __syncwarp(); }
  const long long n = I.n;
  for (long long i = gw; i < n; i += nw) {
    int left = 0;
    if (emit) {
      Encoder<true> E(SM, I, scr, stack, cur);
      E.ent = ents; E.ovp = ov; E.ov_cursor = &totals->ov_used; E.cell_end = ends;
      // (emit 2: every instance has room for the most it can need, nothing was counted before)
      const bool bounded = emit == 2;
      const unsigned base = lane < M.n_cells ? (bounded ? (unsigned)i * M.bound[lane] : counts[(size_t)lane * n + i]) : 0;
      if (lane < M.n_cells) cur[lane] = base;
      __syncwarp();
      InstHdr H{};
      if (bounded) { H.tab = (unsigned)i * M.steps_cap; H.steps = (unsigned short)(M.steps_cap - 1); } else H = hdr[i];
      const unsigned tab0 = H.tab;
      E.run(i, H, tab0, tabs, left);
      if (bounded && lane < M.n_cells) { atomicAdd(&totals->entries[lane], cur[lane] - base); if (cur[lane] - base > M.bound[lane]) E.status = ST_OVERFLOW; }
      if (E.status) atomicCAS(&totals->status, 0, E.status);
      if (bounded && lane == 0) { H.tab = tab0; hdr[i] = H; summarise(totals, H, E.arena4, E.n_ov, E.status, left); }
      if (__any_sync(FULL, E.status) || left) return;          // (its tables are not clean for another instance; the program is void)
    } else {
      Encoder<false> E(SM, I, scr, stack, cur);
      E.ent = nullptr; E.ovp = nullptr; E.ov_cursor = nullptr;
      if (lane < M.n_cells) cur[lane] = 0;
      __syncwarp();
      InstHdr H{};
      E.run(i, H, 0, tabs, left);
      if (lane < M.n_cells) counts[(size_t)lane * n + i] = cur[lane];
      if (lane == 0) {
        hdr[i] = H;
        summarise(totals, H, E.arena4, E.n_ov, E.status, left);
      }
      if (__any_sync(FULL, E.status) || left) return;
    }
    __syncwarp();
  }
}

// Exclusive prefix sums over the instances, a block per cell (the last one: the instances' first table entries).
__global__ void __launch_bounds__(1024) scan_kernel(unsigned* counts, InstHdr* hdr, const long long n, const int n_cells, EncTotals* totals) {
  __shared__ unsigned long long part[32], block_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = blockIdx.x;
  unsigned long long carry = 0;                                // (sums beyond 32 bits void the program: offsets have no more)
  for (long long i0 = 0; i0 < n; i0 += 1024) {
    const long long i = i0 + tid;
    const unsigned v = i >= n ? 0u : c < n_cells ? counts[(size_t)c * n + i] : hdr[i].steps + 1u;
    unsigned long long total, all;                             // (a block's thousand counts may pass 32 bits between them)
    const unsigned long long ex = warp_excl64(v, total);
    if (lane == 31) part[warp] = total;
    __syncthreads();
    if (warp == 0) { const unsigned long long p = warp_excl64(part[lane], all); part[lane] = p; if (lane == 0) block_total = all; }
    __syncthreads();
    const unsigned out = (unsigned)(carry + part[warp] + ex);
    if (i < n) { if (c < n_cells) counts[(size_t)c * n + i] = out; else hdr[i].tab = out; }
    carry += block_total;
    __syncthreads();
  }
  if (tid == 0) {
    if (c < n_cells) totals->entries[c] = (unsigned)carry; else totals->tab = (unsigned)carry;
    if (carry > 0xffffffffull) atomicCAS(&totals->status, 0, ST_OVERFLOW);
  }
}

}  // namespace

int encode_warps_per_block() { return EW; }

static cudaError_t run_encode(const EncModel* m, const DevInst& inst, unsigned* scratch, int blocks, int warps, const Program& prog, InstHdr* hdr, unsigned* counts, Term* ov,
                              EncTotals* totals, int emit, cudaStream_t st) {
  const size_t smem = (size_t)warps * ((size_t)m->stack_cap * sizeof(Item) + (m->near_scratch ? (size_t)m->scratch_words * 4 : 0));
  const cudaError_t e = allow_dynamic_smem((const void*)encode_kernel, smem);
  if (e != cudaSuccess) return e;
  encode_kernel<<<blocks, warps * 32, smem, st>>>(*m, inst, scratch, prog, hdr, counts, ov, totals, emit);
  return cudaGetLastError();
}
cudaError_t encode_count(const EncModel* m, const DevInst& inst, unsigned* scratch, int blocks, int warps, InstHdr* hdr, unsigned* counts, EncTotals* totals, cudaStream_t st) {
  Program none{};
  return run_encode(m, inst, scratch, blocks, warps, none, hdr, counts, nullptr, totals, 0, st);
}
cudaError_t encode_emit(const EncModel* m, const DevInst& inst, unsigned* scratch, int blocks, int warps, const Program& prog, unsigned* counts, Term* ov, EncTotals* totals, cudaStream_t st) {
  return run_encode(m, inst, scratch, blocks, warps, prog, prog.hdr, counts, ov, totals, 1, st);
}
cudaError_t encode_bounded(const EncModel* m, const DevInst& inst, int blocks, int warps, const Program& prog, EncTotals* totals, cudaStream_t st) {
  return run_encode(m, inst, nullptr, blocks, warps, prog, prog.hdr, nullptr, nullptr, totals, 2, st);
}
cudaError_t encode_scan(unsigned* counts, InstHdr* hdr, long long n, int n_cells, EncTotals* totals, cudaStream_t st) {
  scan_kernel<<<n_cells + 1, 1024, 0, st>>>(counts, hdr, n, n_cells, totals);
  return cudaGetLastError();
}

}  // namespace wave
