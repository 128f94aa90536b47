// fp32-compute path of libslim: every supported (d, M, dtype, feature) that the
// tcgen05 tile kernels do not take.  Intermediates are fp32, or 2 (bf16
// problems) or 3 (fp32 problems) bf16 pieces of fp32 values where they are
// operands of a product; products run as warp MMAs over the pieces.
//
// Rows are cut into tiles of up to 64 and every step is a batch over (chain, tile) --
// App. B's "block" evaluation with the block's prefix sums written as masked
// matrix products:
//
//   forward (Sec. 3.2, eqs. 14-16):
//     phiQ, phiK = g(Q), g(K)                    (F, row-wise)
//     Delta_t    = phiK_t^T [V_t | 1]            (the tile's sum of T_l)
//     P_t        = B + sum_{t'<t} Delta_t'       (state before tile t)
//     A_t        = tril(phiQ_t phiK_t^T)         (inclusive causal mask)
//     [num|den]  = phiQ_t P_t + A_t [V_t | 1];  out = num / den   (eq. 4)
//     B         += sum_t Delta_t
//   backward (Sec. 3.3, eqs. 17-18), from B^(n), G^(n):
//     B -= sum_t Delta_t                          (eq. 17), then P_t as above
//     dnum = dout/den, dden = -<dout, out>/den,  W = [dnum | dden]
//     dA_t   = tril(W_t [V_t | 1]^T)
//     dphiQ  = W_t P_t^T + dA_t phiK_t
//     Gd_t   = phiQ_t^T W_t;   G_t = G + sum_{t'>t} Gd_t'   (reversed prefix sum)
//     dphiK  = dA_t^T phiQ_t + [V_t | 1] G_t^T
//     dV     = A_t^T dnum + phiK_t G_t(S part)
//     G     += sum_t Gd_t                           (eq. 18)
//     feature VJP: dq, dk; dOmega += u^T x
// The state B and its gradient G are carried as fp32 value/error pairs so the
// rollback returns the forward's state to within the pair's precision; it undoes
// the forward's own Delta_t, which the backward recomputes bit for bit (same
// kernel, same tiles).
//
// A launch sequence is 3 kernels forward (Delta; the carry; the readout) and 6
// backward (Delta; the rolled-back carry; the query side; the gradient's carry;
// the key side; dOmega).  The kernels are in simt_tiles.cuh and simt_carry.cu;
// this file cuts the rows into sequences and carves the workspace.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "simt_path.h"
#include "simt_short.h"
#include "simt_tiles.h"

namespace slim {
namespace simt {
namespace {

#define SLIM_TRY(x)                                   \
  do {                                                \
    cudaError_t e_ = (x);                             \
    if (e_ != cudaSuccess) return SLIM_ERR_CUDA;      \
  } while (0)

// A launch sequence covers `rows` rows of every chain in tiles of 64, or of the
// whole slice when it is shorter: the state is formed at every slice boundary
// (eq. 16), and a tile's rows are padded to a multiple of 16.  A sequence is a
// slice, or several: as many as fill the chip (kSeqFrames), and beyond that up to
// kSeqSlices within kMostFrames, because a launch of few waves (1 to 3 CTAs on an SM)
// loses much of its last one.  Train steps at 304 / 1216 / 2432 frames: [4,12,8192]
// fp32 relu, C = 512 (384 frames a slice) 6.43 / 5.46 / 5.36 ms; non-causal [8,8,4096]
// bf16, C = 1024 (1024 frames) 2.52 / 2.52 / 2.28 ms; L = 65536, C = 16 9.17 / 8.95 /
// 9.08 ms.  Short slices stay at the first: 1 to 2 % is not worth four to eight times the
// scratch (0.2 GB there).
constexpr int kSeqFrames = 2 * kSms;  // two CTAs on each SM
constexpr int kMostFrames = 16 * kSms;
constexpr int kSeqSlices = 8;
constexpr int kShortRows = 1024; // rows per chain of a sequence of slices below 64 rows, about

struct Seq {
  int chains, d, M, E;
  int slice;             // rows of a slice (of a tile when that is shorter than 64)
  int tile, pitch, per;  // a tile's padded rows and its rows; tiles per frame
  int rows, nt, nf, N;   // rows per sequence, tiles and frames per chain, sequences
  int ns;                // pieces per computed operand
  int slots;             // dOmega partials of a backward launch
  size_t frames, tiles;  // of all chains, that the workspace holds
};

// tiles of the first `rows` rows of a sequence (tiles start anew in every slice)
int tiles_of(int rows, int slice, int pitch) {
  const int per = (int)(((long long)slice + pitch - 1) / pitch);
  return rows / slice * per + (int)(((long long)(rows % slice) + pitch - 1) / pitch);
}

// The sweep of `chains` chains, with at most `limit` frames per sequence (but a slice, or a
// frame of short ones, of every chain at least); the tiles and the bits are the same for
// every limit.
//
// The workspace is sized by the most frames that a sequence may have, not by those
// that the even cut below leaves: it then falls neither with a shorter sequence nor with
// fewer chains, and a buffer for the largest of several problems serves them all.
constexpr long long kNoLimit = kMostFrames * (1LL << 24);
Seq sequence(const Problem& p, int chains, long long limit = kNoLimit) {
  Seq q;
  q.chains = chains;
  q.d = p.d;
  q.M = p.M;
  q.E = p.M * (p.d + 1);
  q.ns = p.dtype == SLIM_F32 ? 3 : 2;
  const int Cs = p.slice_len();
  q.pitch = Cs < kTile ? (Cs > 0 ? Cs : 1) : kTile;
  q.tile = (q.pitch + 15) / 16 * 16;
  q.per = q.tile <= 32 ? kTile / q.tile : 1;
  q.slice = Cs < kTile ? q.pitch : Cs;
  const long long frame = (long long)q.per * q.pitch;  // its rows
  // frames of one slice, or the one frame that several short ones share, of all chains
  const long long slice = Cs < kTile ? chains : (((long long)Cs + kTile - 1) / kTile) * chains;
  long long most = Cs < kTile ? (kShortRows + frame - 1) / frame * chains
                              : std::min<long long>(kSeqSlices * slice, kMostFrames);
  most = std::max(slice, std::min(limit, std::max<long long>(kSeqFrames, most)));
  long long rows = Cs;
  if (Cs < kTile) {
    rows = frame * (most / chains);
  } else if (most / slice > 1) {  // evenly: the same number of sequences, without a small last one
    const long long slices = most / slice, all = ((long long)p.L + Cs - 1) / Cs,
                    seqs = (all + slices - 1) / slices;
    rows = (all + seqs - 1) / seqs * Cs;
  }
  q.rows = (int)(rows < p.L ? rows : p.L);
  q.nt = tiles_of(q.rows, q.slice, q.pitch);
  q.nf = (q.nt + q.per - 1) / q.per;
  q.N = p.L == 0 ? 0 : (int)(((long long)p.L + q.rows - 1) / q.rows);
  const long long nt = tiles_of(p.L, q.slice, q.pitch);
  q.frames = (size_t)std::min(most, (nt + q.per - 1) / q.per * chains);
  q.tiles = (size_t)std::min<long long>(q.frames * q.per, nt * chains);
  const long long ctas = tile_kernels(p.dtype, p.d).slots;
  q.slots = (int)std::min<long long>(q.frames, ctas);
  return q;
}

struct SeqWs {
  int* err;
  float *st_hi, *st_lo, *delta, *zdelta, *om_t, *om_norm;
  __nv_bfloat16 *om_row, *phi_k;
  float *g_hi, *g_lo, *gdelta, *slots;
  __nv_bfloat16 *phi_q, *sA, *sdA, *sW;
};

// spare: room for any call of fewer rows too.  One frame of short tiles per chain keeps a pair
// and its tiles' z, more than the one frame of a slice of 33 to 64 rows.
SeqWs carve_seq(Carver& cv, const Seq& q, bool bwd, bool spare = true) {
  SeqWs w{};
  const size_t C = q.chains, frames = q.frames, least = spare ? C : 0;
  w.err = cv.take<int>(64);
  w.st_hi = cv.take<float>(C * q.E);
  w.st_lo = cv.take<float>(C * q.E);
  w.om_t = cv.take<float>((size_t)(q.M + 63) / 64 * 64 * q.d);
  w.om_row = cv.take<__nv_bfloat16>((size_t)3 * q.M * q.d);
  w.om_norm = cv.take<float>(q.M);
  w.delta = cv.take<float>(std::max(frames * (q.per > 1 ? 2 : 1), 2 * least) * q.E);
  w.zdelta = cv.take<float>(std::max(q.per > 1 ? q.tiles : 0, least) * q.M);
  w.phi_k = cv.take<__nv_bfloat16>(frames * q.ns * q.M * kTile);
  if (bwd) {
    w.g_hi = cv.take<float>(C * q.E);
    w.g_lo = cv.take<float>(C * q.E);
    w.gdelta = cv.take<float>(frames * q.E);
    w.phi_q = cv.take<__nv_bfloat16>(frames * q.ns * q.M * kTile);
    w.sA = cv.take<__nv_bfloat16>(frames * q.ns * kTile * kTile);
    w.sdA = cv.take<__nv_bfloat16>(frames * q.ns * kTile * kTile);
    w.sW = cv.take<__nv_bfloat16>(frames * q.ns * kTile * q.d);
    w.slots = cv.take<float>((size_t)q.slots * q.M * q.d);
  }
  return w;
}

TileArgs seq_args(const Problem& p, const Seq& q, const SeqWs& w, const void* qp, const void* kp,
                  const void* vp, const float* omega) {
  TileArgs A{};
  A.q = qp;
  A.k = kp;
  A.v = vp;
  A.omega = omega;
  A.om_t = w.om_t;
  A.om_row = w.om_row;
  A.om_norm = w.om_norm;
  A.delta = w.delta;
  A.zdelta = w.zdelta;
  A.phi_k = w.phi_k;
  A.gdelta = w.gdelta;
  A.phi_q = w.phi_q;
  A.sA = w.sA;
  A.sdA = w.sdA;
  A.sW = w.sW;
  A.slots = w.slots;
  A.L = p.L;
  A.M = q.M;
  A.E = q.E;
  A.chains = q.chains;
  A.rows = q.tile;
  A.pitch = q.pitch;
  A.slice = q.slice;
  A.slice_tiles = (q.slice + q.pitch - 1) / q.pitch;
  A.per = q.per;
  A.shift = q.per == 4 ? 4 : q.per == 2 ? 5 : 6;
  // reduction groups of short tiles' products over the features: as many as have
  // two k16 steps each
  auto groups = [&](int want) { return q.M >= 32 * want ? want : 1; };
  A.ks_n = A.ks_a = 1;
  if (q.tile == 16) {
    A.ks_n = groups(q.ns == 2 ? 4 : 2);
    A.ks_a = groups(q.ns == 2 ? 8 : 4);
  } else if (q.tile == 32) {
    A.ks_n = A.ks_a = groups(2);
  }
  A.feature = (int)p.feature;
  A.inv_sqrt_m = (float)(1.0 / sqrt((double)p.M));
  return A;
}

// rows [a, a + b) of sequence n, the per-tile state and its gradient in `delta`
// and `gdelta`
void seq_rows(TileArgs& A, const Problem& p, const Seq& q, int n) {
  A.a = n * q.rows;
  A.b = p.L - A.a < q.rows ? p.L - A.a : q.rows;
  A.nt = tiles_of(A.b, q.slice, q.pitch);
  A.nf = (A.nt + A.per - 1) / A.per;
  A.P = A.delta;
  A.p_frame = (q.per > 1 ? 2LL : 1LL) * q.E;
  A.p_chain = A.nf * A.p_frame;
  A.p_lo = q.E;
  A.G = A.gdelta;
  A.g_chain = (long long)A.nf * q.E;
  A.g_frame = q.E;
}

// the carry of the state (over `delta`) or of its gradient (over `gdelta`)
CarryArgs carry(const Seq& q, const SeqWs& w, const TileArgs& A, CarryMode mode, bool first,
                const StateInit& init, const StateOut& out) {
  const bool grad = mode == CARRY_GREV;
  return CarryArgs{grad ? w.gdelta : w.delta, !grad && q.per > 1, grad ? w.g_hi : w.st_hi,
                   grad ? w.g_lo : w.st_lo, q.chains, A.nf, q.M, q.d, mode, first ? 1 : 0, init, out};
}

const float* used_omega(const Problem& p, const float* omega) {
  return p.feature == SLIM_FEAT_SQUARE ? nullptr : omega;
}

// the same problem's pointers from chain c0 on
const void* rows_from(const Problem& p, const void* t, int c0) {
  return static_cast<const char*>(t) + (size_t)c0 * p.L * p.d * (p.dtype == SLIM_BF16 ? 2 : 4);
}
template <typename T>
T* off(T* t, size_t n) {
  return t ? t + n : nullptr;
}

// The forward of `chains` chains from chain c0.
slim_status fwd_chains(const Problem& p, int c0, const Seq& sq, const void* q, const void* k,
                       const void* v, const float* omega, void* out, StateOut st, StateInit init,
                       void* workspace, cudaStream_t s) {
  Carver cv(workspace);
  const SeqWs w = carve_seq(cv, sq, false, false);
  const TileKernels& tk = tile_kernels(p.dtype, p.d);
  const size_t so = (size_t)c0 * p.M * p.d, zo = (size_t)c0 * p.M;
  st = StateOut{off(st.S, so), off(st.z, zo), off(st.S_lo, so), off(st.z_lo, zo)};
  init = StateInit{off(init.S, so), off(init.z, zo), off(init.S_lo, so), off(init.z_lo, zo)};
  TileArgs A = seq_args(p, sq, w, rows_from(p, q, c0), rows_from(p, k, c0), rows_from(p, v, c0), omega);
  if (out)
    A.o = const_cast<void*>(rows_from(p, out, c0));
  else
    A.phi_k = nullptr;  // the state alone
  A.causal = 1;
  SLIM_TRY(launch_setup(s, used_omega(p, omega), sq.M, sq.d, w.om_t, w.om_row, w.om_norm, nullptr,
                        w.err));
  for (int n = 0; n < sq.N; ++n) {
    seq_rows(A, p, sq, n);
    SLIM_TRY(tk.delta(A, s));
    SLIM_TRY(launch_carry(s, carry(sq, w, A, CARRY_FWD, n == 0, init, n + 1 == sq.N ? st : StateOut{})));
    if (out) SLIM_TRY(tk.out(A, s));
  }
  return SLIM_OK;
}

size_t fwd_bytes(const Problem& p, int chains, long long limit) {
  Carver cv(nullptr);
  carve_seq(cv, sequence(p, chains, limit), false, limit == kNoLimit);
  return cv.bytes();
}

// dOmega partials that a launch on A's rows fills
int used_slots(const Seq& q, const TileArgs& A) {
  const long long frames = (long long)A.chains * A.nf;
  return (int)(frames < q.slots ? frames : q.slots);
}

slim_status bwd_impl(const Problem& p, const void* q, const void* k, const void* v,
                     const float* omega, const void* out, const void* dout,
                     const StateIn& st, const GradIO& gio, void* dq, void* dk, void* dv,
                     float* domega, void* workspace, cudaStream_t s) {
  const Seq sq = sequence(p, p.chains());
  Carver cv(workspace);
  const SeqWs w = carve_seq(cv, sq, true);
  const TileKernels& tk = tile_kernels(p.dtype, p.d);
  const float* om = used_omega(p, omega);
  SLIM_TRY(launch_setup(s, om, sq.M, sq.d, w.om_t, w.om_row, w.om_norm, domega, w.err));
  TileArgs A = seq_args(p, sq, w, q, k, v, omega);
  A.out = out;
  A.dout = dout;
  A.dq = dq;
  A.dk = dk;
  A.dv = dv;
  A.causal = 1;
  const StateInit b_in{st.S, st.z, st.S_lo, st.z_lo};
  const StateInit g_in{gio.S_in, gio.z_in, nullptr, nullptr};  // G^(N) (eq. 18), zero when null
  const StateOut g_out{gio.S_out, gio.z_out, nullptr, nullptr};  // G^(0)
  for (int n = sq.N - 1; n >= 0; --n) {
    const bool first = n + 1 == sq.N;
    seq_rows(A, p, sq, n);
    SLIM_TRY(tk.delta(A, s));
    SLIM_TRY(launch_carry(s, carry(sq, w, A, CARRY_ROLLBACK, first, b_in, StateOut{})));
    SLIM_TRY(tk.bwd_q(A, s));
    SLIM_TRY(launch_carry(s, carry(sq, w, A, CARRY_GREV, first, g_in, n == 0 ? g_out : StateOut{})));
    SLIM_TRY(tk.bwd_k(A, s));
    if (om) SLIM_TRY(launch_domega(s, w.slots, used_slots(sq, A), domega, sq.M, sq.d));
  }
  return SLIM_OK;
}

// ------------------------------------------------------------------ non-causal form
// Eq. 2 without the mask: one global state B = sum over all rows (eq. 3 at
// l = L) serves every row.  Memory stays O(C): the forward reads the slices
// twice (accumulate B, then read it out), the backward twice as well (query
// side, which also accumulates G = grad_B, then key/value side, which reads G).
slim_status fwd_bidir_impl(const Problem& p, const void* q, const void* k, const void* v,
                           const float* omega, void* out, const StateOut& st, void* workspace,
                           cudaStream_t s) {
  const Seq sq = sequence(p, p.chains());
  Carver cv(workspace);
  const SeqWs w = carve_seq(cv, sq, false);
  const TileKernels& tk = tile_kernels(p.dtype, p.d);
  SLIM_TRY(launch_setup(s, used_omega(p, omega), sq.M, sq.d, w.om_t, w.om_row, w.om_norm, nullptr,
                        w.err));
  TileArgs A = seq_args(p, sq, w, q, k, v, omega);
  A.o = out;
  A.phi_k = nullptr;
  // sweep 1: B = sum over every tile of g(K)^T [V | 1]
  for (int n = 0; n < sq.N; ++n) {
    seq_rows(A, p, sq, n);
    SLIM_TRY(tk.delta(A, s));
    SLIM_TRY(launch_carry(s, carry(sq, w, A, CARRY_SUM, n == 0, StateInit{}, n + 1 == sq.N ? st : StateOut{})));
  }
  // sweep 2: [num | den] = g(Q) B, out = num / den
  for (int n = 0; n < sq.N; ++n) {
    seq_rows(A, p, sq, n);
    A.P = w.st_hi;
    A.p_chain = sq.E;
    A.p_frame = 0;
    A.p_lo = w.st_lo - w.st_hi;  // the pair, as the forward leaves it per frame
    SLIM_TRY(tk.out(A, s));
  }
  return SLIM_OK;
}

slim_status bwd_bidir_impl(const Problem& p, const void* q, const void* k, const void* v,
                           const float* omega, const void* out, const void* dout,
                           const StateIn& st, void* dq, void* dk, void* dv, float* domega,
                           void* workspace, cudaStream_t s) {
  const Seq sq = sequence(p, p.chains());
  Carver cv(workspace);
  const SeqWs w = carve_seq(cv, sq, true);
  const TileKernels& tk = tile_kernels(p.dtype, p.d);
  const float* om = used_omega(p, omega);
  SLIM_TRY(launch_setup(s, om, sq.M, sq.d, w.om_t, w.om_row, w.om_norm, domega, w.err));
  TileArgs A = seq_args(p, sq, w, q, k, v, omega);
  A.out = out;
  A.dout = dout;
  A.dq = dq;
  A.dk = dk;
  A.dv = dv;
  // the global state as the kernels read it: a carry over no tiles
  SLIM_TRY(launch_carry(s, carry(sq, w, A, CARRY_SUM, true, StateInit{st.S, st.z, st.S_lo, st.z_lo},
                                 StateOut{})));
  // sweep 1, query side: dphiQ = W B^T, G += g(Q)^T W
  for (int n = 0; n < sq.N; ++n) {
    seq_rows(A, p, sq, n);
    A.P = w.st_hi;
    A.p_chain = sq.E;
    A.p_frame = 0;
    SLIM_TRY(tk.bwd_q(A, s));
    CarryArgs g = carry(sq, w, A, CARRY_GREV, n == 0, StateInit{}, StateOut{});
    g.mode = CARRY_SUM;
    SLIM_TRY(launch_carry(s, g));
    if (om) SLIM_TRY(launch_domega(s, w.slots, used_slots(sq, A), domega, sq.M, sq.d));
  }
  // sweep 2, key/value side: dphiK = [V | 1] G^T, dV = g(K) G_S
  A.slots_new = 1;
  for (int n = 0; n < sq.N; ++n) {
    seq_rows(A, p, sq, n);
    A.G = w.g_hi;
    A.g_chain = sq.E;
    A.g_frame = 0;
    SLIM_TRY(tk.bwd_k(A, s));
    if (om) SLIM_TRY(launch_domega(s, w.slots, used_slots(sq, A), domega, sq.M, sq.d));
  }
  return SLIM_OK;
}

}  // namespace

size_t workspace_bytes(const Problem& p, bool bwd, bool small) {
  if (!bwd) return small ? fwd_bytes(p, 1, 0) : fwd_bytes(p, p.chains(), kNoLimit);
  Carver cv(nullptr);
  carve_seq(cv, sequence(p, p.chains()), true);
  return cv.bytes();
}

size_t noalloc_bytes(const Problem& p) {
  const size_t n = p.chains(), M = p.M, d = p.d, dp = p.d + 1;
  const int Cs = p.slice_len();
  long long rows = Cs;
  int tile = Cs >= 64 ? 64 : Cs > 0 ? (Cs + 15) / 16 * 16 : 16;
  if (Cs < 64 && Cs % 16 == 0 && p.L > Cs) {
    tile = Cs;
    const long long whole = ((long long)p.L + tile - 1) / tile * tile, most = 1024 / tile * tile;
    rows = most < whole ? most : whole;
  }
  const size_t nt = (size_t)((rows + tile - 1) / tile), R = n * nt * tile;
  Carver cv(nullptr);
  cv.take<int>(64);
  for (size_t count : {n * M * dp, n * M * dp, R * d, R * d, R * dp, R * M, R * M, n * nt * M * dp,
                       R * tile, R * dp, (M + 127) / 128 * 128 * d, M})
    cv.take<float>(count);
  return cv.bytes();
}

// With less workspace than workspace_bytes asks for, as many chains at a time as fit, and
// then as many frames per sequence.  (A frame per sequence instead: one chain of 8192 rows,
// d = 128, M = 256, bf16, C = 16 in slim_fwd_noalloc's scratch 15.0 ms against 0.37 ms.)
slim_status fwd(const Problem& p, const void* q_ptr, const void* k, const void* v,
                const float* omega, void* out, const StateOut& st, const StateInit& init,
                void* workspace, size_t bytes, cudaStream_t s) {
  int batch = p.chains();
  long long limit = kNoLimit;
  if (out && p.L <= kShortMax && p.C >= p.L) {
    // a few rows on a running state: one launch (a frame of the general kernels
    // holds 64 rows; measured 70 us for one row of 64 chains there, 13 us here)
    const Seq q = sequence(p, 1);
    const TileArgs A = seq_args(p, q, SeqWs{}, q_ptr, k, v, omega);
    SLIM_TRY(launch_short(p, A.ks_n, A.ks_a, q_ptr, k, v, omega, out, st, init,
                          static_cast<int*>(workspace), s));
    return SLIM_OK;
  }
  if (bytes < fwd_bytes(p, batch, kNoLimit)) {
    const size_t one = fwd_bytes(p, 1, 0), two = fwd_bytes(p, 2, 0);
    if (bytes < one) return SLIM_ERR_WORKSPACE;
    // every chain after the first adds the same, give or take the arrays' alignment
    while (batch > 1 && fwd_bytes(p, batch, 0) > bytes) {
      const size_t fit = 1 + (bytes - one) / (two - one);
      batch = fit < (size_t)batch ? (int)fit : batch - 1;
    }
    long long most = sequence(p, batch).frames;
    for (limit = 0; limit < most;) {
      const long long mid = (limit + most + 1) / 2;
      if (fwd_bytes(p, batch, mid) <= bytes)
        limit = mid;
      else
        most = mid - 1;
    }
  }
  for (int c0 = 0; c0 < p.chains(); c0 += batch) {
    const int n = p.chains() - c0 < batch ? p.chains() - c0 : batch;
    const slim_status r = fwd_chains(p, c0, sequence(p, n, limit), q_ptr, k, v, omega, out, st, init,
                                     workspace, s);
    if (r != SLIM_OK) return r;
  }
  return SLIM_OK;
}

slim_status bwd(const Problem& p, const void* q, const void* k, const void* v,
                const float* omega, const void* out, const void* dout, const StateIn& st,
                const GradIO& gio, void* dq, void* dk, void* dv, float* domega, void* workspace,
                cudaStream_t s) {
  return bwd_impl(p, q, k, v, omega, out, dout, st, gio, dq, dk, dv, domega, workspace, s);
}

slim_status fwd_bidir(const Problem& p, const void* q, const void* k, const void* v,
                      const float* omega, void* out, const StateOut& st, void* workspace,
                      cudaStream_t s) {
  return fwd_bidir_impl(p, q, k, v, omega, out, st, workspace, s);
}

slim_status bwd_bidir(const Problem& p, const void* q, const void* k, const void* v,
                      const float* omega, const void* out, const void* dout, const StateIn& st,
                      void* dq, void* dk, void* dv, float* domega, void* workspace,
                      cudaStream_t s) {
  return bwd_bidir_impl(p, q, k, v, omega, out, dout, st, dq, dk, dv, domega, workspace, s);
}

}  // namespace simt
}  // namespace slim
