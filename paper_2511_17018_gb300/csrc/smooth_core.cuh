// Two-filter smoother of a recorded fit (Fraser & Potter): for every cluster,
// the residual against the estimate from all the other clusters.  Included
// after fit_core.cuh and adjoint_core.cuh by each kernel module, so that the
// recomputed filter steps are the module's own arithmetic.
//
// Per cluster c of a fitted track: the outward prediction at c (seed and
// clusters 0..c-1) and the inward prediction at c (the inward pass's prior and
// clusters last..c+1) are independent estimates of the state at c.  Their
// combination x_u has
//   H x_u     = H x_out + H C_out S^-1 (x_in - x_out),
//   H C_u H^T = H C_out S^-1 C_in H^T,        S = C_out + C_in,
// (C_u = C_out S^-1 C_in, without a subtraction), evaluated in square-root
// form (smooth_combine).  Outputs: the residual m_c - H x_u,
// R = V + H C_u H^T and chi2 = r^T R^-1 r (2 degrees of freedom).
//
// Both predictions follow from states that the recorded fit left on its tape, so
// the clusters of a track are smoothed independently of each other
// (smooth_tape_kernel).  Items without a place on the tape, and the last clusters
// of some of the others, go through smooth_kernel.  From the checkpoints:
//
// Work mapping of smooth_kernel: the outward filter runs forward from the seed, cluster by
// cluster.  The inward predictions are needed in the same order, which is the
// reverse of the inward pass; they come from the inward checkpoints segment by
// segment (last segment first): a segment is recomputed into the warp's
// segment store and consumed in reverse, one state copied ahead into shared
// memory, as in the adjoint.
#pragma once

namespace tpcfit {
namespace TPCFIT_NS {

// Residual, its covariance and chi2 of one cluster from the outward (1) and
// inward (2) predictions (p, square-root factor L, C = L L^T), both in
// residual coordinates of that cluster.
//
// Square-root form: with A1 = L1^T, A2 = L2^T and the QR factorisation
// [A1; A2] = Q R (Householder, Q 10x5 with orthonormal columns, Q = [Q1; Q2]),
// S = C1 + C2 = R^T R and C1 S^-1 C2 = A1^T Q1 Q2^T A2, so that
//   H x_u - H x1 = W1 u,  H C_u H^T = W1 W2^T,  u = R^-T (x2 - x1),
//   W1 = [H L1, 0] Q,  W2 = [0, H L2] Q,
// computed by applying the reflectors to the two 2x10 row blocks.  Forming S
// (or C H^T) in FP32 instead squares the condition number of the factors and
// loses the residual next to a diffuse end of the track (the second and the
// second-last cluster).
__device__ __forceinline__ void smooth_combine(const GeoRef& G, const float p1[5], const float L1[5][5], const float p2[5],
                                               const float L2[5][5], float r[2], float R[3], float& chi2) {
  float M[10][5];   // [A1; A2]
  float E[4][10];   // rows 0-1: [H L1, 0]; rows 2-3: [0, H L2]
#pragma unroll
  for (int q = 0; q < 5; ++q)
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      M[q][i] = L1[i][q];
      M[5 + q][i] = L2[i][q];
    }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      E[h][q] = L1[h][q];
      E[h][5 + q] = 0.0f;
      E[2 + h][q] = 0.0f;
      E[2 + h][5 + q] = L2[h][q];
    }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    // reflector of column k, rows k..9: v = x - alpha e_k, alpha = -sign(x_k) |x|
    float nrm2 = M[k][k] * M[k][k];
#pragma unroll
    for (int q = k + 1; q < 10; ++q) nrm2 = nrm2 + M[q][k] * M[q][k];
    float nrm, inrm;
    sqrt_and_inv(nrm2, nrm, inrm);
    const float alpha = M[k][k] > 0.0f ? -nrm : nrm;
    const float v0 = M[k][k] - alpha;
    // y <- y + (v^T y) / (alpha v0) v  (the reflection I - 2 v v^T / v^T v)
    const float g = 1.0f / (alpha * v0);
#pragma unroll
    for (int j = k + 1; j < 5; ++j) {
      float t = v0 * M[k][j];
#pragma unroll
      for (int q = k + 1; q < 10; ++q) t = t + M[q][k] * M[q][j];
      t = t * g;
      M[k][j] = M[k][j] + t * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) M[q][j] = M[q][j] + t * M[q][k];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float t = E[e][k] * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) t = t + E[e][q] * M[q][k];
      t = t * g;
      E[e][k] = E[e][k] + t * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) E[e][q] = E[e][q] + t * M[q][k];
    }
    M[k][k] = alpha;
  }
  // u = R^-T (p2 - p1), R = upper 5x5 of M
  float u[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    float e = p2[i] - p1[i];
#pragma unroll
    for (int q = 0; q < i; ++q) e = e - M[q][i] * u[q];
    u[i] = e / M[i][i];
  }
  float c0 = E[0][0] * u[0], c1 = E[1][0] * u[0];
  float h00 = E[0][0] * E[2][0], h01 = E[0][0] * E[3][0], h10 = E[1][0] * E[2][0], h11 = E[1][0] * E[3][0];
#pragma unroll
  for (int q = 1; q < 5; ++q) {
    c0 = c0 + E[0][q] * u[q];
    c1 = c1 + E[1][q] * u[q];
    h00 = h00 + E[0][q] * E[2][q];
    h01 = h01 + E[0][q] * E[3][q];
    h10 = h10 + E[1][q] * E[2][q];
    h11 = h11 + E[1][q] * E[3][q];
  }
  // the state is relative to the measurement: r = m - H x_u = -(p1 + correction)
  r[0] = -(p1[0] + c0);
  r[1] = -(p1[1] + c1);
  const float v = G.v_meas;
  R[0] = v + h00;
  R[1] = 0.5f * (h01 + h10);
  R[2] = v + h11;
  const float det = R[0] * R[2] - R[1] * R[1];
  chi2 = (R[2] * r[0] * r[0] - 2.0f * R[1] * r[0] * r[1] + R[0] * r[1] * r[1]) / det;
}

// Smoothed state from all clusters at one cluster: the same square-root
// combination, of the outward pass's filtered state there (p1, L1) with the
// inward prediction (p2, L2), but with the five rows of [L1, 0] and of
// [0, L2] carried through the reflectors: W1 = [L1, 0] Q, W2 = [0, L2] Q,
//   x_s = p1 + W1 u,  C_s = W1 W2^T (symmetrised),  u = R^-T (p2 - p1).
__device__ __forceinline__ void smooth_state(const float p1[5], const float L1[5][5], const float p2[5],
                                             const float L2[5][5], float xs[5], float Cs[15]) {
  float M[10][5];   // [A1; A2]
  float E[10][10];  // rows 0-4: [L1, 0]; rows 5-9: [0, L2]
#pragma unroll
  for (int q = 0; q < 5; ++q)
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      M[q][i] = L1[i][q];
      M[5 + q][i] = L2[i][q];
    }
#pragma unroll
  for (int h = 0; h < 5; ++h)
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      E[h][q] = L1[h][q];
      E[h][5 + q] = 0.0f;
      E[5 + h][q] = 0.0f;
      E[5 + h][5 + q] = L2[h][q];
    }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    float nrm2 = M[k][k] * M[k][k];
#pragma unroll
    for (int q = k + 1; q < 10; ++q) nrm2 = nrm2 + M[q][k] * M[q][k];
    float nrm, inrm;
    sqrt_and_inv(nrm2, nrm, inrm);
    const float alpha = M[k][k] > 0.0f ? -nrm : nrm;
    const float v0 = M[k][k] - alpha;
    const float g = 1.0f / (alpha * v0);
#pragma unroll
    for (int j = k + 1; j < 5; ++j) {
      float t = v0 * M[k][j];
#pragma unroll
      for (int q = k + 1; q < 10; ++q) t = t + M[q][k] * M[q][j];
      t = t * g;
      M[k][j] = M[k][j] + t * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) M[q][j] = M[q][j] + t * M[q][k];
    }
#pragma unroll
    for (int e = 0; e < 10; ++e) {
      float t = E[e][k] * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) t = t + E[e][q] * M[q][k];
      t = t * g;
      E[e][k] = E[e][k] + t * v0;
#pragma unroll
      for (int q = k + 1; q < 10; ++q) E[e][q] = E[e][q] + t * M[q][k];
    }
    M[k][k] = alpha;
  }
  float u[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    float e = p2[i] - p1[i];
#pragma unroll
    for (int q = 0; q < i; ++q) e = e - M[q][i] * u[q];
    u[i] = e / M[i][i];
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    float acc = E[i][0] * u[0];
#pragma unroll
    for (int q = 1; q < 5; ++q) acc = acc + E[i][q] * u[q];
    xs[i] = p1[i] + acc;
  }
  int e = 0;
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      float a12 = E[i][0] * E[5 + j][0];
      float a21 = E[j][0] * E[5 + i][0];
#pragma unroll
      for (int q = 1; q < 5; ++q) {
        a12 = a12 + E[i][q] * E[5 + j][q];
        a21 = a21 + E[j][q] * E[5 + i][q];
      }
      Cs[e++] = 0.5f * (a12 + a21);
    }
}

// The clusters of a track without an estimate.  A track that reaches beyond the
// arrays has none; those of its clusters that lie inside are written unless the
// offsets after it come back (they may be other tracks' then).
__device__ __forceinline__ void write_nan_clusters(const SmoothArgs& a, int32_t trk, const RecordedTrack& track) {
  int h0 = track.begin + track.steps, h1 = track.end;
  if (h1 == 0 && a.off[trk + 1] > a.n_hits && a.off[trk] >= 0 &&
      (trk + 1 == a.n_tracks || a.off[trk + 2] >= a.off[trk + 1])) {
    h0 = a.off[trk];
    h1 = (int)a.n_hits;
  }
  const float qnan = __int_as_float(0x7fc00000);
  for (int h = h0; h < h1; ++h) {
    if (a.resid) {
      reinterpret_cast<float2*>(a.resid)[h] = make_float2(qnan, qnan);
      a.rcov[(int64_t)h * 3] = qnan;
      a.rcov[(int64_t)h * 3 + 1] = qnan;
      a.rcov[(int64_t)h * 3 + 2] = qnan;
      a.chi2[h] = qnan;
    }
    if (a.state) {
      for (int q = 0; q < 5; ++q) a.state[(int64_t)h * 5 + q] = qnan;
      for (int q = 0; q < 15; ++q) a.state_cov[(int64_t)h * 15 + q] = qnan;
    }
  }
}

// Shared memory of a smoother block: the tables, the alignment table and,
// per warp, a double buffer for the inward states and a checkpoint buffer.
template <int WARPS>
constexpr size_t smooth_smem_bytes() {
  return sizeof(BwdSmem) + WARPS * sizeof(BwdWarpBufs);
}

// STATES: the smoothed state and its covariance at every cluster as well
// (a.state, a.state_cov); without it the kernel carries none of that code.
//
// After a fit that left a U-D tape it does two things.  Items without a place on
// the tape go through it whole.  Of the others it smooths the last kSmoothEnds
// clusters, the ends, where the outputs depend on rounding: at steep angles
// (|sin phi| towards 1) a filter amplifies it, and the inward prior is diffuse
// there.  They keep the square-root sequence, along the outward filter from the
// seed, and smooth_tape_kernel does the rest.  That keeps the values that users of the
// checkpoint form have; it is not nearer to 64 bits (30,000 tracks of natural length,
// steep ends, error in norm with it and with the tape's combination instead: residuals
// 3.9e-4 and 3.9e-4, their covariance 2.4e-5 and 2.0e-6, states' covariance 4.4e-4 and
// 3.4e-5).  The states' covariance depends on the sequence
// at 3e-5 in norm, so every track's end is smoothed here (30,000 tracks: 169 us for
// the ends, 185 for the rest).  The residuals do in single elements only (1e-3 of
// the largest, and 3e-4 below |sin phi| = 0.9), so only the steep tracks' ends are,
// gathered by each warp from its share of the tracks.
constexpr int kSmoothEnds = kCkptEvery;
constexpr float kSmoothSteep = 0.9f;

// |sin phi| next to the end of a track of `steps` steps above kSmoothSteep; its
// outward states from row0 on.  Read before the last even step, which a tape of every
// state and one of every second state both hold, so that a track's sequence does not
// depend on its batch.  (The inward pass's first state, the very end, would do too, but
// finds a few steep tracks in batches without others, and the first one in a batch
// brings the chain of the ends: residuals of 5,000 tracks 290 -> 380 us.)
__device__ __forceinline__ bool steep_end(const float4* row0, int steps, int every, int pitch) {
  return fabsf(__ldg(row0 + kUDRows * (((steps - 1) & ~1) / every) * pitch).z) > kSmoothSteep;
}

// An outward or inward pass's first state from the U-D tape, as a checkpoint.
__device__ __forceinline__ void tape_first_state(const float4* src, int pitch, StepState& S) {
  float v[32];
#pragma unroll
  for (int e = 20; e < 32; ++e) v[e] = 0.0f;
#pragma unroll
  for (int j = 0; j < kUDRows; ++j) {
    const float4 f = __ldg(src + j * pitch);
    v[4 * j] = f.x;
    v[4 * j + 1] = f.y;
    v[4 * j + 2] = f.z;
    v[4 * j + 3] = f.w;
  }
  unpack_state(v, S);
}

constexpr int kMaxShare = kStateF4 * kWarp * 4;  // tracks that a warp's list holds

template <int WARPS, bool MAT, bool STATES>
__global__ void __launch_bounds__(WARPS * 32, 1) smooth_kernel(const __grid_constant__ SmoothArgs a) {
  const GeoRef& G = a.geo;
  const bool ends_too = a.tape_item && a.ck_form == 1;
  const bool missing = !a.tape_item || a.work[kWorkMissing] > 0;
  if (!ends_too && !missing) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem& B = *reinterpret_cast<BwdSmem*>(smem_raw);
  load_block_tables(G, B.T, B.align, a.align);
  const SmemTables& T = B.T;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  BwdWarpBufs& W = reinterpret_cast<BwdWarpBufs*>(smem_raw + sizeof(BwdSmem))[warp];
  float4* const gs = a.seg + ((int64_t)blockIdx.x * WARPS + warp) * (kCkptEvery * kStateF4 * kWarp) + lane;
  const int64_t n_items = ((int64_t)a.n_tracks + a.item_tracks - 1) / a.item_tracks;
  // residuals: after the items (none if all are on the tape) the tracks once more,
  // `share` of them at a time, for the steep ones' ends
  const bool gather = !STATES && ends_too;
  const int n_warps = gridDim.x * (blockDim.x >> 5);
  const int share = min(kMaxShare, ((a.n_tracks + n_warps - 1) / n_warps + kWarp - 1) / kWarp * kWarp);
  const int64_t lists = gather ? ((int64_t)a.n_tracks + share - 1) / share : 0;
  const int64_t items = STATES || missing ? n_items : 0;
  int* const list = reinterpret_cast<int*>(&W.ck[0][0]);  // no checkpoint is read for the ends
  int listed = 0, taken = 0;
#pragma unroll 1
  for (bool first = true;;) {
    int64_t item = -1;
    if (taken >= listed) {
      const int64_t unit = next_item(a.work, items + lists, first);
      first = false;
      if (unit < 0) break;
      if (unit < items) {
        item = unit;
      } else {
        const int64_t slot0 = (unit - items) * share;
        listed = taken = 0;
        __syncwarp();
#pragma unroll 1
        for (int64_t k = slot0 + lane; k - lane < min(slot0 + share, (int64_t)a.n_tracks); k += kWarp) {
          bool steep = false;
          if (k < a.n_tracks) {
            const int32_t t = a.perm ? a.perm[k] : (int32_t)k;
            const int2 at = a.tape_item[k / a.item_tracks];
            const int n = recorded_track(a, t).steps;
            if (at.x >= 0 && n > 0)
              steep = steep_end(tape_row0(a.tape, at, a.item_tracks, (int)(k % a.item_tracks)) + at.y * a.item_tracks, n,
                                a.tape_every, a.item_tracks);
          }
          const unsigned m = __ballot_sync(0xffffffffu, steep);
          if (steep) list[listed + __popc(m & ((1u << lane) - 1))] = (int)k;
          listed += __popc(m);
        }
        __syncwarp();
        if (listed == 0) continue;
      }
    }
    const bool from_list = item < 0;
    const int64_t slot = from_list ? (taken + lane < listed ? list[taken + lane] : a.n_tracks) : item * a.item_tracks + lane;
    const bool have = (from_list || lane < a.item_tracks) && slot < a.n_tracks;
    if (from_list) taken += kWarp;
    const int2 place = a.tape_item && (have || !from_list) ? a.tape_item[from_list ? slot / a.item_tracks : item]
                                                           : make_int2(-1, 0);
    const bool ends = from_list || (STATES && ends_too && place.x >= 0);
    if (place.x >= 0 && !ends) continue;  // smooth_tape_kernel's
    const int32_t trk = have ? (a.perm ? a.perm[slot] : (int32_t)slot) : 0;
    const RecordedTrack track = have ? recorded_track(a, trk) : RecordedTrack();
    const int begin = track.begin, steps = track.steps;
    const int last = steps - 1;
    if (have && !ends) write_nan_clusters(a, trk, track);
    const int64_t slot0 = (begin >> kCkptShift) + trk;
    const float4* const row0 = ends && have ? tape_row0(a.tape, place, a.item_tracks, (int)(slot % a.item_tracks)) +
                                                  place.y * a.item_tracks
                                            : nullptr;
    // outward filter: from its first state (the seed, factor L0)
    StepState O;
    float omy = 0.0f, omz = 0.0f;  // measurement O's residuals refer to (none for the seed)
    // inward segments, last first: inward step j is cluster last - j
    const int nseg = (steps + kCkptEvery - 1) / kCkptEvery;
    const float* ckp = a.ck + ((int64_t)a.ck_slots + slot0) * kCkptFloats;
    const int h_last = begin + last;
    HitRaw ahead{};  // the cluster after the one taken next
    float m0 = 0.0f, m1 = 0.0f;
    int row = 0, sec = 0;
    if (steps > 0) {
      if (ends) {
        tape_first_state(row0, a.item_tracks, O);
      } else {
        fetch_ckpt(&W.ck[0][lane], a.ck + slot0 * kCkptFloats);
        cp_async_wait<0>();
        read_state(&W.ck[0][lane], O);
        fetch_ckpt(&W.ck[0][lane], ckp + (int64_t)(nseg - 1) * kCkptFloats);
      }
      if (a.ck_form == 1) sqrt_from_ud_ckpt(O);
      decode_hit(B.align, load_hit(a.y, a.z, a.rowsec, begin), m0, m1, row, sec);
      if (last > 0) ahead = load_hit(a.y, a.z, a.rowsec, begin + 1);
    }
    // the segments of all lanes together, so that lanes of different lengths stay
    // converged
#pragma unroll 1
    for (int s = __reduce_max_sync(0xffffffffu, nseg) - 1; s >= 0; --s) {
      __syncwarp();
      if (s >= nseg) continue;
      const int j0 = s * kCkptEvery;
      const int cnt = min(kCkptEvery, steps - j0);
      const bool combine = !ends || s == 0;
      if (combine) {
        StepState S;
        float my = 0.0f, mz = 0.0f;
        HitRaw nx = load_hit(a.y, a.z, a.rowsec, h_last - j0);
        if (j0 > 0) {
          int prow, psec;
          decode_hit(B.align, load_hit(a.y, a.z, a.rowsec, h_last - (j0 - 1)), my, mz, prow, psec);
        }
        if (ends) {
          tape_first_state(row0 + kUDRows * (int)tape_states(place.y, a.tape_every) * a.item_tracks, a.item_tracks, S);
        } else {
          cp_async_wait<0>();
          read_state(&W.ck[0][lane], S);
        }
        if (a.ck_form == 1) sqrt_from_ud_ckpt(S);
        // level 1: the inward segment, storing the state before each step
#pragma unroll 1
        for (int kk = 0; kk < cnt; ++kk) {
          const int j = j0 + kk;
          const HitRaw cur = nx;
          if (kk + 1 < cnt) nx = load_hit(a.y, a.z, a.rowsec, h_last - (j + 1));
          float n0, n1;
          int nrow, nsec;
          decode_hit(B.align, cur, n0, n1, nrow, nsec);
          store_state(gs + kk * (kStateF4 * kWarp), S);
          step_fwd<MAT, 2>(G, T, S, my, mz, j == 0, false, nrow, side_sector(nsec), n0, n1);
        }
        __threadfence_block();  // the states just stored are read back by this thread's copies below
        if (s > 0) fetch_ckpt(&W.ck[0][lane], ckp + (int64_t)(s - 1) * kCkptFloats);
        fetch_state(&W.st[(cnt - 1) & 1][0][lane], gs + (cnt - 1) * (kStateF4 * kWarp));
      }
      // consume in reverse: cluster c = last - j ascending
#pragma unroll 1
      for (int kk = cnt - 1; kk >= 0; --kk) {
        const int j = j0 + kk;
        const int c = last - j;
        const int h = begin + c;
        const int sec18 = side_sector(sec);
        const float X = T.row_x[row];
        // the cluster after this one
        float mpy = 0.0f, mpz = 0.0f;
        int prow = 0, psec = 0;
        if (j > 0) {
          decode_hit(B.align, ahead, mpy, mpz, prow, psec);
          if (j > 1) ahead = load_hit(a.y, a.z, a.rowsec, h + 2);
        }
        // inward prediction at c
        StepState SI;
        float pi[5];
        if (combine) {
          if (kk > 0) {
            fetch_state(&W.st[(kk - 1) & 1][0][lane], gs + (kk - 1) * (kStateF4 * kWarp));
            cp_async_wait<1>();
          } else {
            cp_async_wait<0>();
          }
          read_state(&W.st[kk & 1][0][lane], SI);
          if (j == 0) {  // the inward pass starts on this cluster
#pragma unroll
            for (int q = 0; q < 5; ++q) pi[q] = SI.p[q];
          } else {
            Jac J;
            PredTape tp;
            if (MAT) {  // the layer of row c + 1, undone against the flight
              MatNoise N;
              material_step(G, SI.p, -1, N);
              material_factor(SI.L, N);
            }
            predict_residual<2>(G, T, SI.p, SI.x, SI.sec, mpy, mpz, sec18, X, m0, m1, pi, J, tp);
            transport(SI.L, J);
          }
        }
        // outward prediction at c
        float po[5];
        if (c == 0) {  // the seed, made relative to the first cluster
#pragma unroll
          for (int q = 0; q < 5; ++q) po[q] = O.p[q];
          po[0] = O.p[0] - m0;
          po[1] = O.p[1] - m1;
        } else {
          Jac J;
          PredTape tp;
          predict_residual<2>(G, T, O.p, O.x, O.sec, omy, omz, sec18, X, m0, m1, po, J, tp);
          MatNoise N;
          if (MAT) material_step(G, po, 1, N);  // the layer of row c
          transport(O.L, J);
          if (MAT) material_factor(O.L, N);
        }
        if (a.resid && combine) {
          float r[2], R[3], c2;
          smooth_combine(G, po, O.L, pi, SI.L, r, R, c2);
          reinterpret_cast<float2*>(a.resid)[h] = make_float2(r[0], r[1]);
          a.rcov[(int64_t)h * 3] = R[0];
          a.rcov[(int64_t)h * 3 + 1] = R[1];
          a.rcov[(int64_t)h * 3 + 2] = R[2];
          a.chi2[h] = c2;
        }
        // the outward filter takes cluster c
#pragma unroll
        for (int q = 0; q < 5; ++q) O.p[q] = po[q];
        O.x = X;
        O.sec = sec18;
        omy = m0;
        omz = m1;
        float chi_unused = 0.0f;
        scalar_update<0>(G, O.p, O.L, chi_unused, 0.0f);
        scalar_update<1>(G, O.p, O.L, chi_unused, 0.0f);
        if (STATES && combine) {  // the outward filtered state at c with the inward prediction
          float xs[5], Cs[15];
          smooth_state(O.p, O.L, pi, SI.L, xs, Cs);
          xs[0] = xs[0] + m0;  // residual coordinates back to positions
          xs[1] = xs[1] + m1;
#pragma unroll
          for (int q = 0; q < 5; ++q) a.state[(int64_t)h * 5 + q] = xs[q];
#pragma unroll
          for (int q = 0; q < 15; ++q) a.state_cov[(int64_t)h * 15 + q] = Cs[q];
        }
        m0 = mpy;
        m1 = mpz;
        row = prow;
        sec = psec;
      }
    }
  }
}

// ---------------------------------------------------------------- from the tape
// The two estimates of a state in U-D form combined: the second one, (p2, U2, D2),
// is five measurements V p2 of the state with V = U2^-1 (unit upper triangular)
// and independent errors of variance D2, taken by the first one, (p, U, D), in
// turn with Bierman's scalar update (bierman_update with row k of V in place of a
// unit vector).  About 330 operations; no sum of the covariances is formed, and
// next to a diffuse end of the track, where one side is a cluster or two and the
// prior, the variances stay in D, apart from each other: the covariances are
// closer to 64 bits than those of the orthogonal reduction.
template <int K>
__device__ __forceinline__ void take_component(float p[5], float u[10], float d[5], const float p2[5], const float V[10],
                                               float variance) {
  float gain[5];
  float ap = variance, iap = 0.0f;
  float r = p2[K] - p[K];
#pragma unroll
  for (int i = K + 1; i < 5; ++i) r = r + V[ui(K, i)] * (p2[i] - p[i]);
#pragma unroll
  for (int j = K; j < 5; ++j) {
    float f = 1.0f;  // column j of U against row K of V
    if (j > K) {
      f = V[ui(K, j)] + u[ui(K, j)];
#pragma unroll
      for (int i = K + 1; i < j; ++i) f = f + V[ui(K, i)] * u[ui(i, j)];
    }
    const float g = j == K ? d[j] : d[j] * f;
    const float a = j == K ? ap + g : ap + f * g;
    const float ia = ud_rcp(a);
    if (j > K) {
      const float lam = -(f * iap);
#pragma unroll
      for (int i = 0; i < j; ++i) {
        const float uo = u[ui(i, j)];
        u[ui(i, j)] = uo + lam * gain[i];
        gain[i] = gain[i] + g * uo;
      }
    } else {
#pragma unroll
      for (int i = 0; i < j; ++i) gain[i] = g * u[ui(i, j)];
    }
    d[j] = d[j] * (ap * ia);
    gain[j] = g;
    ap = a;
    iap = ia;
  }
  const float q = r * iap;
#pragma unroll
  for (int i = 0; i < 5; ++i) p[i] = p[i] + gain[i] * q;
}

__device__ __forceinline__ void combine_ud(float p[5], float u[10], float d[5], const float p2[5], const float u2[10],
                                           const float d2[5]) {
  float V[10];  // U2^-1
#pragma unroll
  for (int i = 3; i >= 0; --i)
#pragma unroll
    for (int j = i + 1; j < 5; ++j) {
      float acc = u2[ui(i, j)];
#pragma unroll
      for (int k = i + 1; k < j; ++k) acc = acc + u2[ui(i, k)] * V[ui(k, j)];
      V[ui(i, j)] = -acc;
    }
  take_component<4>(p, u, d, p2, V, d2[4]);
  take_component<3>(p, u, d, p2, V, d2[3]);
  take_component<2>(p, u, d, p2, V, d2[2]);
  take_component<1>(p, u, d, p2, V, d2[1]);
  take_component<0>(p, u, d, p2, V, d2[0]);
}

// Every cluster on its own: the state before the outward step to it and the one
// before the inward step to it come from the tape (with every second state there,
// an odd one is recomputed from the one before it), are predicted to the cluster
// and combined.  A unit of work is a few consecutive clusters of an item's
// tracks, one track per lane.  No lane waits for another cluster, where
// smooth_kernel recomputes both filters along each track.
//
// Bound by its arithmetic and by instruction fetch: the two predictions of a
// cluster are two turns of one loop, since two copies of the prediction and the
// recomputed step miss the instruction cache (1.4 warps waiting for instructions
// per issue, 0.3 as a loop).  Measured: leave-one-out residuals of 100,000 tracks
// 823 -> 593 us (465 without the steep tracks' ends, whose one chain of steps a warp
// is serial), smoothed states of 30,000 tracks, the ends included, 675 -> 363 us.
// The unit's clusters are copied into shared memory once and each state one turn
// ahead; the outputs leave through shared memory too, a track's run of clusters at
// a time instead of single words.
template <bool STATES>
struct SmoothOut {
  static constexpr int kSteps = STATES ? 4 : 8;         // clusters of a track in a unit
  static constexpr int kUnits = kMaxRows / kSteps;      // units of an item (longer tracks: again)
  static constexpr int kFloats = STATES ? 20 : 6;       // per cluster: (state 5, cov 15) or (resid 2, rcov 3, chi2)
  static constexpr int kPitch = kFloats * kSteps + 1;   // odd: lanes fall into different banks
  float v[kWarp][kPitch];
  int first[kWarp];  // the unit's first cluster of each track, and how many
  int count[kWarp];
};

// Per warp: the outputs and, in U-D form, the unit's clusters with two more on
// either side and two states (one in use, one on its way).
template <bool STATES, int FORM>
struct SmoothWarp {
  SmoothOut<STATES> out;
};
template <bool STATES>
struct SmoothWarp<STATES, 1> {
  static constexpr int kClusters = SmoothOut<STATES>::kSteps + 4;
  alignas(16) float4 cluster[kClusters][kWarp];
  float4 state[2][kUDRows][kWarp];
  SmoothOut<STATES> out;
};

// One output of the unit: PER floats to a cluster, at AT in the cluster's record.
// 32 consecutive lanes write consecutive words of a track's run.
template <class Out, int PER, int AT>
__device__ __forceinline__ void write_unit(float* dst, const Out& O, int tracks, int lane) {
  constexpr int kRun = Out::kSteps * PER;
  int t = lane / kRun, r = lane % kRun;  // track and word of its run
#pragma unroll 4
  for (int e = lane; e < tracks * kRun; e += kWarp) {
    const int c = r / PER;
    if (c < O.count[t]) dst[(int64_t)O.first[t] * PER + r] = O.v[t][c * Out::kFloats + AT + (r - c * PER)];
    t += kWarp / kRun;
    r += kWarp % kRun;
    if (r >= kRun) {
      r -= kRun;
      ++t;
    }
  }
}

template <int WARPS, int FORM, bool MAT, bool STATES>
__global__ void __launch_bounds__(WARPS * 32, 1) smooth_tape_kernel(const __grid_constant__ SmoothArgs a) {
  const GeoRef& G = a.geo;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the square-root tape holds no clusters: they need the alignment table
  constexpr size_t kBlock = FORM == 1 ? sizeof(SmemTables) : sizeof(BwdSmem);
  BwdSmem& B = *reinterpret_cast<BwdSmem*>(smem_raw);
  load_block_tables(G, B.T, B.align, FORM == 1 ? nullptr : a.align);
  const SmemTables& T = B.T;
  const int lane = threadIdx.x & 31;
  using Out = SmoothOut<STATES>;
  using Warp = SmoothWarp<STATES, FORM>;
  Warp& W = reinterpret_cast<Warp*>(smem_raw + kBlock)[threadIdx.x >> 5];
  Out& O = W.out;
  const int pitch = a.item_tracks;
  const int64_t n_items = ((int64_t)a.n_tracks + pitch - 1) / pitch;
#pragma unroll 1
  for (bool first = true;; first = false) {
    const int64_t unit = next_item(a.work, n_items * Out::kUnits, first);
    if (unit < 0) break;
    const int64_t item = unit / Out::kUnits;
    const int part = (int)(unit % Out::kUnits);
    const int2 place = a.tape_item[item];
    if (place.x < 0) continue;  // smooth_kernel's
    const int64_t slot = item * pitch + lane;
    const bool have = lane < pitch && slot < a.n_tracks;
    const int32_t trk = have ? (a.perm ? a.perm[slot] : (int32_t)slot) : 0;
    const RecordedTrack track = have ? recorded_track(a, trk) : RecordedTrack();
    const int begin = track.begin, steps = track.steps;
    if (have && part == 0) write_nan_clusters(a, trk, track);
    const float4* const row0 = tape_row0(a.tape, place, pitch, lane);
    const int every = FORM == 1 ? a.tape_every : 1;
    // the last clusters are smooth_kernel's (U-D form: all tracks' states, the steep
    // ones' residuals)
    int upto = steps;
    if (FORM == 1 && steps > 0 && (STATES || steep_end(row0 + place.y * pitch, steps, every, pitch)))
      upto = max(0, steps - kSmoothEnds);
    const int most = __reduce_max_sync(0xffffffffu, upto);
    const int states = (int)tape_states(place.y, every);

    // a track's cluster: measured (y, z), the row's x, sector mod 18
    struct At {
      float m0, m1, X;
      int sec;
    };
#pragma unroll 1
    for (int c0 = part * Out::kSteps; c0 < most; c0 += Out::kUnits * Out::kSteps) {
      if constexpr (FORM == 1) {
#pragma unroll 1
        for (int e = 0; e < Warp::kClusters; ++e) {
          const int c = c0 - 2 + e;
          if (c >= 0 && c < steps) cp_async16(&W.cluster[e][lane], row0 + c * pitch);
        }
        auto cluster = [&](int c) {
          const float4 v = W.cluster[c - c0 + 2][lane];
          At k;
          k.m0 = v.x;
          k.m1 = v.y;
          k.X = v.z;
          k.sec = side_sector(__float_as_int(v.w) & 63);
          return k;
        };
        // turn q: cluster c0 + q / 2, the inward prediction first
        auto fetch = [&](int q) {
          const int c = c0 + (q >> 1), pass = 1 - (q & 1);
          if (q < 2 * Out::kSteps && c < upto) {
            const int i = pass == 0 ? c : steps - 1 - c;
            copy_rows<kUDRows>(&W.state[q & 1][0][lane],
                               row0 + (place.y + kUDRows * (pass * states + (every == 2 ? i >> 1 : i))) * pitch, pitch);
          }
          cp_async_commit();
        };
        fetch(0);
        float p2[5], u2[10], d2[5];
#pragma unroll 1
        for (int q = 0; q < 2 * Out::kSteps; ++q) {
          fetch(q + 1);
          cp_async_wait<1>();
          const int c = c0 + (q >> 1), pass = 1 - (q & 1);
          if (c >= upto) continue;
          const At at = cluster(c);
          const int dir = pass == 0 ? 1 : -1;  // from one step's cluster to the next
          const int i = pass == 0 ? c : steps - 1 - c;
          UDState S;
          read_state_ud<false>(&W.state[q & 1][0][lane], S);
          At prev = at;  // the state's own cluster
          if (i > 0) prev = cluster(c - dir);
          if (every == 2 && (i & 1)) {  // from the state before: its step, to cluster prev
            At pp = prev;
            if (i > 1) pp = cluster(c - 2 * dir);
            S.x = pp.X;
            S.sec = pp.sec;
            float my = pp.m0, mz = pp.m1;
            step_fwd_ud<2>(G, T, S, my, mz, i == 1, pass == 0, prev.X, prev.sec, prev.m0, prev.m1);
          }
          S.x = prev.X;
          S.sec = prev.sec;
          float pn[5];
          if (i == 0) {  // the pass starts on this cluster (outward: the seed, absolute)
#pragma unroll
            for (int e = 0; e < 5; ++e) pn[e] = S.p[e];
            if (pass == 0) {
              pn[0] = S.p[0] - at.m0;
              pn[1] = S.p[1] - at.m1;
            }
          } else {
            Jac J;
            PredTape tp;
            predict_residual<2>(G, T, S.p, S.x, S.sec, prev.m0, prev.m1, at.sec, at.X, at.m0, at.m1, pn, J, tp);
            if (J.rot)
              rotate_ud(S.u, S.d, J);
            else
              transport_ud(S.u, J);
          }
          if (pass == 1) {
#pragma unroll
            for (int e = 0; e < 5; ++e) p2[e] = pn[e];
#pragma unroll
            for (int e = 0; e < 10; ++e) u2[e] = S.u[e];
#pragma unroll
            for (int e = 0; e < 5; ++e) d2[e] = S.d[e];
            continue;
          }
          if (STATES) {  // the outward filtered state: with cluster c
            float chi_unused = 0.0f;
            bierman_update<0>(pn, S.u, S.d, chi_unused, G.v_meas);
            bierman_update<1>(pn, S.u, S.d, chi_unused, G.v_meas);
          }
          combine_ud(pn, S.u, S.d, p2, u2, d2);
          float* const o = &O.v[lane][(q >> 1) * Out::kFloats];
          if (STATES) {
            o[0] = pn[0] + at.m0;  // residual coordinates back to positions
            o[1] = pn[1] + at.m1;
#pragma unroll
            for (int e = 2; e < 5; ++e) o[e] = pn[e];
            int n = 5;
#pragma unroll
            for (int r = 0; r < 5; ++r)
#pragma unroll
              for (int j = 0; j <= r; ++j) {
                float acc = (j == r ? 1.0f : S.u[ui(j, r)]) * S.d[r];
#pragma unroll
                for (int k = r + 1; k < 5; ++k) acc = acc + (S.u[ui(r, k)] * S.d[k]) * S.u[ui(j, k)];
                o[n++] = acc;
              }
          } else {
            // the state is relative to the measurement: r = m - H x_u = -(y, z)
            const float r0 = -pn[0], r1 = -pn[1];
            float R0 = S.d[0], R1 = S.u[ui(0, 1)] * S.d[1], R2 = S.d[1];
#pragma unroll
            for (int k = 1; k < 5; ++k) R0 = R0 + (S.u[ui(0, k)] * S.d[k]) * S.u[ui(0, k)];
#pragma unroll
            for (int k = 2; k < 5; ++k) {
              R1 = R1 + (S.u[ui(1, k)] * S.d[k]) * S.u[ui(0, k)];
              R2 = R2 + (S.u[ui(1, k)] * S.d[k]) * S.u[ui(1, k)];
            }
            R0 = R0 + G.v_meas;
            R2 = R2 + G.v_meas;
            const float det = R0 * R2 - R1 * R1;
            o[0] = r0;
            o[1] = r1;
            o[2] = R0;
            o[3] = R1;
            o[4] = R2;
            o[5] = (R2 * r0 * r0 - 2.0f * R1 * r0 * r1 + R0 * r1 * r1) / det;
          }
        }
        cp_async_wait<0>();
      } else {
        auto cluster = [&](int c) {
          At k;
          int row, sec;
          decode_hit(B.align, load_hit(a.y, a.z, a.rowsec, begin + c), k.m0, k.m1, row, sec);
          k.X = T.row_x[row];
          k.sec = side_sector(sec);
          return k;
        };
#pragma unroll 1
        for (int k = 0; k < Out::kSteps; ++k) {
          const int c = c0 + k;
          if (c >= upto) continue;
          const At at = cluster(c);
          float* const o = &O.v[lane][k * Out::kFloats];
          float pp[2][5];
          StepState S[2];
#pragma unroll
          for (int pass = 1; pass >= 0; --pass) {
            const int i = pass == 0 ? c : steps - 1 - c;
            const float4* src = row0 + kSqrtRows * (pass * place.y + i) * pitch;
            {
              float v[32];
#pragma unroll
              for (int j = 0; j < kSqrtRows; ++j) {
                const float4 f = __ldg(src + j * pitch);
                v[4 * j] = f.x;
                v[4 * j + 1] = f.y;
                v[4 * j + 2] = f.z;
                v[4 * j + 3] = f.w;
              }
              unpack_state(v, S[pass]);
            }
            if (i == 0) {
#pragma unroll
              for (int q = 0; q < 5; ++q) pp[pass][q] = S[pass].p[q];
              if (pass == 0) {
                pp[0][0] = S[0].p[0] - at.m0;
                pp[0][1] = S[0].p[1] - at.m1;
              }
            } else {
              const At prev = cluster(pass == 0 ? c - 1 : c + 1);
              Jac J;
              PredTape tp;
              MatNoise N;
              if (MAT && pass == 1) {  // the layer of row c + 1, undone against the flight
                material_step(G, S[1].p, -1, N);
                material_factor(S[1].L, N);
              }
              predict_residual<2>(G, T, S[pass].p, S[pass].x, S[pass].sec, prev.m0, prev.m1, at.sec, at.X, at.m0,
                                  at.m1, pp[pass], J, tp);
              if (MAT && pass == 0) material_step(G, pp[0], 1, N);  // the layer of row c
              transport(S[pass].L, J);
              if (MAT && pass == 0) material_factor(S[0].L, N);
            }
          }
          if (STATES) {
            float chi_unused = 0.0f;
            scalar_update<0>(G, pp[0], S[0].L, chi_unused, 0.0f);
            scalar_update<1>(G, pp[0], S[0].L, chi_unused, 0.0f);
            float xs[5], Cs[15];
            smooth_state(pp[0], S[0].L, pp[1], S[1].L, xs, Cs);
            o[0] = xs[0] + at.m0;
            o[1] = xs[1] + at.m1;
#pragma unroll
            for (int q = 2; q < 5; ++q) o[q] = xs[q];
#pragma unroll
            for (int q = 0; q < 15; ++q) o[5 + q] = Cs[q];
          } else {
            float r[2], R[3], c2;
            smooth_combine(G, pp[0], S[0].L, pp[1], S[1].L, r, R, c2);
            o[0] = r[0];
            o[1] = r[1];
#pragma unroll
            for (int q = 0; q < 3; ++q) o[2 + q] = R[q];
            o[5] = c2;
          }
        }
      }
      O.first[lane] = begin + c0;
      O.count[lane] = max(0, min(Out::kSteps, upto - c0));
      __syncwarp();
      if (STATES) {
        write_unit<Out, 5, 0>(a.state, O, pitch, lane);
        write_unit<Out, 15, 5>(a.state_cov, O, pitch, lane);
      } else {
        write_unit<Out, 2, 0>(a.resid, O, pitch, lane);
        write_unit<Out, 3, 2>(a.rcov, O, pitch, lane);
        write_unit<Out, 1, 5>(a.chi2, O, pitch, lane);
      }
      __syncwarp();
    }
  }
}

#ifndef __CUDACC_RTC__
constexpr int kSmoothWarps = 8;

template <bool MAT, bool STATES>
Resident& smooth_resident() {
  static Resident r;
  return r;
}

template <bool MAT, bool STATES>
cudaError_t smooth_store_cfg(int& blocks) {
  Resident& r = smooth_resident<MAT, STATES>();
  const cudaError_t e = resident_blocks(smooth_kernel<kSmoothWarps, MAT, STATES>, kSmoothWarps * kWarp,
                                        smooth_smem_bytes<kSmoothWarps>(), r);
  if (r.blocks > blocks) blocks = r.blocks;
  return e;
}

// Segment store (float4 count) the smoother needs (the largest of its variants).
inline cudaError_t smooth_store(int64_t& float4s) {
  int blocks = 0;
  cudaError_t e = smooth_store_cfg<false, false>(blocks);
  if (e == cudaSuccess) e = smooth_store_cfg<true, false>(blocks);
  if (e == cudaSuccess) e = smooth_store_cfg<false, true>(blocks);
  if (e == cudaSuccess) e = smooth_store_cfg<true, true>(blocks);
  float4s = (int64_t)blocks * kSmoothWarps * kCkptEvery * kStateF4 * kWarp;
  return e;
}

template <bool MAT, bool STATES>
cudaError_t launch_smooth_cfg(const SmoothArgs& a, cudaStream_t s) {
  if (!STATES && a.tape && a.ck_form == 1) {  // it may count items and lists
    const cudaError_t e = clear_work(a.work, false, true, s);
    if (e != cudaSuccess) return e;
  }
  return launch_persistent(smooth_kernel<kSmoothWarps, MAT, STATES>, smooth_resident<MAT, STATES>(), kSmoothWarps,
                           sizeof(BwdSmem), sizeof(BwdWarpBufs), a, s);
}

constexpr int kSmoothTapeSqrtWarps = 8;

template <int WARPS, int FORM, bool MAT, bool STATES>
cudaError_t launch_smooth_tape(const SmoothArgs& a, cudaStream_t s) {
  constexpr size_t kBlock = FORM == 1 ? sizeof(SmemTables) : sizeof(BwdSmem);
  static Resident r;
  auto kernel = smooth_tape_kernel<WARPS, FORM, MAT, STATES>;
  cudaError_t e = resident_blocks(kernel, WARPS * kWarp, kBlock + WARPS * sizeof(SmoothWarp<STATES, FORM>), r);
  if (e != cudaSuccess) return e;
  SmoothArgs b = a;
  b.item_tracks = item_tracks(a.n_tracks, r.sms);
  const int64_t units = ((int64_t)a.n_tracks + b.item_tracks - 1) / b.item_tracks * SmoothOut<STATES>::kUnits;
  const int blocks = (int)(units < r.blocks ? units : r.blocks);
  const int64_t per_block = (units + blocks - 1) / blocks;
  const int warps = (int)(per_block < WARPS ? per_block : WARPS);
  e = clear_work(a.work, false, units > (int64_t)blocks * warps, s);
  if (e != cudaSuccess) return e;
  kernel<<<blocks, warps * kWarp, kBlock + warps * sizeof(SmoothWarp<STATES, FORM>), s>>>(b);
  return cudaGetLastError();
}

template <bool STATES>
cudaError_t launch_smooth_of(const SmoothArgs& a, cudaStream_t s) {
  if (a.tape) {
    cudaError_t e;
#if !TPCFIT_DET
    if (a.ck_form == 1)
      e = launch_smooth_tape<STATES ? 10 : 12, 1, false, STATES>(a, s);
    else  // the fast square-root form is on the tape with material layers only
      e = launch_smooth_tape<kSmoothTapeSqrtWarps, 0, true, STATES>(a, s);
#else
    e = a.mat ? launch_smooth_tape<kSmoothTapeSqrtWarps, 0, true, STATES>(a, s)
              : launch_smooth_tape<kSmoothTapeSqrtWarps, 0, false, STATES>(a, s);
#endif
    if (e != cudaSuccess) return e;
  }
  // from checkpoints: everything, or the items that the tape had no room for; and
  // the ends
  return a.mat ? launch_smooth_cfg<true, STATES>(a, s) : launch_smooth_cfg<false, STATES>(a, s);
}

inline cudaError_t launch_smooth(const SmoothArgs& a, cudaStream_t s) {
  if (a.n_tracks <= 0) return cudaSuccess;
  return a.state ? launch_smooth_of<true>(a, s) : launch_smooth_of<false>(a, s);
}
#endif

}  // namespace TPCFIT_NS
}  // namespace tpcfit
