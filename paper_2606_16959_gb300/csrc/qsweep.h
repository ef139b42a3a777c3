// Register-blocked tile sweep ("q-sweep"): launch descriptor shared by the
// host planner (qplan.cpp) and the kernel (qsweep.cu).
//
// A CTA holds a tile of 2^T amplitudes of ONE state (the rows whose bits
// outside the tile's local bit set are fixed by the CTA index, as in the
// staged sweep) in shared memory, and each thread keeps 2^B of the tile's
// rows in registers: the rows l = l_t | pdep(k, reg) for k = 0 .. 2^B - 1,
// where `reg` is a set of B local bits (the register bits) and l_t places the
// thread index on the other local bits.  A factor whose flips lie in the
// register bits is applied in registers with no exchange; a LAYOUT op changes
// the register bits by one pass through shared memory.
//
// A factor of the sweep becomes a short list of ops:
//   TAB    a factor with a value table and at most two slots (x-mask set
//          {0, u}): row r's entries F[r, r] and F[r, r ^ u] are read from the
//          table at the pattern of r's bits on the factor's support;
//   ROT    one non-diagonal term of a factor without such a table: its exact
//          rotation cos(theta) I - i sin(theta) P_j, from the FP64 (cos, sin)
//          of the factor build; an X-type term (y = 0, z = 0) in the form
//          cos(theta') (I - i tan(theta') P_j) (-i P_j)^k, theta = theta' +
//          k pi / 2, |theta'| <= pi / 4: two fused multiply-adds per
//          amplitude, cos(theta') and (-i)^k in one scale per sweep, an odd
//          k a swap of partner rows;
//   ROTN   a run of consecutive X-type single-qubit rotations on distinct
//          register bits (they commute), applied back to back in that form;
//   BOND   the terms XX, YY and ZZ of one qubit pair with one angle theta (they
//          commute): exp(-i theta (XX + YY + ZZ)) = e^{-i theta} (I + w S), where
//          S takes (x01, x10) to (x10 - x01, x01 - x10) and every other row to 0,
//          w = (1 - e^{4 i theta}) / 2; the phase goes into the sweep's scale.
//          10 real operations per pair of rows that change, none for the others,
//          against 32 through a value table;
//   DROT   a single diagonal term between non-diagonal ones: its rotation
//          exp(-i theta (-1)^popcount(z & r)) from the build's FP64 (cos, sin);
//   PHASE  a run of consecutive diagonal terms (x = 0) of such a factor: the
//          phase exp(-i sum_j theta_j (-1)^popcount(z_j & r)) computed for
//          each row from (z_j, theta_j) -- the factor values are generated
//          inside the sweep instead of being read from stored diagonals.
// Terms of a factor are applied in the factor's order, so a factor's ops
// multiply out to the factor itself (F_g = R_last ... R_first).
#pragma once

#include <cstdint>
#include <memory>
#include <utility>

#include "hs_internal.h"

namespace hs {
namespace q {

constexpr int kMaxOps = 160;
constexpr int kMaxLayouts = 40;
constexpr int kMaxRot = 96;
constexpr int kMaxTab = 24;
constexpr int kMaxPhase = 12;
constexpr int kMaxPTerms = 320;
constexpr int kMaxClasses = 256;
constexpr int kMaxVt = 2048;   // value-table entries held in shared memory
constexpr int kMaxB = 5;       // register bits per thread
constexpr int kMaxBond = 64;
constexpr int kMaxRhsChunk = 4;  // states of one tile a CTA runs back to back

enum : uint8_t { OP_ROT = 0, OP_TAB = 1, OP_PHASE = 2, OP_LAYOUT = 3, OP_ROTN = 4, OP_DROT = 5, OP_BOND = 6 };

struct Op {
  uint8_t type;
  uint8_t ku;     // ROT, TAB, BOND: the flip in register coordinates (TAB: 0 for a one-slot factor)
  uint8_t zk;     // ROT: the register coordinates of z's bits in the tile
  uint8_t flags;  // ROT: bit 0 = fast path (y = 0 and z = 0); bits 1-2 = q with -i i^y = i^q;
                  // BOND: 1 = the factor's only terms (it has a value table)
  int16_t idx;    // ROT: rotation slot; TAB: table slot; BOND: bond slot; PHASE: phase slot; LAYOUT: layout slot
  int16_t pad;
  uint32_t zthr;  // ROT: z's bits in the tile on thread positions (local-index mask)
  uint32_t zrest; // ROT: z's bits outside the tile (global mask)
  // ROTN (a run of consecutive rotations exp(-i theta X_q) on distinct single
  // register bits, which commute): ku is the mask of those register bits and
  // byte i of (zthr, zrest) the rotation slot of register bit i.
};

constexpr int kMaxNJB = 4;  // register bits that select a thread's 16-byte chunks

struct alignas(16) Layout {
  // Per register bit above those inside a chunk (complex64: above bit 0): XOR
  // offset of the physical 16-byte chunk index, and the global row offset
  // (global image of the local bit).
  uint32_t qoff[kMaxNJB];
  uint32_t goff[kMaxNJB];
  // A warp's rows (fixed warp bits, all register and lane bits) copied in
  // address order: chunk e = lane + 32 m of the warp's set lies at chunk
  // pdep(lane, wlo) ^ pdep(32 m, W) ^ (the warp's fixed chunk bits), W the
  // warp's chunk bits; mswz / mglob hold the swizzled chunk and global row
  // of pdep(32 m, W) for m = 1, 2, 4, 8 (both maps are linear over XOR).
  uint32_t mswz[kMaxNJB];
  uint32_t mglob[kMaxNJB];
  uint32_t reg;        // local-index mask of the register bits (register bit i = i-th lowest set bit)
  uint32_t g0;         // complex64: global row offset of register bit 0
  int8_t thr[28];      // local positions of the thread-index bits, thread bit 0 first
  int32_t n_thr;
  int8_t wlo[5];       // the five lowest chunk bits of W
  int8_t pad[3];
};

struct Rot {
  int32_t cs;    // index of the term's (cos, sin) pair in the factor set's angle table
  int32_t fast;  // y = 0 and z = 0: kept as a ratio with its larger factor in the sweep's scale
};

struct Tab {
  int32_t vt0;  // first entry in the factor set's value tables
  int32_t s0;   // first entry in shared memory
  int32_t n;    // entries
  uint32_t sm;  // support mask (global bits); the pattern of row r indexes the table
  int8_t sh;    // lowest bit of sm when its bits are consecutive, else -1
  int8_t ns;    // slots (1 or 2)
  int16_t pad;
};

struct Phase {
  int16_t cls0, ncls;  // classes [cls0, cls0 + ncls); class cls0 has the empty local part
  uint32_t mu_mask;    // register patterns mu that have at least one class besides cls0
  int16_t mu_beg[(1 << kMaxB) + 1];  // per mu: first class (relative to cls0; mu = 0 starts
                                     // after the constant class), sentinel last
  int16_t fac0;        // first of the run's factor slots (mu = 0, one per register bit, one per
                       // further pattern present)
  int16_t pad;
};

struct PClass {
  uint32_t thr;   // local part on thread positions (local-index mask)
  int16_t t0, nt; // terms [t0, t0 + nt) of the phase term list
  int16_t c0p;    // the phase op whose constant class (empty local part) this is, else -1
  int16_t mu;     // register part (register coordinates)
};

struct PTerm {
  int32_t th;     // index of theta_j in the factor set's angle table
  uint32_t rest;  // z_j's bits outside the tile (global mask)
};

struct Args {
  const void* src;
  void* dst;
  const double* cs;  // (cos, sin) per kind and term (FP64)
  const double* th;  // theta per kind and term (FP64)
  const double* rq;  // register-sweep record per kind and term (FP64, see the factor build)
  const void* vt;    // value tables (storage type)
  int64_t N;
  int64_t n_vt_g;    // extents of vt and of the per-term records (index checks only)
  int n_terms_g;
  int n_rhs;
  int tile_bits;
  int n_tiles_log2;
  // Work is cut into chunks of up to rhs_chunk consecutive states of one tile
  // (chunk q: tile q / rhs_chunks, states from (q % rhs_chunks) * rhs_chunk).
  int rhs_chunk, rhs_chunks, n_chunks;
  uint32_t m0, m1;  // local index of global row r: (r & m0) | ((r >> sh) & m1)
  int sh;
  Runs rest;
  int n_ops, n_lay, n_rot, n_tab, n_phase, n_cls, n_pterm, n_vt, n_bond;
  int n_fac;         // phase factor slots a thread has in shared memory
  int fac_keep;      // 1: every PHASE run has slots of its own (kept for all states of a chunk);
                     // 0: the runs share slots and their factors are computed on each use
  int lean;          // 1: the instantiation with the factors in local memory (n_fac = 0) and one copy
                     // of the class constants per CTA
  int last_lay;      // index of the last LAYOUT op
  int free_local;    // 1: the last layout's warp bits are the first one's
  int exact_scale;   // complex64 bonds: 1 takes the instantiation that applies the scale unrounded
  int full;          // 1 if a TAB op or a rotation other than tan form occurs (the larger kernel)
  Op ops[kMaxOps];
  Layout lay[kMaxLayouts];
  Rot rot[kMaxRot];
  Tab tab[kMaxTab];
  int32_t bond[kMaxBond];  // index of the bond's angle records
  Phase ph[kMaxPhase];
  PClass cls[kMaxClasses];
  PTerm pt[kMaxPTerms];
};

// Physical 16-byte chunk of natural chunk c in the shared-memory tile: the
// XOR fold of c's higher bit triples into its lowest three bits spreads the
// chunks a quarter-warp touches over distinct 16-byte bank groups.
__host__ __device__ __forceinline__ uint32_t swz(uint32_t c) {
  return c ^ (((c >> 3) ^ (c >> 6) ^ (c >> 9) ^ (c >> 12) ^ (c >> 15)) & 7u);
}

// The register patterns mu of two or more bits among those present, by where
// they lie: inside the lower group of register bits (0 .. (B + 1) / 2 - 1),
// inside the upper group (in coordinates of that group for lower / upper), or
// across the groups.  A set of patterns is a mask with bit mu.
template <int B>
__host__ __device__ __forceinline__ uint32_t lower_patterns(uint32_t mu_mask) {
  uint32_t m = 0;
  for (int mu = 3; mu < (1 << ((B + 1) / 2)); ++mu)
    if (mu & (mu - 1)) m |= 1u << mu;
  return mu_mask & m;
}
template <int B>
__host__ __device__ __forceinline__ uint32_t upper_patterns(uint32_t mu_mask) {
  constexpr int B1 = (B + 1) / 2;
  uint32_t m = 0;
  for (int nu = 3; nu < (1 << (B - B1)); ++nu)
    if ((nu & (nu - 1)) && ((mu_mask >> (nu << B1)) & 1u)) m |= 1u << nu;
  return m;
}
template <int B>
__host__ __device__ __forceinline__ uint32_t inside_patterns(uint32_t mu_mask) {
  constexpr int B1 = (B + 1) / 2;
  uint32_t m = 0;
  for (int nu = 3; nu < (1 << (B - B1)); ++nu)
    if (nu & (nu - 1)) m |= 1u << (nu << B1);
  return lower_patterns<B>(mu_mask) | (mu_mask & m);
}
template <int B>
__host__ __device__ __forceinline__ uint32_t across_patterns(uint32_t mu_mask) {
  uint32_t m = ~1u;
  for (int i = 0; i < B; ++i) m &= ~(1u << (1 << i));
  return mu_mask & m & ~inside_patterns<B>(0xffffffffu);
}

// Host planner: the ops of a fused sweep (factors in order, two-run local mask)
// for tiles of T bits and B register bits.  Returns false (with a reason) when
// a factor cannot be expressed as register ops or a limit is exceeded.
// steps (optional): the step of each factor application, for a sweep that
// spans steps of a time-dependent set whose terms have one record per step:
// a term record is then addressed (step - steps[0]) * step_stride + kind * m
// + term, relative to the records of the sweep's first step.
// reserve: shared memory that a launch needs beside the descriptor's (the header
// and prefix table of a batch).
bool plan_qsweep(const hs_factors* f, const std::vector<int>& factors, uint32_t local_mask, int T, int B,
                 Args& a, std::string* why, const std::vector<int>* steps = nullptr, int step_stride = 0,
                 size_t reserve = 0);

// The tile bits with which HS_METHOD_AUTO takes register sweeps, 0 where it
// takes the staged ones.
int auto_tile_bits(const hs_factors* f, int n_rhs, int n_steps);

// plan_qsweep for a run of factors that may exceed a descriptor's limits: the
// run is split into consecutive shorter runs (same local mask) until each
// fits.  Returns false if a single factor cannot be expressed.
bool plan_qsweep_runs(const hs_factors* f, const std::vector<int>& factors, uint32_t local_mask, int T, int B,
                      std::vector<std::pair<std::vector<int>, std::shared_ptr<Args>>>& out, std::string* why,
                      const std::vector<int>* steps = nullptr, int step_stride = 0, size_t reserve = 0);

// ---------------------------------------------------------------------------
// Tables in shared memory.  A CTA of a single launch makes them from the
// descriptor, its kernel parameter, and the term records: 10,500 cycles (4,000
// to copy the descriptor, 2,700 for the coefficients, 3,800 for the FP64
// scale), which hide behind the sweep before (programmatic dependent launch)
// and serve every chunk of a resident CTA.  A CTA of a batch level runs one
// chunk and starts among running ones, where they would show each time: a
// batch has every descriptor's tables in device memory as the very bytes a CTA
// wants, its image, written by one small kernel per batch launch (launch_fill)
// and copied by the CTA with a few 16-byte loads (32 uneven chains: 2.93 ms
// with tables made by each CTA, 2.37 ms with images; single launches with
// images were 4% slower, 74.4 and 77.2 ms on the 24-qubit MaxCut instance).
// ---------------------------------------------------------------------------

// An op's coefficients: ROTN the tan(theta') of register bits 0 .. 4, ROT and
// DROT (cos, sin) or (tan, 0), BOND w; `swap` the register bits (ROTN) or the
// flag (ROT) of odd quarter turns.  In a template the first five words hold
// the record each coefficient comes from.
template <typename R>
struct alignas(16) Coef {
  R v[5];
  uint32_t swap;
  uint32_t pad[sizeof(R) == 4 ? 2 : 1];
};

// An op with its coefficients; a layout with the local row (x) and the
// swizzled chunk (y) that a lane index (0 .. 31) and a warp index (32 ..)
// deposit: a thread's register row 0 is the XOR of the two.
template <typename R>
struct OpRec {
  Op op;
  Coef<R> c;
};
struct LayRec {
  Layout L;
  uint2 dep[48];
};

// ROTN: the rotation slot of register bit i.
__host__ __device__ __forceinline__ int rotn_slot(const Op& op, int i) {
  return int((i < 4 ? (op.zthr >> (8 * i)) : (op.zrest >> (8 * (i - 4)))) & 0xffu);
}

// The local row that index j of a LayRec deposits (lane j, or warp j - 32), and
// the one it deposits in the copies of a layout's rows in address order.
__host__ __device__ __forceinline__ uint32_t deposit_index(const Layout& L, int j) {
  uint32_t d = 0;
  if (j < 32)
    for (int i = 0; i < 5 && i < L.n_thr; ++i) d |= uint32_t((j >> i) & 1) << L.thr[i];
  else
    for (int i = 5; i < L.n_thr; ++i) d |= uint32_t(((j - 32) >> (i - 5)) & 1) << L.thr[i];
  return d;
}
__host__ __device__ __forceinline__ uint32_t copy_index(const Layout& L, int j, int in_chunk) {
  uint32_t d = 0;
  if (j < 32)
    for (int k = 0; k < 5; ++k) d |= uint32_t((j >> k) & 1) << (L.wlo[k] + in_chunk);
  else
    for (int i = 5; i < L.n_thr; ++i) d |= uint32_t(((j - 32) >> (i - 5)) & 1) << L.thr[i];
  return d;
}

// Byte offsets of a CTA's tables in shared memory: the tile, the image (ops to
// scale), then what the kernel fills itself (fac, e0s, cw).
struct SmemMap {
  uint32_t ops, lays, tabs, vts, ph, cls, pt, thpi, clane, scale, fac, e0s, cw, total;
};

__host__ __device__ inline SmemMap smem_map(const Args& a, uint32_t e, uint32_t nt) {
  SmemMap m;
  uint32_t o = e << a.tile_bits;
  auto take = [&](uint32_t bytes) {
    const uint32_t at = o;
    o += (bytes + 15u) & ~15u;
    return at;
  };
  const uint32_t copies = a.lean ? 1u : nt >> 5;  // of the class constants
  m.ops = take((e == 8 ? sizeof(OpRec<float>) : sizeof(OpRec<double>)) * a.n_ops);
  m.lays = take(sizeof(LayRec) * a.n_lay);
  m.tabs = take(sizeof(Tab) * a.n_tab);
  m.vts = take(e * a.n_vt);
  m.ph = take(sizeof(Phase) * a.n_phase);
  m.cls = take(sizeof(PClass) * a.n_cls);
  m.pt = take(sizeof(PTerm) * a.n_pterm);
  m.thpi = take((e / 2) * a.n_pterm);
  m.clane = take(48 * 4);
  m.scale = take(16);  // complex64: the scale and what its rounding lost
  m.fac = take(e * nt * a.n_fac);
  m.e0s = take(e * copies * a.n_phase);
  m.cw = take(e * copies * a.n_cls);  // a class constant and its mask: the element size
  m.total = o;
  return m;
}

// What a CTA of a batch level needs of its descriptor.
struct Hdr {
  const void* src;
  void* dst;
  const unsigned char* img;  // the image
  int64_t N;
  uint32_t img_bytes;        // a multiple of 16
  uint32_t m0, m1;
  int sh;
  Runs rest;
  int n_rhs;
  int n_tiles_log2;
  int rhs_chunk, rhs_chunks, n_chunks;
  int n_ops, n_phase, n_cls;
  int first_lay;             // layout the sweep starts in
  int last_lay, free_local, fac_keep;
  SmemMap sm;
};

struct FillRec {
  const unsigned char* tmpl;
  unsigned char* img;
  const double* rq;
  const double* cs;
  const void* vt;
  int64_t n_vt_g;
  int n_terms_g;
  uint32_t bytes;            // of the image
  int n_ops, n_tab, n_pterm;
  uint32_t ops, tabs, vts, pt, thpi, scale;  // byte offsets in the image
};

// The images of a set of launches.
class Images {
 public:
  Images(hs_dtype dt, int B) : dt_(dt), B_(B) {}
  // Adds descriptor a (with its job fields: fill_job); returns the image's number.
  int add(const Args& a);
  int count() const { return int(recs_.size()); }
  // Device bytes, the first host_bytes() of which are uploaded from blob(dev).
  size_t device_bytes() const { return host_bytes() + img_bytes_; }
  size_t host_bytes() const { return rec_bytes() + tmpl_.size(); }
  std::vector<unsigned char> blob(unsigned char* dev) const;
  // The header of a launch of a with image number i, the images at dev.
  Hdr header(const Args& a, int i, unsigned char* dev) const;

 private:
  size_t rec_bytes() const { return (recs_.size() * sizeof(FillRec) + 255) / 256 * 256; }
  hs_dtype dt_;
  int B_;
  std::vector<FillRec> recs_;
  std::vector<size_t> tmpl_off_, img_off_;
  std::vector<unsigned char> tmpl_;
  size_t img_bytes_ = 0;
};

// The term records of an op (ROTN: one per register bit).
void op_records(const Args& a, int oi, int32_t (&rec)[5]);

// Write n images (records at the start of dev).
cudaError_t launch_fill(hs_dtype dt, const unsigned char* dev, int n, cudaStream_t s);

size_t qsweep_smem_bytes(const Args& a, hs_dtype dt, int B);

// The job-dependent fields of a descriptor: state (evolved in place), the
// factor set's angle records and value tables, and the chunks of work (tiles
// of the planned local mask times n_rhs states, rhs_chunk states at a time).
void fill_job(const hs_factors* f, Args& a, void* psi, int n_rhs, int rhs_chunk);

// States per chunk for a launch of `tiles` tiles of n_rhs states on `slots`
// resident CTAs.
int pick_rhs_chunk(int64_t tiles, int n_rhs, int slots);

// One level of a batch of register sweeps: CTA c runs chunk c - prefix[e] of
// descriptor lvl_desc[off + e], e the last entry with prefix[off + e] <= c.
struct LevelArgs {
  const Hdr* descs;
  const int* lvl_desc;
  const int* lvl_prefix;
  int off, count;
  uint32_t prefix_smem;  // byte offset in shared memory of a CTA's header, the level's prefix table after it
};
constexpr uint32_t kHdrSmem = 256;
static_assert(sizeof(Hdr) <= kHdrSmem, "a header and the prefix table do not overlap");
cudaError_t launch_qlevel(hs_dtype dt, int B, bool full, bool lean, int tile_bits, const LevelArgs& L, int64_t ctas, size_t smem,
                          bool pdl, cudaStream_t s);
// rq, cs (optional): term records to use instead of the factor set's own
// (n_terms of them), for a sweep over steps of a time-dependent set.
cudaError_t launch_qsweep(const hs_factors* f, Args& a, const void* src, void* dst, int n_rhs, int B,
                          bool pdl, cudaStream_t s, const double* rq = nullptr, const double* cs = nullptr,
                          int n_terms = 0);
cudaError_t prepare_qsweep();

}  // namespace q
}  // namespace hs
