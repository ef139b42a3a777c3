// Images of the register sweep's tables (see qsweep.h): the templates, packed on
// the host (qsweep.cu has the kernel that writes the images from them).
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "hs_internal.h"
#include "qsweep.h"

namespace hs {
namespace q {
namespace {

template <typename R>
void pack_ops(const Args& a, unsigned char* out) {
  for (int i = 0; i < a.n_ops; ++i) {
    OpRec<R> r{};
    r.op = a.ops[i];
    int32_t rec[5];
    op_records(a, i, rec);
    std::memcpy(r.c.v, rec, sizeof(rec));
    std::memcpy(out + sizeof(OpRec<R>) * i, &r, sizeof(r));
  }
}

}  // namespace

int Images::add(const Args& a) {
  const SmemMap m = smem_map(a, uint32_t(elem_bytes(dt_)), 1u << (a.tile_bits - B_));
  const uint32_t bytes = m.fac - m.ops;
  const int in_chunk = dt_ == HS_C64 ? 1 : 0;
  std::vector<unsigned char> t(bytes, 0);
  auto put = [&](uint32_t at, const void* src, size_t n) {
    if (n) std::memcpy(t.data() + (at - m.ops), src, n);
  };
  if (dt_ == HS_C64) pack_ops<float>(a, t.data());
  else pack_ops<double>(a, t.data());
  for (int li = 0; li < a.n_lay; ++li) {
    LayRec r{};
    r.L = a.lay[li];
    for (int j = 0; j < 48; ++j) {
      const uint32_t d = deposit_index(r.L, j);
      r.dep[j] = make_uint2(d, swz(d >> in_chunk));
    }
    put(m.lays + uint32_t(sizeof(LayRec)) * li, &r, sizeof(r));
  }
  put(m.tabs, a.tab, sizeof(Tab) * a.n_tab);
  put(m.ph, a.ph, sizeof(Phase) * a.n_phase);
  put(m.cls, a.cls, sizeof(PClass) * a.n_cls);
  put(m.pt, a.pt, sizeof(PTerm) * a.n_pterm);
  uint32_t clane[48];
  for (int j = 0; j < 48; ++j) clane[j] = copy_index(a.lay[a.ops[0].idx], j, in_chunk);
  put(m.clane, clane, sizeof(clane));
  FillRec f{};
  f.rq = a.rq;
  f.cs = a.cs;
  f.vt = a.vt;
  f.n_vt_g = a.n_vt_g;
  f.n_terms_g = a.n_terms_g;
  f.bytes = bytes;
  f.n_ops = a.n_ops;
  f.n_tab = a.n_tab;
  f.n_pterm = a.n_pterm;
  f.ops = 0;
  f.tabs = m.tabs - m.ops;
  f.vts = m.vts - m.ops;
  f.pt = m.pt - m.ops;
  f.thpi = m.thpi - m.ops;
  f.scale = m.scale - m.ops;
  recs_.push_back(f);
  tmpl_off_.push_back(tmpl_.size());
  tmpl_.insert(tmpl_.end(), t.begin(), t.end());
  tmpl_.resize((tmpl_.size() + 255) / 256 * 256);
  img_off_.push_back(img_bytes_);
  img_bytes_ += (size_t(bytes) + 255) / 256 * 256;
  return int(recs_.size()) - 1;
}

std::vector<unsigned char> Images::blob(unsigned char* dev) const {
  std::vector<unsigned char> b(rec_bytes(), 0);
  for (size_t i = 0; i < recs_.size(); ++i) {
    FillRec f = recs_[i];
    f.tmpl = dev + rec_bytes() + tmpl_off_[i];
    f.img = dev + host_bytes() + img_off_[i];
    std::memcpy(b.data() + i * sizeof(FillRec), &f, sizeof(f));
  }
  b.insert(b.end(), tmpl_.begin(), tmpl_.end());
  return b;
}

Hdr Images::header(const Args& a, int i, unsigned char* dev) const {
  Hdr h{};
  h.src = a.src;
  h.dst = a.dst;
  h.img = dev + host_bytes() + img_off_[i];
  h.N = a.N;
  h.sm = smem_map(a, uint32_t(elem_bytes(dt_)), 1u << (a.tile_bits - B_));
  h.img_bytes = h.sm.fac - h.sm.ops;
  h.m0 = a.m0;
  h.m1 = a.m1;
  h.sh = a.sh;
  h.rest = a.rest;
  h.n_rhs = a.n_rhs;
  h.n_tiles_log2 = a.n_tiles_log2;
  h.rhs_chunk = a.rhs_chunk;
  h.rhs_chunks = a.rhs_chunks;
  h.n_chunks = a.n_chunks;
  h.n_ops = a.n_ops;
  h.n_phase = a.n_phase;
  h.n_cls = a.n_cls;
  h.first_lay = a.ops[0].idx;
  h.last_lay = a.last_lay;
  h.free_local = a.free_local;
  h.fac_keep = a.fac_keep;
  return h;
}

}  // namespace q
}  // namespace hs
