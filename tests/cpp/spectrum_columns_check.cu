// Host-only check of the spectrum columns of a block set (number_columns and
// spectra_need of flgf_api.cu), forward and adjoint phases: every block that a
// block-wise list names has a column, the same one in every list, below the
// phase's count; the components of a vector block set keep one distance; the
// passes between parents cover the groups in turn, each with its own parents'
// columns; the frequency-lane kernel's form and shared memory follow the groups
// that it runs; and the spectra and the sums together take no more room than those of
// every block of the largest phase would, but for a pass of a single group.
// The counts of flgf_work_detail are those of the forward tables.
//
// usage: spectrum_columns_check <mesh file> <list_pct> <fp64 0|1> <mac> <ncomp> <pass bytes>
#include "../../paper_1911_10228_gb300/csrc/flgf_api.cu"

#include <cstdio>

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  FILE* fp = fopen(argv[1], "rb");
  if (!fp) return 2;
  auto rd = [&](int* v, size_t n) { return fread(v, sizeof(int), n, fp) == n; };
  int N = 0, np = 0, nl = 0, nb = 0;
  if (!rd(&N, 1) || !rd(&np, 1)) return 2;
  std::vector<int> nlev(np);
  if (!rd(nlev.data(), np)) return 2;
  for (int v : nlev) nl += v;
  std::vector<int> nblk(nl);
  if (!rd(nblk.data(), nl)) return 2;
  for (int v : nblk) nb += v;
  std::vector<int32_t> coords(3 * (size_t)nb);
  if (!rd(coords.data(), coords.size())) return 2;
  fclose(fp);
  std::vector<double> h0(np, 1.0);
  flgf_ctx ctx;
  ctx.N = N;
  ctx.max_oct = 8;
  ctx.list_pct = atoi(argv[2]);
  ctx.prec = atoi(argv[3]) ? FLGF_FP64 : FLGF_FP32;
  ctx.mac = atoi(argv[4]);
  ctx.pf_bytes = (size_t)atoll(argv[6]);
  auto bs = new flgf_blockset();
  bs->ctx = &ctx;
  bs->ncomp = atoi(argv[5]);
  if (plan_blockset(&ctx, bs, np, nlev.data(), nblk.data(), coords.data(), h0.data()) != FLGF_OK) return 1;
  build_adjoint(bs);  // the lists are complete; its allocations fail without a GPU
  long bad = 0, named = 0, cols = 0, passes = 0;
  bool single = false;  // a pass of one group exceeds the bound
  const size_t csz = ctx.prec == FLGF_FP64 ? 16 : 8, all = csz * (size_t)nfreq(N) * bs->max_phase_blocks;
  int64_t work[FLGF_WORK_COUNT] = {0};
  auto check = [&](const PhaseOff& ph, const std::vector<char>& host, bool forward) {
    std::vector<char> img = host;
    number_columns(ph, img.data());
    auto at = [](const std::vector<char>& v, size_t off) { return reinterpret_cast<const int*>(v.data() + off); };
    // the columns: the transformed blocks in the order of their ids
    std::vector<int> col(ph.nblocks, -1);
    for (int i = 0; i < ph.n_fwd; ++i) col[at(host, ph.fwd_sid)[i]] = 0;
    for (int i = 0; i < ph.n_inv; ++i) col[at(host, ph.inv_sid)[i]] = 0;
    int n = 0;
    for (int& c : col) c = c < 0 ? -1 : n++;
    bad += n != ph.ncol;
    cols += n;
    auto same = [&](size_t off, size_t first, size_t count) {
      for (size_t i = first; i < first + count; ++i, ++named) {
        const int id = at(host, off)[i], c = at(img, off)[i];
        bad += id < 0 ? c != id : id >= ph.nblocks || col[id] < 0 || c != col[id];
      }
    };
    same(ph.fwd_sid, 0, ph.n_fwd);
    same(ph.inv_sid, 0, ph.n_inv);
    const HadGroup* hg = reinterpret_cast<const HadGroup*>(host.data() + ph.hgroups);
    for (int g = 0; g < ph.n_groups_dense; ++g) {
      same(ph.src_ids, hg[g].src_off, 8 * hg[g].ncell);
      same(ph.tgt_ids, hg[g].tgt_off, 8 * hg[g].nact);
    }
    const FlGroup* fg = reinterpret_cast<const FlGroup*>(host.data() + ph.fl_groups);
    for (int g = ph.n_pf; g < ph.n_fl; ++g) {
      same(ph.fl_cells, 8 * fg[g].cell_off, 8 * fg[g].ncell);
      same(ph.fl_tgt, 8 * fg[g].row_off, 8 * fg[g].nact);
      for (int c = 1; c < ph.fl_ncomp; ++c)
        for (int i = 0; i < 8 * fg[g].nact; ++i) {
          const int t = at(host, ph.fl_tgt)[8 * fg[g].row_off + i];
          bad += t >= 0 && col[t + c * ph.fl_cstride] != col[t] + c * (ph.ncol / ph.fl_ncomp);
        }
    }
    long rows = 0, full = 0;
    int cells = 0, parents = 0;
    for (int g = ph.n_pf; g < ph.n_fl; ++g) {
      cells = std::max(cells, fg[g].ncell);
      parents = std::max(parents, fg[g].nact);
      for (int m = fg[g].row_off; m < fg[g].row_off + fg[g].nact; ++m) {
        const int k = reinterpret_cast<const uint16_t*>(host.data() + ph.fl_rows)[(size_t)m * kFlRowStride];
        rows += k;
        for (int j = 0; j < k; ++j)
          full += reinterpret_cast<const uint32_t*>(host.data() + ph.fl_dlms)[(size_t)m * kFlDelta + j] >> 31;
      }
    }
    bad += cells != ph.fl_run_cells || parents != ph.fl_run_parents ||
           ph.fl_run_split != (rows > 0 && (double)full >= kFlSplitFullFraction * (double)rows);
    const FllGroup* qg = reinterpret_cast<const FllGroup*>(host.data() + ph.fll_groups);
    for (int g = 0; g < ph.n_fll; ++g)
      for (int t = qg[g].tgt_off; t < qg[g].tgt_off + qg[g].ntgt; ++t) {
        same(ph.fll_tgt, t, 1);
        for (int j = at(host, ph.fll_beg)[t], e = j + at(host, ph.fll_len)[t]; j < e; ++j, ++named) {
          const uint32_t a = at(host, ph.fll_ent)[j], b = at(img, ph.fll_ent)[j];
          bad += (a & 511) != (b & 511) || col[a >> 9] < 0 || col[a >> 9] != (int)(b >> 9);
        }
      }
    const ListGroup* lg = reinterpret_cast<const ListGroup*>(host.data() + ph.groups);
    for (int g = 0; g < ph.n_groups + ph.n_groups_out; ++g) {
      same(ph.l_tgt, lg[g].tgt_off, lg[g].ntgt);
      same(ph.l_src, lg[g].src_off, lg[g].nsrc);
    }
    const PfGroup* pg = reinterpret_cast<const PfGroup*>(host.data() + ph.pf_groups);
    int g0 = 0, s0 = 0, t0 = 0;
    for (const PfPass& q : ph.pf_pass) {
      bad += q.g0 != g0 || q.s0 != s0 || q.t0 != t0 || q.ng < 1;
      const size_t bytes = csz * (pf_source_values(N, csz == 16) * q.ns + pf_parent_values(N) * q.nt);
      if (ph.fl_ncomp == 1 && bytes > std::max(ctx.pf_bytes, 2 * all)) {
        single = true;
        bad += q.ng != 1;
      }
      std::vector<int> tcol;
      for (int g = q.g0; g < q.g0 + q.ng; ++g) {
        for (int c = 0; c < pg[g].ncell; ++c) {
          const int k = at(host, ph.pf_ccol)[pg[g].cell_off + c];
          if (k < 0 || k >= q.ns) { ++bad; continue; }
          for (int b = 0; b < 8; ++b) {
            const int id = at(host, ph.fl_cells)[8 * (fg[g].cell_off + c) + b];
            bad += at(host, ph.pf_sch)[8 * (q.s0 + k) + b] != (id < 0 ? -1 : id + ph.gid_begin);
          }
        }
        for (int m = 0; m < pg[g].nact; ++m) {
          const int k = at(host, ph.pf_tcol)[pg[g].row_off + m];
          tcol.push_back(k);
          if (k < 0 || k >= q.nt) { ++bad; continue; }
          for (int b = 0; b < 8; ++b) {
            const int id = at(host, ph.fl_tgt)[8 * (fg[g].row_off + m) + b];
            bad += at(host, ph.pf_tch)[8 * (q.t0 + k) + b] != (id < 0 ? -1 : id + ph.gid_begin);
          }
        }
      }
      std::sort(tcol.begin(), tcol.end());
      bad += std::adjacent_find(tcol.begin(), tcol.end()) != tcol.end();
      g0 += q.ng; s0 += q.ns; t0 += q.nt;
      ++passes;
    }
    bad += g0 != ph.n_pf || s0 != ph.n_pfs || t0 != ph.n_pft;
    if (!forward) return;
    for (int g = 0; g < ph.n_pf; ++g)
      for (int m = 0; m < fg[g].nact; ++m)
        work[FLGF_WORK_PARENT_PAIRS] +=
            ph.fl_ncomp * reinterpret_cast<const uint16_t*>(host.data() + ph.fl_rows)[(size_t)(fg[g].row_off + m) * kFlRowStride];
    work[FLGF_WORK_PARENT_FWD] += s0;
    work[FLGF_WORK_PARENT_INV] += t0;
    work[FLGF_WORK_BLOCK_FWD] += ph.n_fwd;
    work[FLGF_WORK_BLOCK_INV] += ph.n_inv;
    for (int g = 0; g < ph.n_fll; ++g)
      for (int t = qg[g].tgt_off; t < qg[g].tgt_off + qg[g].ntgt; ++t) work[FLGF_WORK_BLOCK_PAIRS] += at(host, ph.fll_len)[t];
    for (int g = 0; g < ph.n_groups + ph.n_groups_out; ++g)
      for (int m = 0; m < lg[g].ntgt; ++m) work[FLGF_WORK_BLOCK_PAIRS] += at(host, ph.l_len)[lg[g].len_off + m];
    auto pairs = [&](int level, const int* tgt, const int* src, int e) {
      for (int a = 0; a < 8; ++a)
        for (int b = 0; b < 8; ++b) {
          const int d0 = (a >> 2) - (b >> 2) - 2 * (e / 9 - 1), d1 = (a >> 1 & 1) - (b >> 1 & 1) - 2 * (e / 3 % 3 - 1),
                    d2 = (a & 1) - (b & 1) - 2 * (e % 3 - 1);
          const bool near = std::abs(d0) <= 1 && std::abs(d1) <= 1 && std::abs(d2) <= 1;
          work[FLGF_WORK_BLOCK_PAIRS] += tgt[a] >= 0 && src[b] >= 0 && !(level > 0 && near) ? ph.fl_ncomp : 0;
        }
    };
    for (int g = ph.n_pf; g < ph.n_fl; ++g)
      for (int m = 0; m < fg[g].nact; ++m) {
        const uint16_t* row = reinterpret_cast<const uint16_t*>(host.data() + ph.fl_rows) + (size_t)(fg[g].row_off + m) * kFlRowStride;
        for (int j = 1; j <= row[0]; ++j)
          pairs(fg[g].level, at(host, ph.fl_tgt) + 8 * (fg[g].row_off + m),
                at(host, ph.fl_cells) + 8 * (fg[g].cell_off + (row[j] & 0x7FF)), row[j] >> 11);
      }
    for (int g = 0; g < ph.n_groups_dense; ++g)
      for (int m = 0; m < hg[g].nact; ++m)
        for (int e = 0; e < 27; ++e) {
          const uint16_t c = reinterpret_cast<const uint16_t*>(host.data() + ph.par_tab)[hg[g].par_off + e * hg[g].nact + m];
          if (c == kNbEnd) continue;
          int src[8];
          for (int b = 0; b < 8; ++b) src[b] = at(host, ph.src_ids)[hg[g].src_off + b * hg[g].ncell + c];
          pairs(hg[g].level, at(host, ph.tgt_ids) + hg[g].tgt_off + 8 * m, src, e);
        }
  };
  for (int l = 0; l < bs->Lmax; ++l) {
    check(bs->ph[l], bs->ar.host, true);
    check(bs->aph[l], bs->aar.host, false);
  }
  for (int i = 0; i < FLGF_WORK_COUNT; ++i) bad += work[i] != bs->work[i];
  const auto f = spectra_need(&ctx, bs->ph), a = spectra_need(&ctx, bs->aph);
  const size_t most = std::max(ctx.pf_bytes, 2 * all);
  bad += !single && bs->ncomp == 1 && (f.first + f.second > most || a.first + a.second > most);
  printf("bytes of all blocks' spectra %zu: spectra %zu sums %zu, adjoint %zu %zu\n", all, f.first, f.second, a.first, a.second);
  printf("columns %ld named %ld passes %ld mismatches %ld\n%s\n", cols, named, passes, bad, bad ? "FAILED" : "ok");
  return bad ? 1 : 0;
}
