// Host-only check of the tables of the products between parents (parent.cu):
// in every phase, forward and adjoint, each target of a level between parents is
// written exactly once (a child of a target parent, or of the block-wise
// inverse), the near pairs of the coarser levels are taken out exactly once, the
// parents' items and columns say the same as the frequency-lane groups they are
// made from, and the sources of the block-wise kernels are all transformed.
//
// usage: parent_plan_check <mesh file> <list_pct> <fp64 0|1> <ncomp>
#include "../../paper_1911_10228_gb300/csrc/flgf_api.cu"

#include <array>
#include <cstdio>
#include <map>
#include <set>

int main(int argc, char** argv) {
  if (argc != 5) return 2;
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
  std::vector<double> h0(np);
  for (int p = 0; p < np; ++p) h0[p] = 1.0 + (atoi(argv[4]) > 1 ? 0 : p);
  flgf_ctx ctx;
  ctx.N = N;
  ctx.prec = atoi(argv[3]) ? FLGF_FP64 : FLGF_FP32;
  ctx.max_oct = 8;
  ctx.list_pct = atoi(argv[2]);
  auto bs = new flgf_blockset();
  bs->ctx = &ctx;
  bs->ncomp = atoi(argv[4]);
  if (plan_blockset(&ctx, bs, np, nlev.data(), nblk.data(), coords.data(), h0.data()) != FLGF_OK) return 1;
  build_adjoint(bs);  // the lists are complete; its allocations fail without a GPU
  long bad = 0, parents = 0, blocks = 0, out_pairs = 0;
  auto check = [&](const PhaseOff& ph, const char* base, const std::vector<const Inst*>& insts) {
    auto I = [&](size_t off) { return reinterpret_cast<const int*>(base + off); };
    const bool coarse = ctx.parent_form_coarse();
    std::map<int, double> want;  // target of a level between parents -> scale
    std::map<int, std::pair<const Inst*, std::pair<size_t, size_t>>> where;  // column -> instance, level, index
    for (const Inst* in : insts)
      for (size_t k = 0; k < in->lv.size(); ++k)
        for (size_t i = 0; i < in->lv[k].size(); ++i) {
          if (in->need_tgt[k][i] && (k == 0 || coarse)) want[in->gid0[k] + (int)i] = in->h * in->h;
          where[in->gid0[k] + (int)i - ph.gid_begin] = {in, {k, i}};
        }
    std::map<int, int> written;
    auto wrote = [&](int gid, double scale) {
      bad += want.count(gid) == 0 || want[gid] != scale;
      written[gid]++;
    };
    const double* iscale = reinterpret_cast<const double*>(base + ph.inv_scale);
    const int n_assign = coarse ? ph.n_inv - ph.n_inv_add : ph.n_inv0;
    for (int i = 0; i < n_assign; ++i, ++blocks) wrote(I(ph.inv_gid)[i], iscale[i]);
    const double* pscale = reinterpret_cast<const double*>(base + ph.pf_scale);
    for (int i = 0; i < ph.n_pft; ++i, ++parents)
      for (int a = 0; a < 8; ++a)
        if (I(ph.pf_tch)[8 * i + a] >= 0) wrote(I(ph.pf_tch)[8 * i + a], pscale[i]);
    bad += written.size() != want.size();
    for (const auto& w : written) bad += w.second != 1;
    // the targets whose near pairs are taken out, each added to once
    std::set<int> added;
    for (int i = ph.n_inv - ph.n_inv_add; i < ph.n_inv; ++i) {
      const int gid = I(ph.inv_gid)[i];
      bad += !added.insert(gid - ph.gid_begin).second || want.count(gid) == 0 || iscale[i] != want[gid];
    }
    std::set<int> fwd(I(ph.fwd_sid), I(ph.fwd_sid) + ph.n_fwd);
    const uint32_t* qe = reinterpret_cast<const uint32_t*>(base + ph.fll_ent);
    const FllGroup* Q = reinterpret_cast<const FllGroup*>(base + ph.fll_groups);
    for (int g = 0; g < ph.n_fll; ++g)
      for (int m = 0; m < Q[g].ntgt; ++m)
        for (int j = 0; j < I(ph.fll_len)[Q[g].tgt_off + m]; ++j)
          bad += !fwd.count((int)(qe[I(ph.fll_beg)[Q[g].tgt_off + m] + j] >> 9));
    const ListGroup* LG = reinterpret_cast<const ListGroup*>(base + ph.groups);
    for (int g = 0; g < ph.n_groups + ph.n_groups_out; ++g)
      for (int i = 0; i < LG[g].nsrc; ++i) bad += !fwd.count(I(ph.l_src)[LG[g].src_off + i]);
    const FlGroup* G = reinterpret_cast<const FlGroup*>(base + ph.fl_groups);
    const uint16_t* rows = reinterpret_cast<const uint16_t*>(base + ph.fl_rows);
    const PfGroup* PG = reinterpret_cast<const PfGroup*>(base + ph.pf_groups);
    const uint16_t* items = reinterpret_cast<const uint16_t*>(base + ph.pf_items);
    for (int gi = 0; gi < ph.n_fl; ++gi) {
      const FlGroup& g = G[gi];
      bad += (gi < ph.n_pf) != (g.level == 0 || coarse);
      for (int c = 0; c < g.ncell; ++c)
        for (int b = 0; b < 8; ++b) {
          const int s = I(ph.fl_cells)[(g.cell_off + c) * 8 + b];
          if (gi >= ph.n_pf) { bad += s >= 0 && !fwd.count(s); continue; }
          for (int k = 0; k < ph.fl_ncomp; ++k)
            bad += I(ph.pf_sch)[8 * (I(ph.pf_ccol)[g.cell_off + c] + k * ph.pf_src_stride) + b] !=
                   (s < 0 ? -1 : s + k * ph.fl_cstride + ph.gid_begin);
        }
      if (gi >= ph.n_pf) continue;
      const PfGroup& pg = PG[gi];
      bad += pg.ncell != g.ncell || pg.nact != g.nact || pg.cell_off != g.cell_off || pg.row_off != g.row_off ||
             pg.level != g.level ||
             g.nact > ph.pf_lim.parents || g.ncell > ph.pf_lim.cells || pg.nitem > ph.pf_lim.items;
      std::vector<int> seen(g.nact, 0);
      bad += pg.nquad < 0 || 2 * pg.nquad > pg.nitem;
      for (int i = 0; i < pg.nquad; ++i) {  // quads: two pairs, the second one up along axis 1
        const uint16_t* it = items + (size_t)(pg.item_off + 2 * i) * kPfItem;
        for (int a = 0; a < 4; ++a) {
          const int m = it[48 + a / 2] + a % 2;
          if (m >= g.nact) { ++bad; continue; }
          seen[m]++;
          const uint16_t* row = rows + (size_t)(g.row_off + m) * kFlRowStride;
          int want_cell[27];
          std::fill(want_cell, want_cell + 27, g.ncell);
          for (int j = 0; j < row[0]; ++j) want_cell[row[1 + j] >> 11] = row[1 + j] & 0x7FF;
          for (int e = 0; e < 27; ++e) {
            bad += it[16 * (e / 9) + 4 * ((e / 3) % 3 + a / 2) + e % 3 + a % 2] != 33 * want_cell[e];
            bad += want_cell[e] != g.ncell && !((it[50] >> (e / 9)) & 1);
          }
        }
      }
      for (int i = 2 * pg.nquad; i < pg.nitem; ++i) {
        const uint16_t* it = items + (size_t)(pg.item_off + i) * kPfItem;
        if (it[37] < 1 || it[37] > 2 || it[36] + it[37] > g.nact) { ++bad; continue; }
        for (int p = 0; p < it[37]; ++p) {
          const int m = it[36] + p;
          seen[m]++;
          // the 27 cells that the kernel multiplies for the parent
          const uint16_t* row = rows + (size_t)(g.row_off + m) * kFlRowStride;
          int want_cell[27];
          std::fill(want_cell, want_cell + 27, g.ncell);
          for (int j = 0; j < row[0]; ++j) want_cell[row[1 + j] >> 11] = row[1 + j] & 0x7FF;
          for (int e = 0; e < 27; ++e) {
            if (g.level > 0 && e == 13) continue;  // zero kernel: siblings are near
            bad += it[9 * (e % 3 + p) + e / 3] != 33 * want_cell[e];
            bad += want_cell[e] != g.ncell && !((it[38] >> (e / 9)) & 1);
          }
        }
      }
      for (int m = 0; m < g.nact; ++m) {
        bad += seen[m] != 1;
        for (int k = 0; k < ph.fl_ncomp; ++k)
          for (int a = 0; a < 8; ++a) {
            const int t = I(ph.fl_tgt)[(g.row_off + m) * 8 + a];
            bad += I(ph.pf_tch)[8 * (I(ph.pf_tcol)[g.row_off + m] + k * ph.pf_tgt_stride) + a] !=
                   (t < 0 ? -1 : t + k * ph.fl_cstride + ph.gid_begin);
          }
      }
    }
    // every (target, source) pair of the products between parents of a coarser
    // level that does not interact (near) is in the lists that take pairs out, once
    std::map<std::array<int, 3>, int> extra;
    for (int gi = 0; gi < ph.n_pf; ++gi) {
      const FlGroup& g = G[gi];
      if (g.level == 0) continue;
      for (int m = 0; m < g.nact; ++m) {
        const uint16_t* row = rows + (size_t)(g.row_off + m) * kFlRowStride;
        for (int j = 0; j < row[0]; ++j)
          for (int a = 0; a < 8; ++a)
            for (int b = 0; b < 8; ++b) {
              const int t = I(ph.fl_tgt)[(g.row_off + m) * 8 + a], s = I(ph.fl_cells)[(g.cell_off + (row[1 + j] & 0x7FF)) * 8 + b];
              if (t < 0 || s < 0) continue;
              const auto &tw = where.at(t), &sw = where.at(s);
              bad += tw.first != sw.first || tw.second.first != sw.second.first || (int)tw.second.first != g.level;
              const I3 &tc = tw.first->lv[g.level][tw.second.second], &sc = sw.first->lv[g.level][sw.second.second];
              if (std::abs(tc[0] - sc[0]) > 1 || std::abs(tc[1] - sc[1]) > 1 || std::abs(tc[2] - sc[2]) > 1) continue;
              extra[{t, s, off_index(tc[0] - sc[0], tc[1] - sc[1], tc[2] - sc[2])}]++;
            }
      }
    }
    std::set<int> listed;
    const int* le = I(ph.l_ent);
    for (int g = ph.n_groups; g < ph.n_groups + ph.n_groups_out; ++g)
      for (int m = 0; m < LG[g].ntgt; ++m) {
        const int t = I(ph.l_tgt)[LG[g].tgt_off + m];
        listed.insert(t);
        bad += where.at(t).second.first != (size_t)LG[g].level;
        for (int j = 0; j < I(ph.l_len)[LG[g].len_off + m]; ++j) {
          const int w = le[LG[g].ent_off + j * kListTargets + m];
          if (--extra[{t, I(ph.l_src)[LG[g].src_off + (w >> 9)], w & 511}] != 0) ++bad;
        }
      }
    for (const auto& x : extra) bad += x.second != 0;
    bad += listed != added;
    out_pairs += (long)extra.size();
  };
  for (int adj = 0; adj < 2; ++adj)
    for (int l = 0; l < bs->Lmax; ++l) {
      std::vector<const Inst*> insts;
      for (const Inst& in : bs->inst)
        if (in.l == l && (!adj || in.variant == 0)) insts.push_back(&in);
      if (adj)
        for (const Inst& in : bs->adj_inst)
          if (in.l == l) insts.push_back(&in);
      check(adj ? bs->aph[l] : bs->ph[l], adj ? bs->aar.host.data() : bs->ar.host.data(), insts);
    }
  printf("parents %ld blocks %ld near pairs %ld mismatches %ld\n%s\n", parents, blocks, out_pairs, bad, bad ? "FAILED" : "ok");
  return bad ? 1 : 0;
}
