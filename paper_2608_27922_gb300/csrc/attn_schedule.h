// Which schedule a tensor-core attention call takes, from sizes alone: estimates shared by
// the launcher (which knows the budgets) and the share kernel (which reads the occupancies).
// Both inputs belong to the handle and its bank, so that a call's rounding does not depend on
// how the bank came to its contents, nor on whether the call is captured in a graph.
//
// A unit is one 128-query tile of one head with all of that head's key tiles (128 keys each,
// bank then window; at least one).  Estimates are in key tiles of one unit, 0.775 us each on
// an SM that has work (12 full heads on 152 SMs at 2,070 MHz):
//   whole units, one CTA each:   every wave lasts a unit; a lone wave its longest unit
//   equal shares of key tiles:   all SMs busy to the end; one more segment a CTA (C0 tiles of
//                                fixed cost each), and the store and merge of the cut units' parts
//   two query tiles per CTA:     0.92 of the time per unit (K and V cross from L2 once for
//                                both), waves of two units
// The constants are measured on that part, like the costs they stand for; another part would
// want its own.  Both sides of the lines, us (whole units | shares | two tiles), 9,360 + 4,680
// keys: 12 heads x 4,680 queries 249 | 264 | -; x 1,560 170 | 112 | -; x 256 95 | 37 | -; 16
// heads x 4,680 - | 341 | 315; 17 heads - | 406 | 460; 7 heads x 1,846 queries x 5,903 keys 40 |
// 47 | - (short bursts).
#pragma once

#ifdef __CUDACC__
#define DKV_HD __host__ __device__ __forceinline__
#else
#define DKV_HD inline
#endif

namespace dkv {
namespace attn {

// A share is at least SPLIT_MIN tiles (or there is one per unit): below that a part's fixed
// cost (query tile, first scores, partial store, about 6 us) outweighs its tiles (about 1 us
// for two).  Units of fewer than SPLIT_UNIT tiles are not cut (a boundary inside one moves to
// its start): they are short by themselves.
constexpr int SPLIT_MIN = 4;
constexpr int SPLIT_UNIT = 16;
constexpr int SPLIT_CTAS = 152;      // most shares (the SMs of the GPU): sizes the scratch
constexpr int SHARE_UNITS = 1024;    // fewer units than this are cut in shares: tile numbers of the range
                                     //   stay in an int for any bank and window.  Above, at 6.7 units per SM and
                                     //   more, little is left to gain (us, two tiles per CTA | shares: 1 head x
                                     //   262,144 queries x 9,360 keys 800 | 821, 2 x 80,000 x 18,720 978 | 961)
constexpr float C0 = 6.f;            // fixed cost of a unit or segment
constexpr float MERGE = 23.f;        // store and merge of the parts
// HBM_UNITS units' tiles of keys and values take HBM one tile's time (6.5 TB/s).  Whole units
// in order keep the query tiles of one head side by side, which read its keys once; shares walk
// all heads at once, so where the keys and values of all heads are more than SHARED_BYTES every
// unit reads its own from HBM (whole units | shares, us: 123 heads x 182 queries x 15,832 keys
// 212 | 301, 40 x 1,560 x 14,040 326 | 507; one query tile a head: 160 x 128 x 14,040 232 | 189).
// SHARED_BYTES lies between two measured points, above the L2's 126 MB since some is reused
// beyond it: 24 x 1,560 x 14,040, 173 MB, 242 | 206; 40 heads, 288 MB, above.
constexpr float HBM_UNITS = 77.f;
constexpr float SHARED_BYTES = 180e6f;
constexpr float TILE_BYTES = 2.f * 128 * 128 * 2;   // 128 keys and their values, bf16

// One call: heads, query tiles (128) per head, tiles of a unit on average and of the longest.
struct Sizes {
  int heads, nqt;
  float nt, longest;
};

DKV_HD float larger(float a, float b) { return a > b ? a : b; }
DKV_HD float wave_count(float units, int ctas) { return (float)(((int)units + ctas - 1) / ctas); }

DKV_HD float est_whole(const Sizes& z, int ctas) {
  const float waves = wave_count((float)z.heads * z.nqt, ctas);
  // heads read by a full wave of units, and by the last one
  const float in_wave = (float)ctas / z.nqt, in_last = z.heads - (waves - 1.f) * in_wave;
  const float t = (waves - 1.f) * z.nt * larger(1.f, in_wave / HBM_UNITS) + z.nt * larger(1.f, in_last / HBM_UNITS);
  return larger(z.longest, t) + waves * C0;
}

DKV_HD float est_shares(const Sizes& z, int ctas) {
  const float units = (float)z.heads * z.nqt, per = units / ctas, t = per * z.nt;
  const float e = larger(t, (float)SPLIT_MIN) + (per + 1.f) * C0 + MERGE;
  return TILE_BYTES * z.heads * z.nt > SHARED_BYTES ? larger(e, units * z.nt / HBM_UNITS + 2.f * C0 + MERGE) : e;
}

// Whether shares pay: the share kernel asks this of the occupancies, and walks whole units
// (CTA i units i, i + G, ..) where they do not.
DKV_HD bool shares_pay(const Sizes& z, int ctas) {
  return z.longest >= (float)SPLIT_UNIT && est_shares(z, ctas) < est_whole(z, ctas);
}

enum Schedule { WHOLE = 0, SHARES = 1, TWO = 2 };

// The launcher's choice for banks filled to their budgets.  scratch: the handle has room for
// the parts.
DKV_HD Schedule schedule(const Sizes& z, int nq, int n_sm, bool scratch) {
  const int ctas = n_sm < SPLIT_CTAS ? n_sm : SPLIT_CTAS;
  const float two = (float)((nq + 255) / 256) * z.heads;
  const bool cut = scratch && (float)z.heads * z.nqt < (float)SHARE_UNITS && shares_pay(z, ctas);
  const float least = cut ? est_shares(z, ctas) : est_whole(z, n_sm);
  if (two >= 2.f * n_sm && wave_count(two, n_sm) * (1.84f * z.nt + C0) <= least) return TWO;
  return cut ? SHARES : WHOLE;
}

}  // namespace attn
}  // namespace dkv
