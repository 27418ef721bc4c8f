// How the tree convolution is cut into CTAs and warps: host arithmetic, no CUDA in here.
#pragma once

namespace lumo {

constexpr int kConvWarps = 8;
constexpr int kConvMaxEntries = 128;      // entries per CTA: eight runs of sixteen

// Runs and channel groups of a CTA (a warp per pair): groups is a power of two.
struct ConvSplit { int runs, groups, log_groups, slabs; };
inline ConvSplit conv_split(int C, int Ns, int run, int seqs, int sms) {
  const int need = (Ns + run - 1) / run, parts = (need + kConvWarps - 1) / kConvWarps, even = (need + parts - 1) / parts;
  ConvSplit c;
  c.runs = need < kConvWarps ? need : kConvWarps;
  // Eleven runs are eight and three, and the second CTA's idle warps help to load: fastest while all CTAs run at once.  Where
  // they do not (more than four per SM), idle warps hold places: an even share of at most six runs lets five CTAs or more onto
  // an SM.  4096 channels, runs of four, convolution and scan together: 12 sequences of 41 entries (768 CTAs), fused, 27.0 ->
  // 26.1 us, 11 of 46 26.2 -> 24.9; 32 of 140 in runs of sixteen 213 -> 206 us.  Below the line the even share loses (4
  // sequences of 46, 256 CTAs: 18.5 -> 18.9 us), and of seven runs no more CTAs fit (32 x 200 entries: 136.0 -> 136.7 us).
  if (need > kConvWarps && even <= 6 && (long long)((C + 127) / 128) * parts * seqs > 4LL * sms) c.runs = even;
  c.log_groups = c.runs == 1 ? 3 : c.runs == 2 ? 2 : c.runs <= 4 ? 1 : 0;
  c.groups = 1 << c.log_groups;
  c.slabs = (C + c.groups * 128 - 1) / (c.groups * 128);
  return c;
}

}  // namespace lumo
