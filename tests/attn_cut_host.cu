// The flat list of an attention kernel walked on the host, as its thread blocks walk it: one compilation unit per kernel
// (-DKERNEL_ROWS: csrc/attn_rows.cu, else csrc/attn_tc.cu), no GPU.
#ifdef KERNEL_ROWS
#include "../paper_2402_11809_b200/csrc/attn_rows.cu"
#else
#include "../paper_2402_11809_b200/csrc/attn_tc.cu"
#endif

// Pieces of all groups in order: {group, sequence, head, tiles, tiles of the pair, cut.x, cut.y} in out[7 * i]; returns how
// many.  prefix: entries of the list before each sequence, and in all.
extern "C" int host_list_pieces(const int* seq_len, int* prefix, int B, int H_kv, int n_q, int n_groups, int* out) {
  prefix[0] = 0;
  for (int b = 0; b < B; ++b) {
    const int T = seq_len[b] < 0 ? 0 : (seq_len[b] + n_q + TILE_N - 1) / TILE_N;
    prefix[b + 1] = prefix[b] + (T ? (T + SHARE_COST) * H_kv : 0);
  }
  int n = 0;
  for (int g = 0; g < n_groups; ++g) {
    Partition part;
    Seg sg;
#ifdef KERNEL_ROWS
    part.init(seq_len, prefix, B, H_kv, n_q, g, n_groups);
#else
    part.init(seq_len, prefix, -1, nullptr, B, H_kv, n_q, g, n_groups);
#endif
    while (part.next(sg)) {
#ifdef KERNEL_ROWS
      const int2 c = share_cut(prefix, B, n_groups, sg, g);
#else
      const int2 c = share_cut(prefix, B, H_kv, n_groups, sg);
#endif
      const int v[7] = {g, sg.b, sg.h, sg.n, sg.T, c.x, c.y};
      for (int x : v) *out++ = x;
      ++n;
    }
  }
  return n;
}
