// Decode-and-aggregate, Elias path, optionally fused with the SGD step (Section 3.1, end of
// "Efficient Coding of Gradients": scale first, then the codes of the nonzeros in index order;
// Appendix A.2 decoder; Algorithm 1 for the sum and the step): the choice among the decoders. The one that
// reads streams of consecutive strings by table is in elias_decode_ring.cu (s <= 15) and, for the dense code,
// elias_decode_dense.cu, the ones with a lane per
// string in elias_decode_bytes.cu (s <= 15) and elias_decode_fields.cu (larger s), the one with a team of lanes per string
// in elias_decode_teams.cu, the nonzero-driven decoder of the sparse regime in elias_decode_sparse.cu; what they
// share is in elias_decode.cuh.
#include "elias_decode.cuh"

namespace qsgd {

namespace {

// Coordinates x peers up to which the sparse-regime decoder is not launched beside the teams (one launch less, and a
// string's latency decides: n = 2^20, d = 4096, s = 1, K = 8 in the packed form 15.5 against 27.3 us; at 2^22 41.0 against
// 33.9), and has to itself only what sparse_though_small gives it.
constexpr uint64_t kSmallWork = 8ull << 20;

// Strings of a small problem that are known to be short, `mean` bits behind the scale: a lane reads one as fast as a team
// does, and the sums of a bucket are spread over the warps better. 482 such problems measured, sparse-regime decoder
// against teams: up to 300 bits, with at most 8 peers or more than 2 M coordinates x peers, 0.42 to 1.36 of the time
// (n = 54 K, d = 1024, s = 1, K = 4 8.0 / 12.3 us); the others 0.68 to 2.7 (n = 57 K, d = 1024, s = 1, K = 17 10.4 / 9.1).
bool sparse_though_small(uint32_t mean, uint32_t K, uint64_t work) { return mean < 300u && (K <= 8u || work > (2ull << 20)); }

// A lane per string (or stream of strings), or a team of lanes? A lane per string is the cheaper reading (a team
// reads its string almost twice) but needs strings enough for the GPU's lanes, and room in shared memory for the whole
// bucket where s > 15. Measured (us, a team against a lane). s <= 15: 20 K strings of d = 128 27 / 29, 23 K of d = 512
// 32 / 38, 23 K of d = 4096 93 / 125; 39 K of d = 512 36 / 37, of d = 128 39 / 30, 62 K of d = 512 48 / 40. s = 255:
// 13 K of d = 96 31 / 34, 16 K of d = 256 50 / 83; 26 K of d = 96 37 / 34, 31 K of d = 64 29 / 24, of d = 256 89 / 87,
// 524 K of d = 256 1042 / 664; from d = 512 on always teams: 16 K 82 / 149, 262 K 912 / 937, d = 1024 915 / 1632. Code'_s
// has a symbol per coordinate: teams, or streams (use_streams).
bool use_teams(uint64_t B, uint32_t K, uint32_t d, uint32_t s) {
  return (s > 15u && d >= 512u) || B * K <= (24u << 10);
}

// Code'_s: a lane per stream, or teams, which read a string several times but with all lanes of the GPU? 60 problems measured
// both ways; strings, and us by streams / by teams. K >= 8: 16 K 169 / 157 (d = 4096, s = 64), 40 / 38 (d = 512, s = 22), 28 / 24
// (d = 64, s = 15); 24 K 179 / 218, 40 / 48, 26 / 26; 64 K 243 / 544, 48 / 93, 26 / 36. Fewer peers, whose sums the teams spread
// better: K = 4 24 K 212 / 173, 32 K 216 / 222, 64 K 265 / 427; K = 2 24 K 38 / 34, 32 K 38 / 42; K = 1 32 K 151 / 126, 64 K
// 177 / 218. Symbols of levels above 15, which the streams' table seldom holds, only where the bucket's largest level is likely
// far above the others: max-norm, n = 17 M, K = 8: d = 512, s = 64 552 / 751, d = 4096 705 / 700, but d = 128 633 / 570, d = 64,
// s = 48 627 / 574; d = 128, s = 100 718 / 599.
// Few levels in short buckets, where opening a bucket is most of a stream's work (5200 problems; speed of streams over that of
// teams): s <= 7, d = 32 0.74 to 0.99 up to 400 K strings, 1.06 to 1.27 beyond, with one or two peers 0.74 to 1.03 at any number;
// s <= 3, d = 64 and 96 1.1 to 1.3 up to 80 K, 0.93 to 1.02 from there to 256 K, 1.05 to 1.2 beyond, with one or two peers 0.84 to
// 1.1; s <= 3 and one peer with d = 128 to 192 0.94 to 0.99 from 100 K to 512 K, with longer ones about 1 from 64 K to 256 K.
bool use_streams(uint64_t B, uint32_t K, uint32_t d, uint32_t s) {
  if (K > 32u || s > (d >= 512u ? 64u : 32u)) return false;
  const uint64_t strings = B * K;
  uint32_t line = K == 1u ? 48u : K < 8u ? 30u : 22u, from = 0, to = 0;       // in 1024 strings; from .. to: teams all the same
  if (s <= 7u && d < 64u) {
    if (K <= 2u) return false;
    line = 400u;
  } else if (s <= 3u && d < 128u) {
    from = K == 1u ? 100u : K == 2u ? 64u : 80u;
    to = K <= 2u ? ~0u : 256u;
  } else if (s <= 3u && K == 1u) {
    from = d < 256u ? 100u : 64u;
    to = d < 256u ? 512u : 256u;
  }
  return strings > (uint64_t)line << 10 && (strings <= (uint64_t)from << 10 || strings > (uint64_t)to << 10);
}

// Mean bits of a string behind its scale, where the host can tell: in a message the offset table follows the padded
// payload, so table - payload is the payload size. kNoBound: it cannot.
uint32_t mean_bits(const PeerSet& peers, uint32_t K, uint64_t B, uint64_t n) {
  if (peers.packed) return kNoBound;
  uint64_t bits = 0;
  for (uint32_t k = 0; k < K; ++k) {
    const uint8_t* w = reinterpret_cast<const uint8_t*>(peers.payload[k]);
    const uint8_t* t = reinterpret_cast<const uint8_t*>(peers.table[k]);
    const uint64_t longest = align16((B * 32ull + n * 40ull + 7ull) / 8ull);   // no legal payload is longer
    if (t <= w || (uint64_t)(t - w) > longest) return kNoBound;
    bits += 8ull * (uint64_t)(t - w);
  }
  const uint64_t mean = bits / ((uint64_t)K * B);
  return mean > 32u ? (uint32_t)(mean - 32u) : 0u;
}

// Below this many bits per string, a quarter of a bit per coordinate, the sparse-regime decoder: an entry of a sparse
// bucket costs 11 to 14 bits, so a list with room for one entry per 32 positions then fills to about 60 % on average
// and rarely overflows.
uint32_t sparse_line(uint32_t d) { return d / 4u; }

// A lane per string, s <= 15: bytes or ring? The ring's tables and rings cost 10 us to set up, and a round per 128
// positions reads little where strings are short; where they are long, or peers many, it is up to twice as fast. 3700
// problems of more than 22 K strings measured; the time by ring over that by bytes, means for the coordinates x peers (work)
// and bits per coordinate behind the scale: d <= 48 1.1 to 2.4 up to 4 M, up to 12 M 0.9 to 1.6 with 8 peers and fewer but
// 0.63 to 1.03 with more, beyond 1.04 to 1.55 with 1 or 2 and less than 1 with more; d = 64 and 96 1.0 to 2.0 up to 4 M, 0.91 to
// 1.8 up to 12 M with 16 peers and fewer; d = 97 to 200 up to 12 M 1.1 to 1.7 below 1.5 bits, 0.68 to 0.96 above.
// (n = 266 K, d = 32, s = 1, K = 4 6.5 / 15.3 us; n = 3 M, d = 96, s = 15, K = 4 24 / 28.)
bool use_bytes(uint32_t K, uint32_t d, uint32_t s, uint64_t work) {
  if (d <= 48u) return K <= 2u || work <= (K <= 8u ? 6ull << 20 : 4ull << 20);
  if (d <= 96u) return work <= (K <= 16u ? 12ull << 20 : 4ull << 20);
  return d <= 200u && work <= (s <= 3u ? 12ull << 20 : 4ull << 20);       // (few levels: strings are likely short)
}
// For other problems, below how many bits per string by bytes: 1.0 to 1.5 there, 0.5 to 1.05 above (n = 16.8 M, d = 256,
// s = 3, K = 16, half a bit per coordinate 120 / 136 us).
uint32_t bytes_line(uint32_t K, uint32_t d, uint64_t work) {
  if (d <= 48u || d >= 1024u) return 0u;
  if (d <= 96u) return K <= 2u ? 7u * d / 4u : K <= 4u ? 7u * d / 8u : K <= 16u ? 5u * d / 8u : 0u;
  if (d <= 300u && work <= (12ull << 20)) return 11u * d / 8u;
  if (d <= 300u) return K <= 16u || d > 200u ? 3u * d / 4u : d / 2u;
  return K > 8u ? d / 2u : 0u;
}

}  // namespace

int launch_decode_elias(const PeerSet& peers, uint32_t K, uint64_t n, uint32_t d, uint32_t s,
                        bool dense, float* acc_or_x, bool fused, float eta, uint32_t* status_dev,
                        const BucketMap& map, cudaStream_t stream) {
  const uint64_t B = (n + d - 1) / d, work = n * K;
  FieldParams f;
  f.peers = peers; f.K = K; f.n = n; f.d = d; f.s = s; f.B = B;
  f.out = acc_or_x; f.c = eta / (float)K; f.minus_zero = -0.f; f.status = status_dev; f.map = map;
  f.when = Regime{0u, kNoBound};
  if (dense && use_streams(B, K, d, s)) return launch_elias_dense(f, fused, stream);
  const uint32_t mean = mean_bits(peers, K, B, n);
  if (dense || K > 32u) return launch_elias_teams(f, dense, mean, fused, stream);

  const bool teams = use_teams(B, K, d, s), small = teams && work <= kSmallWork;
  if (mean != kNoBound) {
    if (mean < sparse_line(d) && (!small || sparse_though_small(mean, K, work))) return launch_elias_sparse(f, fused, stream);
  } else if (!small) {                            // decided on the device: both are launched, one stands down
    f.when = Regime{0u, sparse_line(d)};
    const int st = launch_elias_sparse(f, fused, stream);
    if (st) return st;
    f.when = Regime{sparse_line(d), kNoBound};
  }
  if (teams) return launch_elias_teams(f, false, mean, fused, stream);
  if (s > 15u) return launch_elias_fields(f, fused, stream);
  const uint32_t line = bytes_line(K, d, work);
  const bool likely = use_bytes(K, d, s, work) && (d <= 96u || mean == kNoBound);
  if (likely || mean < line) return launch_elias_bytes(f, fused, stream);
  // Few levels, buckets of about 256 and time enough: strings short enough for the bytes are likely enough, and enough is
  // gained, for a third launch (2 to 4 us where it is not the one).
  if (mean == kNoBound && s <= 3u && d > 200u && d <= 300u && work > (64ull << 20)) {
    f.when.hi = line;
    const int st = launch_elias_bytes(f, fused, stream);
    if (st) return st;
    f.when = Regime{line, kNoBound};
  }
  return launch_elias_ring(f, fused, stream);
}

}  // namespace qsgd
