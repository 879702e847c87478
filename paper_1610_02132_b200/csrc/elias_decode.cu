// Decode-and-aggregate, Elias path, optionally fused with the SGD step (Section 3.1, end of
// "Efficient Coding of Gradients": scale first, then the codes of the nonzeros in index order;
// Appendix A.2 decoder; Algorithm 1 for the sum and the step): the choice among the decoders. The one that
// reads streams of consecutive strings by table is in elias_decode_ring.cu (s <= 15), the one with a lane per
// string for larger s in elias_decode_fields.cu, the one with a team of lanes per string in
// elias_decode_teams.cu, the nonzero-driven decoder of the sparse regime in elias_decode_sparse.cu; what they
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
bool sparse_though_small(uint64_t mean, uint32_t K, uint64_t work) { return mean < 300u && (K <= 8u || work > (2ull << 20)); }

// A lane per string (or stream of strings), or a team of lanes? A lane per string is the cheaper reading (a team
// reads its string almost twice) but needs strings enough for the GPU's lanes, and room in shared memory for the whole
// bucket where s > 15. Measured (us, a team against a lane). s <= 15: 20 K strings of d = 128 27 / 29, 23 K of d = 512
// 32 / 38, 23 K of d = 4096 93 / 125; 39 K of d = 512 36 / 37, of d = 128 39 / 30, 62 K of d = 512 48 / 40. s = 255:
// 13 K of d = 96 31 / 34, 16 K of d = 256 50 / 83; 26 K of d = 96 37 / 34, 31 K of d = 64 29 / 24, of d = 256 89 / 87,
// 524 K of d = 256 1042 / 664; from d = 512 on always teams: 16 K 82 / 149, 262 K 912 / 937, d = 1024 915 / 1632. Code'_s
// has a symbol per coordinate: always teams.
bool use_teams(uint64_t B, uint32_t K, uint32_t d, uint32_t s, bool dense) {
  return dense || K > 32u || (s > 15u && d >= 512u) || B * K <= (24u << 10);
}

}  // namespace

int launch_decode_elias(const PeerSet& peers, uint32_t K, uint64_t n, uint32_t d, uint32_t s,
                        bool dense, float* acc_or_x, bool fused, float eta, uint32_t* status_dev,
                        const BucketMap& map, cudaStream_t stream) {
  // Which decoder? In a message the offset table follows the padded payload, so table - payload is
  // the payload size and the host can evaluate the regime predicate itself (to within the padding)
  // and launch one kernel. With tables kept elsewhere the sizes are only known on the device: both
  // kernels are launched and exactly one does the work. Either decoder is correct on any input;
  // the choice is about speed only.
  const uint64_t B = (n + d - 1) / d;
  bool sizes_known = !dense && K <= 32u && !peers.packed;
  uint64_t payload_bits = 0;
  for (uint32_t k = 0; k < K && sizes_known; ++k) {
    const uint8_t* w = reinterpret_cast<const uint8_t*>(peers.payload[k]);
    const uint8_t* t = reinterpret_cast<const uint8_t*>(peers.table[k]);
    const uint64_t longest = align16((B * 32ull + n * 40ull + 7ull) / 8ull);   // no legal payload is longer
    if (t <= w || (uint64_t)(t - w) > longest) sizes_known = false;
    else payload_bits += 8ull * (uint64_t)(t - w);
  }
  const bool host_sparse = sizes_known && payload_bits < (uint64_t)K * B * (32ull + d / 4u);
  FieldParams f;
  f.peers = peers; f.K = K; f.n = n; f.d = d; f.s = s; f.B = B;
  f.out = acc_or_x; f.c = eta / (float)K; f.minus_zero = -0.f; f.status = status_dev; f.map = map;
  const bool teams = use_teams(B, K, d, s, dense);
  const bool small = teams && n * K <= kSmallWork;
  bool sparse = false;
  if (!dense && (host_sparse ? !small || sparse_though_small(payload_bits / (K * B) - 32u, K, n * K) : !sizes_known && !small)) {
    const int st = launch_elias_sparse(peers, K, n, d, s, acc_or_x, fused, f.c, status_dev, !sizes_known, map, stream, &sparse);
    if (st) return st;
    if (sparse && sizes_known) return 0;                    // the host chose the sparse-regime kernel
  }
  f.defer_sparse = sparse ? 1u : 0u;
  if (teams) return launch_elias_teams(f, dense, fused, stream);
  return s <= 15u ? launch_elias_ring(f, fused, stream) : launch_elias_fields(f, fused, stream);
}

}  // namespace qsgd
