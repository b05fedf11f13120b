// Prints the split over the SMs of batches read from standard input, one per line: L Hkv group d m key-bytes n_tokens...; called with
// an argument, the form of their prompts: 2 resident with the maxima in registers, 1 resident, 0 two-pass.
// Includes the host side of the fused path as it is; nothing of it runs on a device.
#include <iostream>
#include <sstream>
#include <vector>

#include "score_fused.cu"

namespace spf {
int32_t fail(int32_t code, const char*, ...) { return code; }
int32_t fused_launch_d64(const FusedArgs&, const FusedLaunch&, cudaStream_t) { return 0; }
int32_t fused_launch_d128(const FusedArgs&, const FusedLaunch&, cudaStream_t) { return 0; }
int32_t fused_launch_d64_fp8(const FusedArgs&, const FusedLaunch&, cudaStream_t) { return 0; }
int32_t fused_launch_d128_fp8(const FusedArgs&, const FusedLaunch&, cudaStream_t) { return 0; }
}  // namespace spf

using namespace spf;

int main(int argc, char**) {
  constexpr int kSms = 148;
  for (std::string line; std::getline(std::cin, line);) {
    std::istringstream in(line);
    ScoreProblem p{};
    int key_bytes;
    in >> p.n_layers >> p.n_kv_heads >> p.group >> p.head_dim >> p.n_lookahead >> key_bytes;
    p.n_q_heads = p.n_kv_heads * p.group;
    p.k_scale = key_bytes == 1 ? reinterpret_cast<const float*>(4096) : nullptr;
    std::vector<Geometry> g;
    std::vector<int64_t> tiles;
    bool same = true;
    while (in >> p.n_tokens) {
      p.stride_tok = p.head_dim;
      p.stride_head = p.n_tokens * p.head_dim;
      const Geometry gi = geometry(p, kSms);
      same = same && gi.ok && (tiles.empty() || gi.once == g[0].once);
      g.push_back(gi);
      tiles.push_back(ceil_div(p.n_tokens, kTileKeys));
    }
    if (argc > 1) {
      for (size_t i = 0; i < g.size(); ++i)
        std::cout << (g[i].ok ? (int)g[i].once + (int)(g[i].once && g[i].max_in_regs((int)ceil_div(tiles[i], kSms))) : -1) << ' ';
      std::cout << '\n';
      continue;
    }
    // which prompts share the first launch, and the CTAs of each: groups, CTAs per group, tiles per CTA
    const int n = same ? group_size(g.data(), tiles.data(), (int)tiles.size(), kSms) : 0;
    Split split[kFusedMaxBatch];
    const bool ok = n > 0 && split_group(g.data(), tiles.data(), n, kSms, split);
    std::cout << same << ' ' << n << ' ' << ok;
    for (int i = 0; ok && i < n; ++i) std::cout << ' ' << split[i].parts << ' ' << split[i].per_part << ' ' << split[i].tiles;
    std::cout << '\n';
  }
}
