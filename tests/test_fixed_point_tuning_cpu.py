"""The slab that the pass-B tuner times the fixed-point passes on (fx::slab_value of csrc/fx64.cuh),
compiled for the host: like production data and unlike zeros, it goes through the y transform's two
stages, pruned and full, without a stage that finds its input outside its range and shifts it."""
from tests.test_fixed_point_scales_cpu import HOST, run

SRC = HOST + r"""
template <int A, int B, int CW>
int shifts(bool zeros) {
  constexpr unsigned MW = fftr::edge_mask<A, CW>();  // (the inputs outside it are zero)
  constexpr int N = A * B, kWin = fx::kLimit(fftr::popc(MW)), kLoad = kWin - 1, W3 = N / 2 - 1;
  static fx::Cx Q[W3][N];
  long long n = 0;
  // as fx_inverse loads them: the plane's size brought to kLoad, zeros outside the window
  const int E = (zeros ? -1000 : 0) + fx::kSlabBits - kLoad, rs = zeros ? -1000 : 0;
  for (int u = 0; u < W3; ++u)
    for (int y = 0; y < N; ++y) {
      const bool in = CW == 0 || y < B * CW || y >= N - B * CW;
      const long long a = zeros ? 0 : fx::slab_value(n), b = zeros ? 0 : fx::slab_value(n + 1);
      n += 2;
      Q[u][y] = in ? fx::Cx{fx::scale2(a, E - rs), fx::scale2(b, E - rs)} : fx::Cx{0, 0};
    }
  fx::Mag m1, m2;
  for (int u = 0; u < W3; ++u)
    for (int r = 0; r < B; ++r) {
      fx::Cx v[A];
      for (int i = 0; i < A; ++i) v[i] = Q[u][r + B * i];
      fftr::rdft<A>(v, 1);
      v[0] = fx::Cx{fx::shr_round(v[0].x, 2), fx::shr_round(v[0].y, 2)};
      for (int k = 1; k < A; ++k)
        v[k] = fx::rot_small<true>(v[k], fx::rot_limbs(fx::kcos62(r * k, N), -fx::ksin62(r * k, N)));
      for (int k = 0; k < A; ++k) {
        m1.see(v[k]);
        Q[u][r + B * k] = v[k];
      }
    }
  int s = fx::fit(fx::mag_bits(m1.acc), fx::kLimit(B)) != 0;
  for (int u = 0; u < W3; ++u)
    for (int k = 0; k < A; ++k) {
      fx::Cx v[B];
      for (int j = 0; j < B; ++j) v[j] = Q[u][B * k + j];
      fftr::rdft<B>(v, 1);
      for (int j = 0; j < B; ++j) m2.see(v[j]);
    }
  return s + (fx::fit(fx::mag_bits(m2.acc), kWin) > 0);
}
template <int A, int B> void both(bool zeros, int& s) {
  s += shifts<A, B, 0>(zeros);
  if constexpr (2 * ((A + 3) / 4) < A) s += shifts<A, B, (A + 3) / 4>(zeros);
}
int main() {
  int s[2] = {0, 0};
  for (int z = 0; z < 2; ++z) {
    both<4, 6>(z, s[z]);
    both<5, 6>(z, s[z]);
    both<6, 6>(z, s[z]);
    both<8, 5>(z, s[z]);
    both<9, 6>(z, s[z]);
    both<12, 5>(z, s[z]);
    both<8, 12>(z, s[z]);
    both<12, 8>(z, s[z]);
  }
  printf("%d %d\n", s[0], s[1]);
}
"""


def test_tuning_slab_needs_no_shift(tmp_path):
    slab, zeros = map(int, run(tmp_path, SRC))
    assert zeros > 0   # (what made zeros unfit)
    assert slab == 0
