"""The reduction of a split product's FP32 slices into FP64 (the Gram matrix): the sum in three
floats against the exact one, and the FP64 sum that takes its place where the FP32 range does not
hold the slices' sum, or a part of it. On the CPU, from the kernel's source.

Tolerance: of 40 slices, each addition drops at most 2^-24 of the third float, which is at most
2^-46 of the running magnitude: 40 * 2^-70 of the sum of magnitudes, plus the rounding to FP64."""
import cuda_on_host


def test_three_float_sums(tmp_path):
    cuda_on_host.run(tmp_path, [("gemm_simt.cu", n) for n in
                                ("sum_slices", "two_sum32", "sum_slices_exact", "k_splitk_reduce")], r"""
static double uniform() { return std::rand() / (RAND_MAX + 1.0); }
int main() {
  const int splits = 40, M = 5, N = 7, total = M * N;
  const float inf = INFINITY, big = 3e38f;
  std::vector<float> part(splits * total);
  std::vector<double> out(M * 8, -9.0);
  for (int e = 0; e < total; ++e)
    for (int z = 0; z < splits; ++z) {
      const double scale = e < 14 ? 1.0 : std::exp2(40.0 * uniform() - 20.0);
      part[z * total + e] = (float)((2.0 * uniform() - 1.0) * scale);
    }
  for (int z = 0; z < splits; ++z) {   // element 0 .. 4 of the last row
    const int e = total - 7;
    part[z * total + e] = big;                                      // past FLT_MAX
    part[z * total + e + 1] = z == 0 || z == 1 ? big : z < 4 ? -big : 1.f;  // on the way only
    part[z * total + e + 2] = z == 17 ? inf : 1.f;
    part[z * total + e + 3] = z == 17 ? inf : z == 30 ? -inf : 1.f;
    part[z * total + e + 4] = z == 39 ? NAN : 1.f;
  }
  launch({2}, {32}, [&] {
    k_splitk_reduce<float, double>(part.data(), splits, M, N, total, out.data(), 8, true);
  });
  for (int e = 0; e < total; ++e) {
    const double got = out[e / N * 8 + e % N];
    long double sum = 0, mag = 0;
    for (int z = 0; z < splits; ++z) {
      sum += part[z * total + e];
      mag += std::fabs((long double)part[z * total + e]);
    }
    const int special = e - (total - 7);
    if (special == 2) CHECK(got == INFINITY);
    else if (special == 3 || special == 4) CHECK(std::isnan(got));
    else if (special == 0 || special == 1)  // the FP64 sum, rounded at 2^-53 forty times
      CHECK(std::fabs((double)(got - sum)) <= 40 * 0x1p-53 * (double)mag);
    else
      CHECK(std::fabs((double)(got - sum)) <=
            40 * 0x1p-70 * (double)mag + 0x1p-52 * std::fabs((double)sum));
  }
}
""")
