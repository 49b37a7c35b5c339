"""The kernels that read a matrix at the row or column numbers a pivoted LU left behind: an LU whose
exchange gave up (RLU_ETIMEOUT) carries on without it, so P and Q may keep entries that nothing has
written. Entries outside the matrix read as zero, never out of bounds; all others as ever. On the
CPU, from the kernels' source."""
import cuda_on_host

# rows or columns in reverse order, every third entry one that no LU writes
PERM = r"""
static std::vector<int32_t> perm_of(int n) {
  const int32_t bad[] = {-1, n, n + 1, INT32_MAX, INT32_MIN, 7 * n};
  std::vector<int32_t> p(n);
  for (int i = 0; i < n; ++i) p[i] = i % 3 == 1 ? bad[i / 3 % 6] : n - 1 - i;
  return p;
}
static bool ok(int32_t p, int n) { return p >= 0 && p < n; }
"""


def test_l_b_and_u(tmp_path):
    cuda_on_host.run(tmp_path, [("small.cu", "tf32_split"), ("small.cu", "k_gather_lb_u")],
                     PERM + r"""
int main() {
  const int k = 7, n = 300, ldb = 300;
  auto Q = perm_of(n);
  std::vector<float> B(k * ldb), U(k * n, -9.f), Lb(k * k, -9.f), Lh(k * 8), Ll(k * 8);
  for (size_t i = 0; i < B.size(); ++i) B[i] = 1.f + i;
  launch({2, 2 + 1}, {256}, [&] {
    k_gather_lb_u<float>(B.data(), ldb, Q.data(), k, n, Lb.data(), Lh.data(), Ll.data(), 8, U.data(), n);
  });
  for (int i = 0; i < k; ++i)
    for (int j = 0; j < n; ++j)
      CHECK(U[i * n + j] == (j >= i && ok(Q[j], n) ? B[i * ldb + Q[j]] : 0.f));
  for (int i = 0; i < k; ++i)
    for (int j = 0; j < k; ++j)
      CHECK(Lb[j * k + i] == (i > j ? (ok(Q[j], n) ? B[i * ldb + Q[j]] : 0.f) : i == j));
}
""")


def test_rows_of_a(tmp_path):
    cuda_on_host.run(tmp_path, [("fast.cu", "k_frlu_gather_aj")], PERM + r"""
int main() {
  const int m = 40, n = 70, l = 25;
  auto P = perm_of(m);
  std::vector<float> A(m * n), AJ(l * n, -9.f);
  for (size_t i = 0; i < A.size(); ++i) A[i] = 1.f + i;
  launch({1, l}, {256}, [&] { k_frlu_gather_aj(A.data(), n, m, n, P.data(), AJ.data(), n); });
  for (int i = 0; i < l; ++i)
    for (int c = 0; c < n; ++c) CHECK(AJ[i * n + c] == (ok(P[i], m) ? A[P[i] * n + c] : 0.f));
}
""")


def test_rows_in_pivot_order(tmp_path):
    cuda_on_host.run(tmp_path, [("fast.cu", "k_c_cm_to_rm_perm")], PERM + r"""
int main() {
  const int R = 70, C = 33;
  auto P = perm_of(R);
  std::vector<float2> X(R * C), Y(R * C);
  for (int i = 0; i < R * C; ++i) X[i] = {1.f + i, -1.f - i};
  launch({3, 2}, {32, 8}, [&] { k_c_cm_to_rm_perm(X.data(), R, R, C, P.data(), Y.data(), C); });
  for (int p = 0; p < R; ++p)
    for (int c = 0; c < C; ++c) {
      CHECK(Y[p * C + c].x == (ok(P[p], R) ? X[c * R + P[p]].x : 0.f));
      CHECK(Y[p * C + c].y == (ok(P[p], R) ? X[c * R + P[p]].y : 0.f));
    }
}
""")
