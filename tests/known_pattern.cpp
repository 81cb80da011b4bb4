// Products on a known pattern (csr_product_numeric) against the canonical sums on
// the host, with rows of C past every class of the kernels; run by
// test_gpu_refresh.py on a GPU.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>
#include <set>
#include <vector>

#include "amg.cuh"

#define TRY(x)                                                           \
  do {                                                                   \
    const cudaError_t e_ = (x);                                          \
    if (e_ != cudaSuccess) {                                             \
      std::printf("%s: %s\n", #x, cudaGetErrorString(e_));               \
      std::exit(1);                                                      \
    }                                                                    \
  } while (0)

struct Csr {
  int n, m;
  std::vector<int> rp, col;
  std::vector<double> val;
};

static tp::DevCSR upload(const Csr& a, tp::Pool& pool) {
  tp::DevCSR d;
  d.n = a.n;
  d.m = a.m;
  d.nnz = (int)a.col.size();
  d.rowptr = pool.alloc<int>(a.n + 1);
  d.col = pool.alloc<int>(d.nnz);
  d.val = pool.alloc<double>(d.nnz);
  TRY(cudaMemcpy(d.rowptr, a.rp.data(), sizeof(int) * (a.n + 1), cudaMemcpyHostToDevice));
  TRY(cudaMemcpy(d.col, a.col.data(), sizeof(int) * d.nnz, cudaMemcpyHostToDevice));
  TRY(cudaMemcpy(d.val, a.val.data(), sizeof(double) * d.nnz, cudaMemcpyHostToDevice));
  return d;
}

// rows of the given lengths, distinct ascending columns out of m
static Csr random_rows(const std::vector<int>& len, int m, std::mt19937_64& rng) {
  Csr a{(int)len.size(), m, {0}, {}, {}};
  std::uniform_int_distribution<int> c(0, m - 1);
  std::normal_distribution<double> v;
  for (int l : len) {
    std::set<int> s;
    while ((int)s.size() < l) s.insert(c(rng));
    for (int j : s) {
      a.col.push_back(j);
      a.val.push_back(v(rng));
    }
    a.rp.push_back((int)a.col.size());
  }
  return a;
}

// one product: rows of A of these lengths, rows of B of about `mean` entries
static int check(const std::vector<int>& len, int k, int mean, int m, unsigned seed) {
  std::mt19937_64 rng(seed);
  const Csr A = random_rows(len, k, rng);
  std::vector<int> lb(k);
  for (int i = 0; i < k; ++i) lb[i] = 1 + (int)(rng() % (unsigned)(2 * mean - 1));
  const Csr B = random_rows(lb, m, rng);
  tp::Pool pool, scratch;
  tp::DevCSR a = upload(A, pool), b = upload(B, pool);
  const tp::DevCSR C = tp::csr_product(a, b, pool, scratch, nullptr);
  // other values of A on the same pattern; C's are overwritten
  std::vector<double> nv(A.val.size());
  std::normal_distribution<double> v;
  for (double& x : nv) x = v(rng);
  TRY(cudaMemcpy(a.val, nv.data(), sizeof(double) * nv.size(), cudaMemcpyHostToDevice));
  TRY(cudaMemset(C.val, 0xff, sizeof(double) * C.nnz));
  scratch.release();
  tp::csr_product_numeric(a, b, C, scratch, nullptr);
  TRY(cudaDeviceSynchronize());
  std::vector<int> rp(C.n + 1), col(C.nnz);
  std::vector<double> val(C.nnz);
  TRY(cudaMemcpy(rp.data(), C.rowptr, sizeof(int) * (C.n + 1), cudaMemcpyDeviceToHost));
  TRY(cudaMemcpy(col.data(), C.col, sizeof(int) * C.nnz, cudaMemcpyDeviceToHost));
  TRY(cudaMemcpy(val.data(), C.val, sizeof(double) * C.nnz, cudaMemcpyDeviceToHost));
  int longest = 0;
  for (int i = 0; i < A.n; ++i) {
    std::map<int, double> sum;
    for (int e = A.rp[i]; e < A.rp[i + 1]; ++e)
      for (int f = B.rp[A.col[e]]; f < B.rp[A.col[e] + 1]; ++f)
        sum.emplace(B.col[f], 0.0).first->second += nv[e] * B.val[f];
    if ((int)sum.size() != rp[i + 1] - rp[i]) {
      std::printf("row %d: %d columns, not %zu\n", i, rp[i + 1] - rp[i], sum.size());
      return -1;
    }
    int q = rp[i];
    for (const auto& s : sum) {
      if (col[q] != s.first || val[q] != s.second) {
        std::printf("row %d (%zu columns): column %d %.17g, not %d %.17g\n", i, sum.size(), col[q],
                    val[q], s.first, s.second);
        return -1;
      }
      ++q;
    }
    longest = std::max(longest, rp[i + 1] - rp[i]);
  }
  return longest;
}

int main() {
  // mean row lengths of B in each lane-group choice (4, 8, 16 lanes and up)
  for (int mean : {3, 8, 20}) {
    // short rows on the whole, some past 48 and 192 columns
    std::vector<int> len(400, 5);
    for (int i = 0; i < 400; i += 7) len[i] = 1 + (i % 90);
    if (check(len, 3000, mean, 5000, 1 + mean) < 0) return 1;
    // long rows on the whole, around 192 and 1536 columns and past
    len.assign(60, 300 / mean);
    for (int i = 0; i < 60; i += 5) len[i] = (1000 + 45 * i) / mean;
    const int longest = check(len, 3000, mean, 20000, 100 + mean);
    if (longest < 0) return 1;
    if (longest < 1700) {
      std::printf("no row past the longest class (%d)\n", longest);
      return 1;
    }
  }
  return 0;
}
