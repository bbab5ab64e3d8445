// Host part of the integer tensor path (step_split.cu, step_rows.cu): the balanced base-256 digits of the gossip polynomial, and
// the groups of inputs that tell which coordinates may share one scale.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "detag_internal.h"

namespace detag {

// Groups of inputs for the test described in step_split.cu, for the n x n matrix whose first `rows` rows are given (the others
// follow from the block structure).  For each theta and group size a greedy cover: take an output that no group serves yet
// and add those of its inputs, one after the other, that keep the most other such outputs served.  Kept is the one with the
// least expected work: reads of its groups against coordinates in float64, if operands were drawn alike (an operand is below
// tau of the largest with a probability of about 2 tau, a group with its size's power of that) and, weighing less, if their
// magnitudes were spread evenly over four decades.
// Counting bits is most of it: in one instruction where the processor has it (256 workers, K = 4 15.8 -> 3.8 ms).
#if defined(__x86_64__) && defined(__GNUC__) && !defined(__clang__)
__attribute__((target_clones("popcnt", "default")))
#endif
void split_guard(int n, const std::vector<double>& poly, int rows, SplitPoly& out) {
  constexpr int kWords = 4, kLevels = 7;
  // level[i][j] = k: output i gives input j between 2^-k and 2^(1 - k) of its largest weight (0: all of it)
  std::vector<uint8_t> level(static_cast<size_t>(n) * n, 255);
  int terms = 1;
  for (int i = 0; i < n; ++i) {
    uint8_t* const to = &level[static_cast<size_t>(i) * n];
    if (i >= rows) {  // beyond the given ones: the block structure moves them
      const uint8_t* const from = &level[static_cast<size_t>(i % rows) * n];
      const int shift = i / rows * rows;
      std::copy(from, from + n - shift, to + shift);
      std::copy(from + n - shift, from + n, to);
      continue;
    }
    const double* row = &poly[static_cast<size_t>(i) * n];
    double top = 0.0;
    int count = 0;
    for (int j = 0; j < n; ++j) {
      const double v = std::fabs(row[j]);
      top = v > top ? v : top;
      count += v != 0.0 ? 1 : 0;
    }
    terms = std::max(terms, count);
    for (int j = 0; j < n; ++j) {
      int k = 0;
      for (int q = 0; q < kLevels; ++q) k += std::fabs(row[j]) < 0.999999 * top / (1 << q) ? 1 : 0;
      to[j] = static_cast<uint8_t>(k < kLevels ? k : 255);
    }
  }
  const int stride = n % 2 == 0 ? n / 2 - (n % 4 == 0 ? 1 : 2) : n / 2;  // coprime to n: ties go to inputs far apart
  double best = 1e300;
  std::vector<uint64_t> readers(static_cast<size_t>(n) * kWords, 0);  // [input]: outputs that give it at least theta
  std::vector<int> inputs, have_list(n);
  std::vector<uint8_t> groups, list(static_cast<size_t>(n) * n);  // [output]: its inputs of at least theta, once they have been asked for
  for (int k = 0; k < kLevels && best > 0.25 * n; ++k) {
    const double tau = std::sqrt(static_cast<double>(terms)) / 4096.0 * (1 << k);
    if (tau > 0.5) break;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        if (level[static_cast<size_t>(i) * n + j] == k) readers[static_cast<size_t>(j) * kWords + i / 64] |= 1ull << (i % 64);
    std::fill(have_list.begin(), have_list.end(), -1);
    const double small = std::fmax(0.0, 1.0 - std::log2(1.0 / tau) / 13.3);
    int largest = 32;  // of a group, as far as its outputs have such inputs
    for (int size = 2; size <= 32 && size / 2 <= largest && best > 0.25 * n; size *= 2) {
      // what even a single group of this size would cost
      const double least = size + n * (6000.0 * std::fmin(std::pow(2.0 * tau, size), 1.0) + 40.0 * std::fmin(std::pow(small, size), 1.0));
      if (least >= best) continue;
      uint64_t open[kWords] = {0, 0, 0, 0};
      for (int i = 0; i < n; ++i) open[i / 64] |= 1ull << (i % 64);
      groups.clear();
      largest = 0;
      double fail = 0.0, fail_spread = 0.0;
      for (int i = 0; i < n && groups.size() <= 2 * static_cast<size_t>(n) && groups.size() < best; ++i) {
        if ((open[i / 64] >> (i % 64) & 1) == 0) continue;
        uint8_t* const of = &list[static_cast<size_t>(i) * n];
        if (have_list[i] < 0) {
          have_list[i] = 0;
          for (int v = 0, j = i; v < n; ++v, j = j + stride < n ? j + stride : j + stride - n)
            if (level[static_cast<size_t>(i) * n + j] <= k) of[have_list[i]++] = static_cast<uint8_t>(j);
        }
        inputs.assign(of, of + have_list[i]);
        uint64_t served[kWords];
        std::copy(open, open + kWords, served);
        int have = 0;
        uint8_t last = 0;
        double p = 1.0, p_spread = 1.0;
        for (; have < size && have < static_cast<int>(inputs.size()); ++have, p *= 2.0 * tau, p_spread *= small) {
          int pick = have, most = -1;
          for (int v = have; v < static_cast<int>(inputs.size()); ++v) {
            const uint64_t* r = &readers[static_cast<size_t>(inputs[v]) * kWords];
            int count = 0;
            for (int w = 0; w < kWords; ++w) count += __builtin_popcountll(served[w] & r[w]);
            if (count > most) {
              most = count;
              pick = v;
            }
          }
          std::swap(inputs[have], inputs[pick]);
          const int j = inputs[have];
          for (int w = 0; w < kWords; ++w) served[w] &= readers[static_cast<size_t>(j) * kWords + w];
          last = static_cast<uint8_t>(j);
          groups.push_back(last);
        }
        largest = std::max(largest, have);
        for (; have < size; ++have) groups.push_back(last);
        for (int w = 0; w < kWords; ++w) open[w] &= ~served[w];
        fail += p;
        fail_spread += p_spread;
      }
      const double work = groups.size() + n * (6000.0 * std::fmin(fail, 1.0) + 40.0 * std::fmin(fail_spread, 1.0));
      if (groups.size() <= 2 * static_cast<size_t>(n) && work < best) {
        best = work;
        out.guard = groups;
        out.guard_size = size;
        out.guard_tau = static_cast<float>(tau);
      }
    }
  }
  if (out.guard.empty()) {  // nothing to tell the coordinates by: all in float64 (one input is as good as another)
    out.guard.assign(2, 0);
    out.guard_size = 2;
    out.guard_tau = 2.f;
  }
  // Magnitudes spread evenly over four decades, times a normal: the largest of many is some 2 10^2, and an operand is below tau of it with
  // a probability of 1 - (log10(1 / tau) - 0.6) / 4.
  const double below = std::fmin(std::fmax(1.0 - (-std::log10(std::fmin(out.guard_tau, 1.f)) - 0.6) / 4.0, 0.0), 1.0);
  out.unequal = static_cast<float>(std::fmin(static_cast<double>(out.guard.size()) / out.guard_size * std::pow(below, out.guard_size), 1.0));
}

// Digits of the `rows` given rows of the n x n matrix, as bytes of 64-bit integers (`wide` per row, zeros beyond n), and the exponent
// of every row's scale (rows beyond the given ones: the block structure repeats them).  False if an entry or a row cannot be scaled.
bool split_digits(int n, const std::vector<double>& poly, int rows, int wide, std::vector<int64_t>& digits, std::vector<int32_t>& row_exp) {
  constexpr long long kMaxDigits = 0x7F7F7F7F7FLL;  // largest integer with five balanced digits
  digits.assign(static_cast<size_t>(rows) * wide, 0);
  row_exp.assign(n, 0);
  for (int i = 0; i < rows; ++i) {
    const double* row = &poly[static_cast<size_t>(i) * n];
    double top = 0.0;
    for (int j = 0; j < n; ++j) {
      const double v = std::fabs(row[j]);
      if (!(v <= 1e30)) return false;  // also NaN
      top = v > top ? v : top;
    }
    if (!(top >= 1e-30)) return false;
    int e = std::ilogb(top);
    if (std::nearbyint(std::ldexp(top, 38 - e)) > static_cast<double>(kMaxDigits)) ++e;
    for (int k = i; k < n; k += rows) row_exp[k] = e - 30;
    const double scale = std::ldexp(1.0, 38 - e);
    for (int j = 0; j < n; ++j)
      digits[static_cast<size_t>(i) * wide + j] = (std::llrint(row[j] * scale) + 0x8080808080LL) ^ 0x8080808080LL;
  }
  return true;
}

}  // namespace detag
