/* Compares igen_exp2_by with igen_exp2 for every fraction and every power from 2^0 to 2^30; prints how many differ. */
#include <stdio.h>

#include "../paper_2406_05221_b200/csrc/igen.h"

int main(void) {
  static igen_exp2_tables_t t;
  long differ = 0;
  for (int e = 0; e < (1 << IGEN_LEAD_BITS) + 2 * (1 << IGEN_TAIL_BITS); ++e) igen_exp2_entry(&t, e);
#pragma omp parallel for reduction(+ : differ)
  for (long f = 0; f < (1L << IGEN_FRAC_BITS); ++f) {
    const uint64_t low = (uint64_t)f << (32 - IGEN_FRAC_BITS);
    for (uint64_t k = 0; k <= 30; ++k) differ += igen_exp2_by(&t, (k << 32) | low) != igen_exp2((k << 32) | low);
  }
  printf("%ld\n", differ);
  return 0;
}
