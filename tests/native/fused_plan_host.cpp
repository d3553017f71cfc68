// Host entry points over the tile plans of the one-barrier solves (csrc/fused_plan.h), for the CPU tests.
#include "ccm.h"
#include "fused_plan.h"

using namespace ccm;

extern "C" {

long noalloc_max_elems(void) { return CCM_NOALLOC_MAX_ELEMS; }

void plan_of(int nx, int ny, int sms, long max_slots, int out[4]) {
  fused_tiles(nx, ny, sms, &out[0], &out[1], &out[2], &out[3], kResidentCells, 512, max_slots < 0 ? SIZE_MAX : (size_t)max_slots);
}

// 0 if the built-in resident plan of (nx, ny) covers the grid with one tile per SM, within max_slots
// mailbox slots, smem bytes of shared memory and the rows that a thread can take; else which of them fails
static int check(int nx, int ny, int sms, size_t max_slots, size_t smem) {
  int TX = 0, TY = 0, nbx = 0, nt = 0;
  fused_tiles(nx, ny, sms, &TX, &TY, &nbx, &nt, kResidentCells, 512, max_slots);
  if (nt < 1 || nt > sms || nt != nbx * ((ny + TY - 1) / TY) || nbx * TX < nx) return 1;
  if (fused_mail_slots(nx, TX, TY, nt) > max_slots) return 2;
  if (fused_resident_smem_min(TX, TY) > smem) return 3;
  if (TX * TY > kFusedRows * fused_threads(TX, TY, nt, sms)) return 4;
  return 0;
}

// Every grid that the allocation-free solve takes: the first (nx, ny) that fails, into bad; how many passed.
long check_noalloc(int sms, long smem, int bad[3]) {
  const size_t elems = CCM_NOALLOC_MAX_ELEMS;
  long n = 0;
  bad[0] = bad[1] = bad[2] = 0;
  for (int nx = 4; (size_t)((nx + 3 + 31) / 32 * 32) * 7 <= elems; ++nx)
    for (int ny = 4; (size_t)((nx + 3 + 31) / 32 * 32) * (size_t)(ny + 3) <= elems; ++ny) {
      const int e = check(nx, ny, sms, 2 * elems, (size_t)smem);
      if (e) {
        bad[0] = nx;
        bad[1] = ny;
        bad[2] = e;
        return n;
      }
      ++n;
    }
  return n;
}

// Slots that a case's plan set by the caller can need beyond what its mailboxes hold: the excess
long mail_excess(int nx, int ny, int TX, int TY) {
  const int nbx = (nx + TX - 1) / TX, nt = nbx * ((ny + TY - 1) / TY);
  if (nt > kFusedTilesMax || fused_resident_smem_min(TX, TY) > 227 * 1024) return 0;
  return (long)fused_mail_slots(nx, TX, TY, nt) - (long)fused_mail_slots_max(nx, ny);
}
}
