// The warps that issue copies and matrix instructions, as sequences of waits
// and issues on rings of shared-memory slots (coarse stencil on the tensor
// cores).  No CUDA type appears here: the kernels pass the waits and the issues
// in, and the host compiles the same text with waits that give up, so that what
// a role does then is tested without a GPU.
//
// Every wait is bounded.  Whichever role gives up, and however late, each role
// ends by waiting (bounded again) for what it has issued itself: copies land
// and matrix instructions complete before the CTA gives its shared and tensor
// memory back.  Where nothing gave up these waits return at once.
#pragma once

#ifdef __CUDACC__
#define DWF_ROLE __device__ __forceinline__
#else
#define DWF_ROLE inline
#endif

namespace dwfk {

// Waits for the copies of a ring's last uses (the older slots were freed, so
// their copies have landed); full(slot, parity).
template <unsigned SLOTS, class Full>
DWF_ROLE void ring_drain(unsigned issued, const Full& full) {
  for (unsigned k = issued > SLOTS ? issued - SLOTS : 0; k < issued; k++) full(k % SLOTS, (k / SLOTS) & 1);
}

// Coarse stencil, copies: stage g goes to slot g % S once the matrix
// instructions of stage g - S are done.
template <int S, class Done, class Full, class Issue, class Raise>
DWF_ROLE void tc_copy_role(int nst, const Done& done, const Full& full, const Issue& issue, const Raise& raise) {
  int issued = 0;
  for (; issued < nst; issued++) {
    if (issued >= S && !done(issued % S, (issued / S - 1) & 1)) {
      raise();
      break;
    }
    issue(issued, issued % S);
  }
  ring_drain<S>((unsigned)issued, full);
}

// Coarse stencil, matrix instructions: nine stages (directions) a group of
// sites, NBUF accumulators; multiply(h, d, t, slot) also commits.
template <int S, int NBUF, class Empty, class Full, class Done, class Multiply, class Raise>
DWF_ROLE void tc_mma_role(int nst, const Empty& acc_empty, const Full& full, const Done& done, const Multiply& multiply,
                          const Raise& raise) {
  int h = 0;
  for (; h < nst; h++) {
    const int ql = h / 9, d = h % 9, t = ql % NBUF;
    if ((d == 0 && ql >= NBUF && !acc_empty(t, (ql / NBUF - 1) & 1)) || !full(h % S, (h / S) & 1)) {
      raise();
      break;
    }
    multiply(h, d, t, h % S);
  }
  if (h > 0) done((h - 1) % S, ((h - 1) / S) & 1);  // a commit covers all that was issued before it
}

}  // namespace dwfk
