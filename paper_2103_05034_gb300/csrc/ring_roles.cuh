// The warps that issue copies and matrix instructions, as sequences of waits
// and issues on rings of shared-memory slots (streaming hopping kernel, coarse
// stencil on the tensor cores).  No CUDA type appears here: the kernels pass
// the waits and the issues in, and the host compiles the same text with waits
// that give up, so that what a role does then is tested without a GPU.
//
// Every wait is bounded.  Whoever gives up, and however late, each role
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

// Streaming hopping kernel: rings of centre slices and links (three slots) and
// of the halo's y and z rows (two slots each); empty(ring, slot, parity),
// full(ring, slot, parity), centre(i, slot), links(i, slot), halo(i, part,
// slot).
enum { RING_C = 0, RING_L = 1, RING_Y = 2, RING_Z = 3 };

struct StreamProducer {
  unsigned kc = 0, kl = 0, ky = 0, kz = 0;  // copies issued per ring
  bool ok = true;

  template <unsigned SLOTS, class Empty>
  DWF_ROLE bool acquire(const Empty& empty, int ring, unsigned k) {
    if (k >= SLOTS) ok = ok && empty(ring, k % SLOTS, (k / SLOTS - 1) & 1);
    return ok;
  }
  // A run of nt steps; step s reads slices s, s + 1, s + 2 of the run's nt + 2.
  template <class Empty, class Centre, class Links, class Halo>
  DWF_ROLE void run(int nt, const Empty& empty, const Centre& centre, const Links& links, const Halo& halo) {
    const auto slice = [&](int i) {
      if (acquire<3>(empty, RING_C, kc)) {
        centre(i, kc % 3);
        kc++;
      }
    };
    slice(0);
    slice(1);
    for (int s = 0; ok && s < nt; s++) {
      if (acquire<3>(empty, RING_L, kl)) {
        links(s, kl % 3);
        kl++;
      }
      if (acquire<2>(empty, RING_Y, ky)) {
        halo(s, 0, ky & 1);
        ky++;
      }
      if (acquire<2>(empty, RING_Z, kz)) {
        halo(s, 1, kz & 1);
        kz++;
      }
      slice(s + 2);
    }
  }
  template <class Full, class Raise>
  DWF_ROLE void finish(const Full& full, const Raise& raise) {
    if (!ok) raise();
    ring_drain<3>(kc, [&](unsigned slot, unsigned par) { full(RING_C, slot, par); });
    ring_drain<3>(kl, [&](unsigned slot, unsigned par) { full(RING_L, slot, par); });
    ring_drain<2>(ky, [&](unsigned slot, unsigned par) { full(RING_Y, slot, par); });
    ring_drain<2>(kz, [&](unsigned slot, unsigned par) { full(RING_Z, slot, par); });
  }
};

}  // namespace dwfk
