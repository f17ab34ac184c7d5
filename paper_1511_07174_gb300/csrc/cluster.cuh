// Thread-block clusters: shared memory of the other CTAs, mbarriers that count
// the bytes pushed into it, and the cluster barrier.
#pragma once
#include "common.cuh"

namespace gbla {

GBLA_DEVINL uint32_t cl_smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
GBLA_DEVINL uint32_t cl_mapa(uint32_t a, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// 16 bytes to another CTA's shared memory, completing them on that CTA's mbarrier.
GBLA_DEVINL void cl_push16(uint32_t rdst, ulonglong2 v, uint32_t rbar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(rdst),
      "l"(v.x), "l"(v.y), "r"(rbar)
      : "memory");
}
GBLA_DEVINL void cl_store_remote_u32(uint32_t raddr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(raddr), "r"(v) : "memory");
}
GBLA_DEVINL void cl_mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
GBLA_DEVINL void cl_mbar_arm(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// Count `bytes` as arrived on this CTA's mbarrier (bytes that no copy will bring).
GBLA_DEVINL void cl_mbar_complete_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
GBLA_DEVINL bool cl_mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
GBLA_DEVINL bool cl_mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase of the given parity. A limit of 0 does not wait
// at all (one non-blocking test), so that "give up at once" is what it says:
// try_wait may itself suspend the thread for a while before it answers.
GBLA_DEVINL bool cl_mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  if (limit_ns == 0) return cl_mbar_test(bar, parity);
  if (cl_mbar_try(bar, parity)) return true;
  const uint64_t t0 = gbla_now_ns();
  while (!cl_mbar_try(bar, parity))
    if (gbla_now_ns() - t0 > limit_ns) return false;
  return true;
}
GBLA_DEVINL uint32_t cl_nctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
GBLA_DEVINL uint32_t cl_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
GBLA_DEVINL void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

}  // namespace gbla
