// Host side of the decoder: the launch entry points, which group a batch by
// dtype family, choose the kernel and its shared memory, and call the
// translation unit of the family (decode_16/32/u8.cu; the kernels are in
// decode_kernels.cuh).
#include "decode_kernels.cuh"
#include "host_internal.h"

namespace zipnn {

// Kernels of each dtype family (decode_<family>.cu) by kind, CTA size
// and CTAs per SM.
const void* decode_kernel_16(int kind, int threads, bool three);
const void* decode_kernel_32(int kind, int threads, bool three);
const void* decode_kernel_u8(int kind, int threads, bool three);

namespace {

// The kernel of a launch and its shared memory: ntab table slots | stage |
// raw-word rings.
struct DecodeConfig {
  int kind;
  uint32_t ntab, stage, ring;
};

// The stage is meant to hold the coded payloads of the largest chunk: a fraction
// of it (frac64 / 64, see stage_frac64) or what a plan read from the chunk maps
// (stage_need).  It takes all the shared memory that the most CTAs per SM with
// room for that leave it: as many as the kernel's registers allow, at least two of
// 256 threads (a launch of fewer work items than that: one).  Payloads that do not
// fit are decoded in slices, so there is always room, with the raw-word rings
// behind the stage, for the tables of every coded group after the first ntab and
// for the least slice.  Where payloads much larger than the stage are expected (1 MiB
// chunks: one CTA per SM) or there is no such room, and for U8, they are not staged: the
// stage holds the readers' rings, kRingSlotsMax pieces of 16 B per thread.  FP32 plans
// most of whose chunks do not take the weight loop (`general`) take the kernel for
// deltas, which has the general loop alone, while their payloads fit its stage (256 MiB
// pruned to 10%: 267 us, by rings 832), else the rings (16 values: 512 us; by slices 667).
DecodeConfig decode_config(const DecodeShape& sh, int threads, uint64_t items_per_sm) {
  DecodeConfig c;
  const uint32_t per_cta = kSmReserve + kStaticReserve;
  const bool fp32 = sh.family == ZIPNN_FP32;
  c.kind = sh.delta || sh.general ? kDeltas : kWeights;
  c.ntab = c.kind == kDeltas && sh.max_groups > 1 ? 2u : 1u;
  c.ring = fp32 && c.kind == kWeights ? kRingBytes * (uint32_t)threads : 0u;
  const uint32_t tabs =
      sh.max_groups > (int)c.ntab ? (uint32_t)(sh.max_groups - (int)c.ntab) * kLutBytes : 0u;
  auto cap = [&](uint32_t ctas) -> uint32_t {  // the stage that leaves `ctas` per SM
    return kSmPerSm / ctas - per_cta - c.ntab * kLutBytes - c.ring;
  };
  const uint64_t want =
      sh.stage_need ? sh.stage_need : sh.max_chunk * (uint64_t)sh.frac64 / 64 + 1024;
  // the least slice: of every coded group the longest sub-stream that the codes allow
  // (12 bits a symbol), the bitmap, and what its pieces are rounded to.  FP32 weights
  // slice chunks of one HUFF group only, which need no other table (kReadsDirect).
  const uint64_t vecs = (sh.max_chunk / 16 + sh.min_lanes - 1) / sh.min_lanes;
  const uint64_t fixed =
      fp32 && c.kind == kWeights ? 192 : tabs + (sh.max_chunk / 128 + 192) * (uint64_t)sh.max_groups;
  const uint64_t slice = fixed + vecs * (fp32 && c.kind == kWeights ? 6 : 24);
  const uint32_t two = 2u * (256u / (uint32_t)threads);
  const uint32_t least = items_per_sm >= two ? two : (items_per_sm ? (uint32_t)items_per_sm : 1u);
  // (the register budgets of the kernels, see kernel_of)
  uint32_t ctas = threads == 256 && (!fp32 || c.kind == kWeights) ? 3u : two;
  while (ctas > least && cap(ctas) < want) ctas--;
  while (ctas > 1u && (cap(ctas) < fixed || cap(ctas) + c.ring < tabs)) ctas--;
  const uint64_t room = cap(ctas);
  const bool over = want > room + (sh.general ? 0 : room / 8);
  if (sh.family == ZIPNN_U8 || (over && (!sh.stage_need || sh.general)) || room < slice) {
    c.kind = kRings;
    c.ring = 0;
    c.stage = kRingSlotsMax * 16u * (uint32_t)threads + tabs;
  } else {
    c.stage = (uint32_t)room;
  }
  return c;
}

}  // namespace

int group_decode_jobs(std::vector<Job>& jobs, const std::vector<uint64_t>& chunks,
                      DecodeGroup* groups) {
  std::vector<Job> sorted;
  sorted.reserve(jobs.size());
  int n = 0;
  for (int family : {(int)ZIPNN_BF16, (int)ZIPNN_FP32, (int)ZIPNN_U8}) {
    DecodeGroup g;
    g.first = (int)sorted.size();
    for (size_t i = 0; i < jobs.size(); i++) {
      Job J = jobs[i];
      if (dtype_family(J.dtype) != family) continue;
      J.chunk_begin = g.nchunks;
      g.nchunks += chunks[i];
      g.shape.add(J.dtype, J.flags, J.chunk_bytes, J.lanes);
      sorted.push_back(J);
    }
    g.count = (int)sorted.size() - g.first;
    if (g.nchunks) groups[n++] = g;
  }
  jobs.swap(sorted);
  return n;
}

cudaError_t launch_decode_groups(const Job* d_jobs, const DecodeGroup* groups, int ngroups,
                                 const zipnn_tuning* tuning, uint32_t* d_err,
                                 unsigned long long* d_tickets, cudaStream_t st) {
  for (int k = 0; k < ngroups; k++) {
    const cudaError_t e =
        launch_decode_ex(d_jobs + groups[k].first, nullptr, groups[k].count, groups[k].nchunks,
                         groups[k].shape, tuning, d_err, d_tickets + 2 * k, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_decode_ex(const Job* d_jobs, const Job* h_one, int njobs,
                             uint64_t nchunks_total, const DecodeShape& shape,
                             const zipnn_tuning* tuning, uint32_t* d_err,
                             unsigned long long* d_ticket, cudaStream_t st) {
  if (nchunks_total == 0) return cudaSuccess;
  JobRef r;
  r.table = h_one ? nullptr : d_jobs;
  if (h_one) r.one = *h_one;
  else memset(&r.one, 0, sizeof(Job));
  r.n = njobs;
  const int sms = device_sms();
  const int want_threads = (tuning && tuning->threads) ? tuning->threads : 256;
  const int want_parts = tuning ? tuning->parts : 0;
  // Launches with few chunks split every chunk's sub-streams over `parts` work
  // items so that more SMs work on them (tuning->parts: 0 = this rule, 1 =
  // never, 2, 4 or 8 = always): the most parts that keep the items within one
  // per SM and 64 sub-streams in each
  uint32_t parts = 1;
  if (want_parts == 2 || want_parts == 4 || want_parts == 8) {
    parts = (uint32_t)want_parts;
  } else if (want_parts == 0) {
    while (parts < 8 && nchunks_total * parts * 2 <= (uint64_t)sms &&
           shape.max_lanes >= parts * 2 * 64)
      parts *= 2;
  }
  const int threads = want_threads == 256 && shape.max_lanes / parts > 128 ? 256 : 128;
  const DecodeConfig cfg =
      decode_config(shape, threads, (nchunks_total * parts + (uint64_t)sms - 1) / (uint64_t)sms);
  const int smem = (int)(cfg.ntab * kLutBytes + cfg.stage + cfg.ring);
  const bool three = 3u * ((uint32_t)smem + kStaticReserve + kSmReserve) <= kSmPerSm;
  const void* kern = shape.family == ZIPNN_BF16   ? decode_kernel_16(cfg.kind, threads, three)
                     : shape.family == ZIPNN_FP32 ? decode_kernel_32(cfg.kind, threads, three)
                                                  : decode_kernel_u8(cfg.kind, threads, three);
  // (all of the unified L1 / shared array as shared memory, so the CTAs per SM
  // that the occupancy query reports are the ones that become resident)
  int occ = 0;
  const cudaError_t e = prepare_kernel(kern, smem, threads, &occ);
  if (e != cudaSuccess) return e;
  int per_sm = tuning && tuning->ctas_per_sm > 0 ? tuning->ctas_per_sm : occ;
  if (per_sm > occ) per_sm = occ;
  uint64_t grid = (uint64_t)sms * per_sm;
  if (grid > nchunks_total * parts) grid = nchunks_total * parts;
  uint32_t dbg = tuning ? (uint32_t)tuning->debug_flags : 0u;
  // the loops' L2 prefetch budget, shared by the CTAs that run at once
  uint64_t pf64 = kPfBudget / grid;
  uint32_t pf = (uint32_t)(pf64 > (64u << 20) ? (64u << 20) : pf64);
  uint32_t ntab = cfg.ntab, stage = cfg.stage, ring = cfg.ring;
  // the kernel's parameters, in the order of k_decode's signature
  void* args[] = {&r, &nchunks_total, &d_err, &d_ticket, &dbg, &ntab, &stage, &ring, &pf, &parts};
  return cudaLaunchKernel(kern, dim3((unsigned)grid), dim3((unsigned)threads), args, (size_t)smem,
                          st);
}

}  // namespace zipnn
