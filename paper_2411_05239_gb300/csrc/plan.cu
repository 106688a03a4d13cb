// Plans: a batch of tensors prepared once (device job table, scratch, work
// ticket) and captured as a CUDA graph, so that every later batched
// compression or persistent-kernel decompression of the same tensors costs one
// cudaGraphLaunch.  This is the batching form of the codec: many tensors of
// uneven sizes in one launch per kernel (ZipNN Sec. 5.1: chunks and byte groups
// are independent, so one grid serves them all).
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "zipnn.h"
#include "host_internal.h"


using namespace zipnn;

struct zipnn_plan {
  int kind = 0;                 // 1 = decompress, 2 = compress, 3 = load
  int device = 0;
  void* dmem = nullptr;         // job table + ticket + scratch
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  uint64_t nchunks = 0;
  int count = 0;
};

namespace {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// What a decode launch needs, read from its containers' chunk maps: per chunk
// the shared-memory stage that holds its coded (HUFF / SPARSE) payloads, 16-B
// padded, plus 32 B and the tables of its coded groups past those that have slots
// (the decoder's staging rule).
struct MapNeed {
  uint64_t max_stage = 0;  // largest per-chunk need
  uint64_t chunks = 0;     // chunks seen
  uint64_t over = 0;       // chunks whose need exceeds the default stage
};
// Of FP32 weights the chunks of one HUFF group in front, and the others, which the
// kernel for weights does not stage.
struct MapNeeds {
  MapNeed weights, others;
};

void add_map_need(const uint8_t* map, uint32_t n_chunks, uint32_t G, uint64_t dflt, MapNeeds* nd) {
  for (uint32_t c = 0; c < n_chunks; c++) {
    uint64_t used = 0;
    uint32_t ncoded = 0;
    bool first = false;
    for (uint32_t g = 0; g < G; g++) {
      const uint8_t* e = map + ((uint64_t)c * G + g) * kEntryBytes;
      uint32_t size;
      memcpy(&size, e + 8, 4);
      const uint32_t mode = e[12];
      if (mode == kHuff || mode == kSparse) {
        used += align_up(size, 16);
        ncoded++;
        if (g == 0) first = mode == kHuff;
      }
    }
    const bool other = G == 4 && ncoded && !(ncoded == 1 && first);
    MapNeed& m = other ? nd->others : nd->weights;
    m.chunks++;
    if (ncoded) {
      const uint32_t slots = other ? 2 : 1;
      const uint64_t need =
          used + 32 + (ncoded > slots ? (uint64_t)(ncoded - slots) * 4u * kLutSize : 0u);
      if (need > m.max_stage) m.max_stage = need;
      if (need > dflt) m.over++;
    }
  }
}

// The stage a plan asks for: 0 (the launcher's default rule) while the default
// stage holds the payloads of at least 99% of the chunks, else the largest
// need (which the launcher takes as far as two CTAs still share an SM).  FP32 plans
// most of whose chunks do not take the weight loop ask for the others' need.
void planned_stage(const MapNeeds& nd, DecodeShape* sh) {
  auto need = [](const MapNeed& m) -> uint32_t {
    return (uint32_t)(m.max_stage > 0xFFFFFFFFull ? 0xFFFFFFFFull : m.max_stage);
  };
  if (!sh->delta && nd.others.chunks > nd.weights.chunks) {
    sh->general = true;
    sh->stage_need = std::max(need(nd.others), need(nd.weights));
    return;
  }
  MapNeed m = nd.weights;
  if (sh->delta) {
    m.max_stage = std::max(m.max_stage, nd.others.max_stage);
    m.chunks += nd.others.chunks;
    m.over += nd.others.over;
  }
  sh->stage_need = m.over * 100 <= m.chunks ? 0 : need(m);
}

zipnn_status fail(zipnn_plan* p, cudaError_t e) {
  if (p) {
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    if (p->dmem) cudaFree(p->dmem);
    delete p;
  }
  return e == cudaErrorMemoryAllocation ? ZIPNN_ENOMEM : ZIPNN_ECUDA;
}

// Capture `body` on a private stream into p->graph / p->exec.
template <class F>
cudaError_t capture(zipnn_plan* p, F body) {
  cudaStream_t cs;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e != cudaSuccess) return e;
  e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    cudaError_t eb = body(cs);
    e = cudaStreamEndCapture(cs, &p->graph);
    if (eb != cudaSuccess) e = eb;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&p->exec, p->graph, 0);
  cudaStreamDestroy(cs);
  return e;
}

}  // namespace

extern "C" {

// Decode plan over the global chunk range [lo, hi) of the containers taken in
// order as one sequence (all of it for zipnn_plan_decompress; a rank's share
// for zipnn_plan_decompress_range).  A container whose chunks fall partly in
// the range becomes a job over those chunks only (Job.chunk0), and its
// destination (and base) pointer is shifted so that the kernel's
// dst + chunk * chunk_bytes lands in the caller's buffer of the range.
static zipnn_status plan_decode_range(const zipnn_stream* streams, const void* const* d_bases,
                                      void* const* d_dsts, int count, uint64_t lo, uint64_t hi,
                                      const zipnn_tuning* tuning, zipnn_plan** out) {
  if (!out || count <= 0 || !streams || !d_dsts || lo > hi) return ZIPNN_EINVAL;
  *out = nullptr;
  std::vector<Job> jobs;
  std::vector<uint64_t> chunks;
  uint64_t chunk = 0, g = 0;
  for (int i = 0; i < count; i++) {
    const zipnn_stream* s = &streams[i];
    if (s->n_groups != (uint32_t)elem_size(s->dtype) || s->dtype < 0 || s->dtype > ZIPNN_U8 ||
        s->lanes < 1 || s->lanes > ZIPNN_MAX_LANES || s->chunk_bytes < ZIPNN_MIN_CHUNK ||
        (uint64_t)s->n_chunks != (s->orig_nbytes + s->chunk_bytes - 1) / s->chunk_bytes)
      return ZIPNN_EINVAL;
    const uint64_t a = lo > g ? lo - g : 0;
    const uint64_t b = hi < g + s->n_chunks ? (hi > g ? hi - g : 0) : s->n_chunks;
    g += s->n_chunks;
    if (a >= b) continue;  // no chunk of this container in the range
    if (!s->data || !aligned16(s->data)) return ZIPNN_EINVAL;
    const void* base = d_bases ? d_bases[i] : nullptr;
    if (((s->flags & ZIPNN_FLAG_DELTA) != 0) != (base != nullptr)) return ZIPNN_EINVAL;
    if (!d_dsts[i] || !aligned16(d_dsts[i]) || !aligned16(base)) return ZIPNN_EINVAL;
    const uintptr_t shift = (uintptr_t)(a * s->chunk_bytes);
    Job J;
    memset(&J, 0, sizeof(J));
    J.src = static_cast<const uint8_t*>(s->data);
    J.base = base ? reinterpret_cast<const uint8_t*>(reinterpret_cast<uintptr_t>(base) - shift)
                  : nullptr;
    J.dst = reinterpret_cast<uint8_t*>(reinterpret_cast<uintptr_t>(d_dsts[i]) - shift);
    J.nbytes = s->orig_nbytes;
    J.chunk_bytes = s->chunk_bytes;
    J.lanes = s->lanes;
    J.n_chunks = s->n_chunks;
    J.dtype = s->dtype;
    J.flags = s->flags;
    J.stream_bytes = s->nbytes;
    J.chunk0 = (uint32_t)a;
    chunk += b - a;
    jobs.push_back(J);
    chunks.push_back(b - a);
  }
  if (hi > g) return ZIPNN_EINVAL;
  if (jobs.empty()) return ZIPNN_EINVAL;  // nothing to decode in the range
  const int njobs = (int)jobs.size();
  DecodeGroup groups[kDecodeFamilies];
  const int ngroups = group_decode_jobs(jobs, chunks, groups);
  // stages from the chunk maps present now
  std::vector<uint8_t> mb;
  for (int k = 0; k < ngroups; k++) {
    DecodeGroup& G = groups[k];
    MapNeeds nd;
    const uint64_t dflt = G.shape.max_chunk * (uint64_t)G.shape.frac64 / 64 + 1024;
    for (int i = G.first; i < G.first + G.count; i++) {
      const Job& J = jobs[(size_t)i];
      const uint64_t end = i + 1 < G.first + G.count ? jobs[(size_t)i + 1].chunk_begin : G.nchunks;
      const uint32_t ng = (uint32_t)elem_size(J.dtype);
      const uint64_t mbytes = (uint64_t)J.n_chunks * ng * kEntryBytes;
      if (J.stream_bytes < kHdrBytes + mbytes) continue;  // malformed: the decoder reports it
      mb.resize((size_t)mbytes);
      if (mbytes && cudaMemcpy(mb.data(), J.src + kHdrBytes, (size_t)mbytes,
                               cudaMemcpyDeviceToHost) != cudaSuccess)
        return ZIPNN_ECUDA;
      add_map_need(mb.data() + (uint64_t)J.chunk0 * ng * kEntryBytes, (uint32_t)(end - J.chunk_begin),
                   ng, dflt, &nd);
    }
    planned_stage(nd, &G.shape);
  }
  uint32_t* err = plan_err_word();
  if (!err) return ZIPNN_ECUDA;
  zipnn_plan* p = new zipnn_plan();
  p->kind = 1;
  p->count = njobs;
  p->nchunks = chunk;
  cudaGetDevice(&p->device);
  const size_t tbytes = align_up(sizeof(Job) * (size_t)njobs, 256);
  cudaError_t e = cudaMalloc(&p->dmem, tbytes + 256);
  if (e != cudaSuccess) return fail(p, e);
  Job* d_jobs = static_cast<Job*>(p->dmem);
  auto* ticket = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(p->dmem) + tbytes);
  e = cudaMemcpy(d_jobs, jobs.data(), sizeof(Job) * (size_t)njobs, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(ticket, 0, 2 * sizeof(unsigned long long) * kDecodeFamilies);
  if (e != cudaSuccess) return fail(p, e);
  zipnn_tuning tu;
  memset(&tu, 0, sizeof(tu));
  if (tuning) tu = *tuning;
  e = capture(p, [&](cudaStream_t cs) {
    return launch_decode_groups(d_jobs, groups, ngroups, &tu, err, ticket, cs);
  });
  if (e != cudaSuccess) return fail(p, e);
  *out = p;
  return ZIPNN_OK;
}

zipnn_status zipnn_plan_decompress(const zipnn_stream* streams, const void* const* d_bases,
                                   void* const* d_dsts, int count, const zipnn_tuning* tuning,
                                   zipnn_plan** out) {
  if (!out || count <= 0 || !streams || !d_dsts) return ZIPNN_EINVAL;
  uint64_t total = 0;
  for (int i = 0; i < count; i++) {
    total += streams[i].n_chunks;
    // every container decodes in full: its destination must be given (an
    // empty tensor has no chunks and needs none)
    if (streams[i].orig_nbytes && !d_dsts[i]) return ZIPNN_EINVAL;
  }
  if (total == 0) {
    // only empty containers: a plan whose launch does nothing
    zipnn_plan* p = new zipnn_plan();
    p->kind = 1;
    cudaGetDevice(&p->device);
    cudaError_t e = capture(p, [&](cudaStream_t) { return cudaSuccess; });
    if (e != cudaSuccess) return fail(p, e);
    *out = p;
    return ZIPNN_OK;
  }
  return plan_decode_range(streams, d_bases, d_dsts, count, 0, total, tuning, out);
}

zipnn_status zipnn_plan_decompress_range(const zipnn_stream* streams, const void* const* d_bases,
                                         void* const* d_dsts, int count, uint64_t chunk_lo,
                                         uint64_t chunk_hi, const zipnn_tuning* tuning,
                                         zipnn_plan** out) {
  return plan_decode_range(streams, d_bases, d_dsts, count, chunk_lo, chunk_hi, tuning, out);
}

zipnn_status zipnn_plan_compress(const void* const* d_srcs, const void* const* d_bases,
                                 const size_t* nbytes, const int* dtypes, int count,
                                 size_t chunk_bytes, uint32_t lanes, void* const* d_outs,
                                 const size_t* out_capacities, uint64_t* d_out_nbytes,
                                 zipnn_plan** out) {
  if (!out || count <= 0 || !nbytes || !dtypes || !d_outs || !out_capacities) return ZIPNN_EINVAL;
  *out = nullptr;
  std::vector<Job> jobs((size_t)count);
  uint64_t nch = 0, ngc = 0;
  int max_lanes = 1, max_groups = 1, uniform = dtypes[0];
  for (int i = 0; i < count; i++) {
    const int dt = dtypes[i];
    if (dt != uniform) uniform = -1;
    if (dt < ZIPNN_BF16 || dt > ZIPNN_U8) return ZIPNN_EINVAL;
    const uint32_t ln =
        lanes ? lanes : default_lanes_for(dt, chunk_bytes, d_bases && d_bases[i]);
    const int es = elem_size(dt);
    if (nbytes[i] % es || chunk_bytes < ZIPNN_MIN_CHUNK || chunk_bytes > ZIPNN_MAX_CHUNK ||
        chunk_bytes % 16 || ln < 1 || ln > ZIPNN_MAX_LANES || ln > chunk_bytes / 16)
      return ZIPNN_EINVAL;
    const void* src = d_srcs ? d_srcs[i] : nullptr;
    const void* base = d_bases ? d_bases[i] : nullptr;
    if ((nbytes[i] && !src) || !d_outs[i] || !aligned16(src) || !aligned16(base) ||
        !aligned16(d_outs[i]))
      return ZIPNN_EINVAL;
    if (out_capacities[i] < zipnn_compress_bound(nbytes[i], dt, chunk_bytes)) return ZIPNN_ENOMEM;
    Job J;
    memset(&J, 0, sizeof(J));
    J.src = static_cast<const uint8_t*>(src);
    J.base = static_cast<const uint8_t*>(base);
    J.dst = static_cast<uint8_t*>(d_outs[i]);
    J.nbytes = nbytes[i];
    J.chunk_bytes = (uint32_t)chunk_bytes;
    J.lanes = ln;
    J.n_chunks = (uint32_t)((nbytes[i] + chunk_bytes - 1) / chunk_bytes);
    J.dtype = dt;
    J.flags = base ? ZIPNN_FLAG_DELTA : 0u;
    J.out_capacity = out_capacities[i];
    J.out_nbytes = d_out_nbytes ? d_out_nbytes + i : nullptr;
    J.chunk_begin = nch;
    J.gc_begin = ngc;
    nch += J.n_chunks;
    ngc += (uint64_t)J.n_chunks * es;
    if ((int)ln > max_lanes) max_lanes = (int)ln;
    if (es > max_groups) max_groups = es;
    jobs[i] = J;
  }
  uint32_t* err = plan_err_word();
  if (!err) return ZIPNN_ECUDA;
  zipnn_plan* p = new zipnn_plan();
  p->kind = 2;
  p->count = count;
  p->nchunks = nch;
  cudaGetDevice(&p->device);
  const size_t tbytes = align_up(sizeof(Job) * (size_t)count, 256);
  const size_t sbytes = encode_scratch_bytes(nch, ngc, count);
  cudaError_t e = cudaMalloc(&p->dmem, tbytes + sbytes);
  if (e != cudaSuccess) return fail(p, e);
  Job* d_jobs = static_cast<Job*>(p->dmem);
  EncodeScratch s;
  encode_scratch_carve(static_cast<uint8_t*>(p->dmem) + tbytes, nch, ngc, count, &s);
  e = cudaMemcpy(d_jobs, jobs.data(), sizeof(Job) * (size_t)count, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return fail(p, e);
  e = capture(p, [&](cudaStream_t cs) {
    return launch_encode(d_jobs, nullptr, count, nch, ngc, s, err, cs, max_groups, max_lanes,
                         uniform, false, 0, 0, any_base(d_bases, count));
  });
  if (e != cudaSuccess) return fail(p, e);
  *out = p;
  return ZIPNN_OK;
}

zipnn_status zipnn_plan_load(const zipnn_stream* streams, const void* const* h_containers,
                             const void* const* d_bases, void* const* d_dsts, int count,
                             size_t segment_bytes, const zipnn_tuning* tuning, zipnn_plan** out) {
  if (!out || count <= 0 || !streams || !h_containers || !d_dsts) return ZIPNN_EINVAL;
  *out = nullptr;
  if (segment_bytes == 0) segment_bytes = (size_t)512 << 20;
  // jobs as in zipnn_plan_decompress, grouped into segments of consecutive
  // containers holding about segment_bytes each
  std::vector<Job> jobs((size_t)count);
  std::vector<int> seg_first;
  size_t seg_fill = 0;
  for (int i = 0; i < count; i++) {
    const zipnn_stream* s = &streams[i];
    if (!s->data || !aligned16(s->data) || !h_containers[i]) return ZIPNN_EINVAL;
    const void* base = d_bases ? d_bases[i] : nullptr;
    if (((s->flags & ZIPNN_FLAG_DELTA) != 0) != (base != nullptr)) return ZIPNN_EINVAL;
    if ((s->orig_nbytes && !d_dsts[i]) || !aligned16(d_dsts[i]) || !aligned16(base))
      return ZIPNN_EINVAL;
    if (s->n_groups != (uint32_t)elem_size(s->dtype) || s->dtype < 0 || s->dtype > ZIPNN_U8 ||
        s->lanes < 1 || s->lanes > ZIPNN_MAX_LANES || s->chunk_bytes < ZIPNN_MIN_CHUNK ||
        (uint64_t)s->n_chunks != (s->orig_nbytes + s->chunk_bytes - 1) / s->chunk_bytes)
      return ZIPNN_EINVAL;
    if (i == 0 || seg_fill >= segment_bytes) {
      seg_first.push_back(i);
      seg_fill = 0;
    }
    seg_fill += s->nbytes;
    Job J;
    memset(&J, 0, sizeof(J));
    J.src = static_cast<const uint8_t*>(s->data);
    J.base = static_cast<const uint8_t*>(base);
    J.dst = static_cast<uint8_t*>(d_dsts[i]);
    J.nbytes = s->orig_nbytes;
    J.chunk_bytes = s->chunk_bytes;
    J.lanes = s->lanes;
    J.n_chunks = s->n_chunks;
    J.dtype = s->dtype;
    J.flags = s->flags;
    J.stream_bytes = s->nbytes;
    jobs[i] = J;
  }
  const int nseg = (int)seg_first.size();
  seg_first.push_back(count);
  // each segment's jobs, grouped by dtype family (chunk numbering restarts in
  // every group: each has its own part of the table and its own tickets), and
  // their stages from the host copies' chunk maps
  struct Segment {
    DecodeGroup groups[kDecodeFamilies];
    int n = 0;
  };
  std::vector<Segment> segs((size_t)nseg);
  for (int k = 0; k < nseg; k++) {
    const int a = seg_first[k], b = seg_first[k + 1];
    Segment& sg = segs[(size_t)k];
    std::vector<Job> part(jobs.begin() + a, jobs.begin() + b);
    std::vector<uint64_t> chunks;
    for (const Job& J : part) chunks.push_back(J.n_chunks);
    sg.n = group_decode_jobs(part, chunks, sg.groups);
    std::copy(part.begin(), part.end(), jobs.begin() + a);
    for (int f = 0; f < sg.n; f++) {
      DecodeGroup& G = sg.groups[f];
      MapNeeds nd;
      const uint64_t dflt = G.shape.max_chunk * (uint64_t)G.shape.frac64 / 64 + 1024;
      for (int i = a; i < b; i++) {
        const zipnn_stream* s = &streams[i];
        if (dtype_family(s->dtype) != G.shape.family) continue;
        const uint64_t mbytes = (uint64_t)s->n_chunks * s->n_groups * kEntryBytes;
        if (s->nbytes < kHdrBytes + mbytes) continue;
        add_map_need(static_cast<const uint8_t*>(h_containers[i]) + kHdrBytes, s->n_chunks,
                     s->n_groups, dflt, &nd);
      }
      planned_stage(nd, &G.shape);
    }
  }
  uint32_t* err = plan_err_word();
  if (!err) return ZIPNN_ECUDA;
  zipnn_plan* p = new zipnn_plan();
  p->kind = 3;
  p->count = count;
  cudaGetDevice(&p->device);
  const size_t tbytes = align_up(sizeof(Job) * (size_t)count, 256);
  const size_t kbytes =
      align_up(2 * sizeof(unsigned long long) * kDecodeFamilies * (size_t)nseg, 256);
  cudaError_t e = cudaMalloc(&p->dmem, tbytes + kbytes);
  if (e != cudaSuccess) return fail(p, e);
  Job* d_jobs = static_cast<Job*>(p->dmem);
  auto* tickets = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(p->dmem) + tbytes);
  e = cudaMemcpy(d_jobs, jobs.data(), sizeof(Job) * (size_t)count, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(tickets, 0, kbytes);
  if (e != cudaSuccess) return fail(p, e);
  zipnn_tuning tu;
  memset(&tu, 0, sizeof(tu));
  if (tuning) tu = *tuning;
  // graph: the copy stream issues the H2D copies segment by segment and marks
  // each segment's end with an event; the capture stream decodes a segment as
  // soon as its copies have landed, while the copies of the next ones proceed
  cudaStream_t sc = nullptr;
  std::vector<cudaEvent_t> evs((size_t)nseg + 1, nullptr);
  e = cudaStreamCreateWithFlags(&sc, cudaStreamNonBlocking);
  for (int k = 0; k <= nseg && e == cudaSuccess; k++)
    e = cudaEventCreateWithFlags(&evs[(size_t)k], cudaEventDisableTiming);
  if (e == cudaSuccess) e = capture(p, [&](cudaStream_t cs) {
    cudaError_t r = cudaEventRecord(evs[(size_t)nseg], cs);  // fork
    if (r == cudaSuccess) r = cudaStreamWaitEvent(sc, evs[(size_t)nseg], 0);
    for (int k = 0; k < nseg && r == cudaSuccess; k++) {
      const int a = seg_first[k], b = seg_first[k + 1];
      // one copy per run of containers that sit back to back in both host and
      // device memory (each copy costs the copy engine a few microseconds of
      // setup); exact adjacency only, so no byte outside a container is written
      for (int i = a; i < b && r == cudaSuccess; i++) {
        const uint8_t* hs = static_cast<const uint8_t*>(h_containers[i]);
        uint8_t* ds = static_cast<uint8_t*>(streams[i].data);
        size_t run = streams[i].nbytes;
        while (i + 1 < b && static_cast<const uint8_t*>(h_containers[i + 1]) == hs + run &&
               static_cast<uint8_t*>(streams[i + 1].data) == ds + run)
          run += streams[++i].nbytes;
        r = cudaMemcpyAsync(ds, hs, run, cudaMemcpyHostToDevice, sc);
      }
      if (r == cudaSuccess) r = cudaEventRecord(evs[(size_t)k], sc);
      if (r == cudaSuccess) r = cudaStreamWaitEvent(cs, evs[(size_t)k], 0);
      const Segment& sg = segs[(size_t)k];
      if (r == cudaSuccess)
        r = launch_decode_groups(d_jobs + a, sg.groups, sg.n, &tu, err,
                                 tickets + 2 * kDecodeFamilies * k, cs);
    }
    // the last wait above joined the copy stream back into the capture stream
    return r;
  });
  for (cudaEvent_t ev : evs)
    if (ev) cudaEventDestroy(ev);
  if (sc) cudaStreamDestroy(sc);
  if (e != cudaSuccess) return fail(p, e);
  *out = p;
  return ZIPNN_OK;
}

zipnn_status zipnn_plan_launch(zipnn_plan* p, void* cuda_stream) {
  if (!p || !p->exec) return ZIPNN_EINVAL;
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != p->device) return ZIPNN_EINVAL;
  cudaError_t e = cudaGraphLaunch(p->exec, static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? ZIPNN_OK : ZIPNN_ECUDA;
}

void zipnn_plan_destroy(zipnn_plan* p) {
  if (!p) return;
  if (p->exec) cudaGraphExecDestroy(p->exec);
  if (p->graph) cudaGraphDestroy(p->graph);
  if (p->dmem) cudaFree(p->dmem);
  delete p;
}

}  // extern "C"
